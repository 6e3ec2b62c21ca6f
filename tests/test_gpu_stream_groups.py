"""Streaming where a warp takes four cells (large plasmas) and one: groups that
fit a warp's registers together (128 slots) and that do not, cells with more
slots than one keeps (160), empty cells, a last group that is not full, boxes
two cells wide; against the oracle, bit for bit (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import transport as TR  # noqa: E402
from test_gpu_stream import C, FIELDS, Species, make, random_axions  # noqa: E402

H = 1e-4
DT = 0.95 * H / C


def load(pl, cap, cnt, cols):
    """All cells' axions, flat by cell: cols [7][sum cnt] in FIELDS order."""
    n = len(cnt)
    first = np.concatenate([[0], np.cumsum(cnt)[:-1]])
    at = np.repeat(np.arange(n) * cap - first, cnt) + np.arange(int(cnt.sum()))
    slab = pl.slabs["axions"]
    for name, fs in (("wp", (0, 1, 2, 3)), ("xyz", (4, 5, 6))):
        arr = np.zeros((n * cap, 4), np.float32)
        for j, f in enumerate(fs):
            arr[at, j] = cols[f]
        slab.storage[name].copy_(torch.from_numpy(arr.reshape(-1)))
    slab.count.copy_(torch.from_numpy(cnt.astype(np.int32)))
    return first


def rows(pl, cap, c, n):
    slab = pl.slabs["axions"]
    wp = slab.storage["wp"].view(-1, cap, 4)[c, :n].cpu().numpy()
    xyz = slab.storage["xyz"].view(-1, cap, 4)[c, :n].cpu().numpy()
    return np.concatenate([wp, xyz[:, :3]], 1)


def stack(sp):
    return np.stack([np.asarray(getattr(sp, f), np.float32) for f in FIELDS], 1)


@pytest.mark.parametrize("dims,periodic", [((5, 3, 3), True), ((2, 11, 1), False), ((2, 2, 2), True)])
def test_single_cells_match_oracle(dims, periodic):
    cap, n = 256, int(np.prod(dims))
    rng = np.random.default_rng(n)
    cells = [random_axions(rng, int(k)) for k in rng.integers(60, 190, n)]
    pl = make(n, cap)
    cnt = np.array([len(sp) for sp in cells])
    load(pl, cap, cnt, np.concatenate([stack(sp) for sp in cells]).T)
    for _ in range(2):
        pl.stream_axions(dims, H, DT, periodic)
        cells, _, dropped = TR.stream(cells, dims, H, DT, periodic, cap)
        assert dropped == 0
    torch.cuda.synchronize()
    assert np.array_equal(pl.slabs["axions"].count.cpu().numpy(), [len(sp) for sp in cells])
    for c, sp in enumerate(cells):
        assert np.array_equal(rows(pl, cap, c, len(sp)), stack(sp)), c
    pl.close()


# the smallest plasmas that take groups of four, for slabs of 64 slots and for
# larger ones, the last group not full. Thin cells, and columns of dense
# runs that end a group's fit; cells sampled on both, with their neighbours.
@pytest.mark.parametrize("dims,cap,dense", [((487, 481, 1), 132, (20, 60)), ((487, 481, 1), 132, (60, 100)),
                                            ((127, 231, 1), 64, (20, 50))])
def test_groups_match_oracle(dims, cap, dense):
    nx, ny, _ = dims
    n = nx * ny
    assert n % 4
    rng = np.random.default_rng(n + cap + dense[0])
    cnt = rng.integers(0, 21, n)
    starts = rng.integers(2 * nx, n - 3 * nx, 400)
    for c0 in starts:
        for row in (-nx, 0, nx):
            k = int(rng.integers(1, 7))
            cnt[c0 + row:c0 + row + k] = rng.integers(dense[0], dense[1], k)
    pool = random_axions(rng, int(cnt.sum()))
    pl = make(n, cap)
    first = load(pl, cap, cnt, stack(pool).T)
    pl.stream_axions(dims, H, DT, True)
    torch.cuda.synchronize()
    got_n = pl.slabs["axions"].count.cpu().numpy()
    assert got_n.sum() == cnt.sum()
    sample = [c for c0 in starts[:60] for c in (c0, c0 + 3)] + [0, n - 1, n - 2, n - 3, nx - 1] + \
        list(rng.integers(0, n, 40))
    for c in sample:
        i, j = c % nx, c // nx
        cells = []
        for dj in (-1, 0, 1):
            for di in (-1, 0, 1):
                b = (j + dj) % ny * nx + (i + di) % nx
                sel = slice(first[b], first[b] + cnt[b])
                cells.append(Species(*[getattr(pool, f)[sel] for f in FIELDS]))
        want = TR.stream(cells, (3, 3, 1), H, DT, False, cap)[0][4]
        assert got_n[c] == len(want), c
        assert np.array_equal(rows(pl, cap, c, len(want)), stack(want)), c
    pl.close()
