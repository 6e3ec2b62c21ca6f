"""The network's kernel at the edges of its 128-row tiles and of its
persistent grid, and with row arrays that are not 16-byte aligned, against the
FP64 oracle within the bounds of test_gpu_mlp (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import surrogate as S

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib  # noqa: E402
from paper_2604_24627_gb300.mlp import SurrogateNet  # noqa: E402
from test_gpu_mlp import forward_bound, gradient_bounds, seeded  # noqa: E402


def placed(a, off):
    """A device copy of a whose first element lies off floats into its
    allocation."""
    a = np.asarray(a, np.float32)
    t = torch.empty(a.size + off, device="cuda:0")[off:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


# one row; a tile less, exactly and one more than full; one row more than one
# tile on each of the 152 SMs (the second tile of a persistent CTA)
@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 1])
@pytest.mark.parametrize("off", [0, 1])
def test_tiles_match_oracle(n, off):
    P, X, Zt = seeded(20 + n, n)
    net = SurrogateNet()
    net.set_params(P)
    Xd, Zd = placed(X, off), placed(Zt, off)
    loss, G = net.gradients(Xd, Zd)
    want = S.backward(P, X, Zt, bf16_mma=True)
    B = gradient_bounds(P, X, Zt)
    for k in want:
        assert np.all(np.abs(G[k] - want[k]) <= B[k] + 1e-12), k
    assert abs(loss - S.loss(P, X, Zt, bf16_mma=True)) <= 1e-4 * loss
    # outputs at an offset, the words around them left alone
    buf = torch.full((n * 96 + off + 5,), 7.0, device="cuda:0")
    _lib.axpic_mlp_forward(net.h, Xd.data_ptr(), n, buf[off:].data_ptr())
    out = buf.cpu().numpy()
    zw, _ = S.forward(P, X, bf16_mma=True)
    assert np.all(np.abs(out[off:off + 96 * n].reshape(n, 96) - zw) <= forward_bound(P, X) + 1e-7)
    assert np.all(out[:off] == 7.0) and np.all(out[off + 96 * n:] == 7.0)
    # the sums run in a fixed order
    loss2, G2 = net.gradients(Xd, Zd)
    assert loss2 == loss and all(np.array_equal(G[k], G2[k]) for k in G)
    net.close()
