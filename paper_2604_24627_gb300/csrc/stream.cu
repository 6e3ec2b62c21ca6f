// Axion free streaming and cell migration: x += (p / E) c dt with E =
// sqrt(p^2 + m_a^2) (Sec. II.B: massless axions at c, massive ones
// sub-luminal; the transport of the axion macroparticles between steps) on
// the cell-sorted slabs, positions being fractions of the cell.
//
// Two kernels, a warp for K consecutive cells each:
//  * stream_move_kernel moves every axion of its cells, in binary32 with each
//    rounding fixed (the result decides the destination cell), writes the
//    new position in place, a bit per slot that does not stay, the first
//    staging row of each of the 27 directions (16-bit prefix sums, 64 bytes a
//    cell), and the leaving axions into the cell's staging rows, grouped by
//    direction in slot order.
//  * stream_place_kernel takes the arrivals from its neighbours' staging
//    rows, ordered by the neighbour's position relative to it, (dz, dy, dx)
//    ascending, then by source slot, into the slots its own leavers freed
//    (ascending), then after the old count; freed slots left over are closed
//    by the tail fill. Staying axions keep their slots unless the tail fill
//    moves them. Slots beyond the capacity are dropped, counted, and latch
//    ERR_CAPACITY.
// The first kernel writes only its own cells' slots and rows; the second
// reads the neighbours' rows and writes only its own slabs, so neither needs
// a barrier across cells.
//
// Bound by instruction issue and memory latency together; the bytes are 48 an
// axion (32 read, 16 written) and 96 a leaver (staged, read, placed). So a
// warp takes as many cells as keep its lanes full, an axion's records stay in
// registers from the move to the staging, the direction ranks and counts come
// from one match per 32 slots, an arrival finds its group by a 5-step search
// and its slot by a bit count, and a neighbour's group is two 16-bit loads.
// Warp instructions a cell, move + place: 912 + 1371 -> 696 + 727 with 128
// axions in 2-D, 404 + 595 -> 156 + 253 with 13 in 3-D. Time of a call:
// 65,536 cells of 128 249 -> 216 us, 262,144 cells of 13 in 3-D 350 -> 166 us
// (ncu, both kernels).
#include "stream.h"

namespace axpic {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr float kBelowOne = 0x1.fffffep-1f;

// New fraction of one position component and the cell shift in {-1, 0, 1}:
// t = q + d, s = floor(t), t - s (the largest binary32 below 1 where that
// rounds up to 1).
__device__ __forceinline__ float advance(float q, float d, int* shift) {
  const float t = __fadd_rn(q, d);
  const float s = floorf(t);
  float r = __fsub_rn(t, s);
  if (r >= 1.0f) r = kBelowOne;
  // in {-1, 0, 1} for positions in [0, 1) and kappa < 1; clamped so that no
  // input can index beyond the 27 directions
  *shift = max(-1, min(1, (int)s));
  return r;
}

// One axion moved: its new position in u (unchanged where it has no
// momentum), the direction returned.
__device__ __forceinline__ int move_axion(const StreamArgs& a, const float4& r, float4& u) {
  // E = sqrt(p^2 + mu^2): v = p / E in units of c
  const float en = __fsqrt_rn(__fadd_rn(
      __fadd_rn(__fadd_rn(__fmul_rn(r.y, r.y), __fmul_rn(r.z, r.z)), __fmul_rn(r.w, r.w)), __fmul_rn(a.mu, a.mu)));
  int sx = 0, sy = 0, sz = 0;
  if (en > 0.f) {
    const float k = __fdiv_rn(a.kappa, en);
    u.w = 0.f;
    if (a.nx > 1) u.x = advance(u.x, __fmul_rn(k, r.y), &sx);
    if (a.ny > 1) u.y = advance(u.y, __fmul_rn(k, r.z), &sy);
    if (a.nz > 1) u.z = advance(u.z, __fmul_rn(k, r.w), &sz);
  }
  return (sz + 1) * 9 + (sy + 1) * 3 + (sx + 1);
}

// Whether the neighbour of cell c in direction o lies outside an open box.
__device__ __forceinline__ bool escapes(const StreamArgs& a, int c, int o) {
  const int ii = c % a.nx + o % 3 - 1, jj = (c / a.nx) % a.ny + (o / 3) % 3 - 1, kk = c / (a.nx * a.ny) + o / 9 - 1;
  return ii < 0 || ii >= a.nx || jj < 0 || jj >= a.ny || kk < 0 || kk >= a.nz;
}

// This warp's row of the sums. One row's cache line took all the additions of
// an open box one after the other: 216,000 cells of 100 axions, a tenth of the
// cells at a face, 2014 us with one row, 719 with kStreamRows (periodic 619).
__device__ __forceinline__ double* stats_row(const StreamArgs& a) {
  return a.stats + (blockIdx.x * kWarps + (threadIdx.x >> 5)) % kStreamRows * kStreamRow;
}

__device__ __forceinline__ void count_escape(const StreamArgs& a, const float4& r) {
  const double wd = (double)r.x;
  const double pm = sqrt((double)r.y * r.y + (double)r.z * r.z + (double)r.w * r.w + (double)a.mu * a.mu);
  double* const row = stats_row(a);
  atomicAdd(row + 0, 1.0);
  atomicAdd(row + 1, wd);
  atomicAdd(row + 2, wd * pm * kMeC2);
}

// The warp's K cells as one flat range of slots: cell k's slots start at
// off[k].
template <int K>
struct FlatCells {
  int off[K + 1];
  __device__ __forceinline__ void set(int n) {  // lanes < K hold their cell's count, the others 0
    off[0] = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) off[k + 1] = off[k] + __shfl_sync(kAll, n, k);
  }
  __device__ __forceinline__ int total() const { return off[K]; }
  // cell of flat slot f, and the slot in it
  __device__ __forceinline__ int cell(int f, int* slot) const {
    int k = 0, o = 0;
#pragma unroll
    for (int j = 1; j < K; ++j)
      if (f >= off[j]) k = j, o = off[j];
    *slot = f - o;
    return k;
  }
};

__device__ __forceinline__ int incl_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(kAll, v, d);
    if (lane >= d) v += t;
  }
  return v;
}

// Slots a warp holds in registers from the move to the staging, passes of 32:
// four cells together, one cell. A cell with more is read twice beyond them.
constexpr int kHoldGroup = 4, kHoldOne = 5;
constexpr int kGroup = 4;  // cells a warp
constexpr int kWords = 32 / kGroup;  // words of freed bits a cell of a group has in shared memory
static_assert(kHoldGroup <= kWords, "freed words");

// The box that an instance is for: four cells a warp spill with an open one's code
// (62,500 cells of 60 131 us without it, 133 with; open 156), one cell does not, and
// was slower without (10,000 of 400 129 and 137 us).
enum { BOX_PERIODIC, BOX_OPEN, BOX_EITHER };

struct MoveShared {
  int cnt[kGroup * 32];      // leavers per direction so far
  int off[kGroup * 32];      // first staging row of a direction
  uint32_t freed[32];
};

// The K cells from c0 on with n_l slots in lane k < K: all of them in R
// register passes, or (K = 1) more than those hold.
template <int K, int R, int BOX>
__device__ __forceinline__ void move_cells(const StreamArgs& a, int c0, int n_l, MoveShared& S) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int W = (a.s.cap + 31) >> 5;
  const bool open = BOX == BOX_EITHER ? !a.periodic : BOX == BOX_OPEN;
  FlatCells<K> F;
  F.set(n_l);
  const int N = F.total();
#pragma unroll
  for (int k = 0; k < K; ++k) S.cnt[32 * k + lane] = 0;
  if (K > 1) S.freed[lane] = 0u;
  __syncwarp();

  // the freed bit of flat slot f, slot sl of cell k (all lanes call it)
  auto mark = [&](int f, int k, int sl, bool fr) {
    if (K == 1) {
      const unsigned m = __ballot_sync(kAll, fr);
      if (lane == 0) a.freed[(size_t)c0 * W + (f >> 5)] = m;
    } else if (fr) {
      atomicOr(&S.freed[kWords * k + (sl >> 5)], 1u << (sl & 31));
    }
  };
  // rank of a leaver among its cell and direction, in slot order
  auto rank = [&](bool leave, int key) {
    const unsigned m = __match_any_sync(kAll, leave ? key : 32 * K + lane);
    const int base = leave ? S.cnt[key] : 0;
    __syncwarp();
    if (leave && (m & lt) == 0) S.cnt[key] = base + __popc(m);
    __syncwarp();
    return base + __popc(m & lt);
  };
  auto staged = [&](int key, int rk) {
    return reinterpret_cast<float4*>(a.buf) + ((size_t)(c0 + (key >> 5)) * a.s.cap + S.off[key] + rk) * 2;
  };

  // every pass's records are loaded before any is moved
  float4 r[R], u[R];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int f = 32 * i + lane;
    if (f < N) {
      int sl;
      const int k = F.cell(f, &sl);
      const long q = (long)(c0 + k) * a.s.cap + sl;
      r[i] = a.s.wp[q];
      u[i] = a.s.xyz[q];
    }
  }
  int kr[R];  // a leaver's rank << 8 | its cell and direction, or -1
#pragma unroll
  for (int i = 0; i < R; ++i) {
    kr[i] = -1;
    if (32 * i >= N) continue;
    const int f = 32 * i + lane;
    bool leave = false, fr = false;
    int key = 0, k = 0, sl = 0;
    if (f < N) {
      k = F.cell(f, &sl);
      const int o = move_axion(a, r[i], u[i]);
      a.s.xyz[(long)(c0 + k) * a.s.cap + sl] = u[i];
      fr = leave = o != kStreamStay;
      if (open && leave && escapes(a, c0 + k, o)) {
        leave = false;
        count_escape(a, r[i]);
      }
      key = 32 * k + o;
    }
    mark(f, k, sl, fr);
    const int rk = rank(leave, key);
    if (leave) kr[i] = rk << 8 | key;
  }
  // slots beyond the register passes: counted now, moved and staged below
  int held = 0;
  if (K == 1 && N > 32 * R) {
    held = S.cnt[lane];
    __syncwarp();
    for (int f0 = 32 * R; f0 < N; f0 += 32) {
      const int f = f0 + lane;
      bool fr = false;
      if (f < N) {
        const long q = (long)c0 * a.s.cap + f;
        const float4 rr = a.s.wp[q];
        float4 uu = a.s.xyz[q];
        const int o = move_axion(a, rr, uu);
        fr = o != kStreamStay;
        if (fr && (!open || !escapes(a, c0, o))) atomicAdd(&S.cnt[o], 1);
      }
      mark(f, 0, f, fr);
    }
    __syncwarp();
  }
  // staging offset of each direction's group: the leavers of the lower
  // directions (those that stay and those that escape hold none)
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int v = S.cnt[32 * k + lane];
    const int e = incl_scan(v) - v;
    S.off[32 * k + lane] = e;
    if (K == 1 || c0 + k < a.ncells) a.goff[(size_t)(c0 + k) * kStreamOffs + lane] = (uint16_t)e;
  }
  if (K > 1) {
    const int k = lane / kWords, w = lane % kWords;
    if (32 * w < __shfl_sync(kAll, n_l, k)) a.freed[(size_t)(c0 + k) * W + w] = S.freed[lane];
  }
  __syncwarp();
#pragma unroll
  for (int i = 0; i < R; ++i) {
    if (kr[i] < 0) continue;
    float4* dst = staged(kr[i] & 255, kr[i] >> 8);
    dst[0] = r[i];
    dst[1] = u[i];
  }
  if (K == 1 && N > 32 * R) {
    S.cnt[lane] = held;
    __syncwarp();
    for (int f0 = 32 * R; f0 < N; f0 += 32) {
      const int f = f0 + lane;
      bool leave = false;
      int o = 0;
      float4 rr, uu;
      if (f < N) {
        const long q = (long)c0 * a.s.cap + f;
        rr = a.s.wp[q];
        uu = a.s.xyz[q];
        o = move_axion(a, rr, uu);
        a.s.xyz[q] = uu;
        leave = o != kStreamStay;
        if (open && leave && escapes(a, c0, o)) {
          leave = false;
          count_escape(a, rr);
        }
      }
      const int rk = rank(leave, o);
      if (leave) {
        float4* dst = staged(o, rk);
        dst[0] = rr;
        dst[1] = uu;
      }
    }
  }
  __syncwarp();
}

// A warp takes K cells (kGroup, or 1): together where their slots fit the
// register passes, else one after the other.
template <int K, int BOX>
__global__ void __launch_bounds__(kThreads, 3) stream_move_kernel(StreamArgs a) {
  wait_predecessor();
  __shared__ MoveShared S[kWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int c0 = (blockIdx.x * kWarps + wid) * K;
  if (c0 >= a.ncells) return;
  const int n_l = lane < K && c0 + lane < a.ncells ? min(max(a.s.count[c0 + lane], 0), a.s.cap) : 0;
  if (K > 1 && __reduce_add_sync(kAll, (unsigned)n_l) <= 32 * kHoldGroup) {
    move_cells<K, kHoldGroup, BOX>(a, c0, n_l, S[wid]);
  } else {
    for (int k = 0; k < K && c0 + k < a.ncells; ++k) {
      const int n = __shfl_sync(kAll, n_l, k);
      move_cells<1, kHoldOne, BOX>(a, c0 + k, lane == 0 ? n : 0, S[wid]);
    }
  }
}

// Cell coordinates, stepped to the next cell without dividing again.
struct CellAt {
  int i, j, k;
  __device__ __forceinline__ void next(const StreamArgs& a) {
    if (++i == a.nx) {
      i = 0;
      if (++j == a.ny) j = 0, ++k;
    }
  }
};

constexpr int kPlace = 2;  // words of freed slots whose arrivals are loaded together

template <int K>
__global__ void __launch_bounds__(kThreads, 6) stream_place_kernel(StreamArgs a) {
  wait_predecessor();
  // a cell's arrival groups, lane r the neighbour at (dz, dy, dx) = r's
  // digits - 1: arrivals up to and with the group, the neighbour, and the
  // staging row of arrival 0 of the cell's numbering
  __shared__ int g_incl[kWarps][K * 32], g_src[kWarps][K * 32], g_row[kWarps][K * 32];
  __shared__ uint32_t freed[kWarps][K * 4];
  __shared__ int sA[kWarps][K], sH[kWarps][K];  // arrivals, freed slots
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const SpeciesPtrs& s = a.s;
  const int c0 = (blockIdx.x * kWarps + wid) * K;
  if (c0 >= a.ncells) return;
  const int W = (s.cap + 31) >> 5;
  const int n_l = lane < K && c0 + lane < a.ncells ? min(max(s.count[c0 + lane], 0), s.cap) : 0;
  FlatCells<K> F;
  F.set(n_l);
  // the cells' slots as one flat range where they are few, else cell by cell
  const bool flat = K > 1 && F.total() <= 128;
  // the arrival groups: the neighbour's axions that moved here have the shift
  // -(dz, dy, dx), direction 26 - r. All K cells' loads are issued together.
  const int dz = lane / 9 - 1, dy = (lane / 3) % 3 - 1, dx = lane % 3 - 1;
  const bool dir = lane < kStreamDirs && lane != kStreamStay && !(dx && a.nx == 1) && !(dy && a.ny == 1) &&
                   !(dz && a.nz == 1);
  int m[K], g[K], src[K];
  CellAt at;
  {
    const int row = c0 / a.nx;
    at.i = c0 - row * a.nx;
    at.k = row / a.ny;
    at.j = row - at.k * a.ny;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    m[k] = g[k] = src[k] = 0;
    if (c0 + k < a.ncells && dir) {
      int si = at.i + dx, sj = at.j + dy, sk = at.k + dz;
      bool ok = true;
      if (a.periodic) {
        si += si < 0 ? a.nx : (si >= a.nx ? -a.nx : 0);
        sj += sj < 0 ? a.ny : (sj >= a.ny ? -a.ny : 0);
        sk += sk < 0 ? a.nz : (sk >= a.nz ? -a.nz : 0);
      } else {
        ok = si >= 0 && si < a.nx && sj >= 0 && sj < a.ny && sk >= 0 && sk < a.nz;
      }
      if (ok) {
        src[k] = (sk * a.ny + sj) * a.nx + si;
        const uint16_t* o = a.goff + (size_t)src[k] * kStreamOffs + (kStreamDirs - 1 - lane);
        g[k] = o[0];
        m[k] = o[1];
      }
    }
    at.next(a);
  }
  if (flat) {  // at most 4 words a cell
    const int n_k = __shfl_sync(kAll, n_l, lane >> 2);
    if (lane < K * 4)
      freed[wid][lane] = 32 * (lane & 3) < n_k ? a.freed[(size_t)(c0 + (lane >> 2)) * W + (lane & 3)] : 0u;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    m[k] -= g[k];
    const int e = incl_scan(m[k]);
    g_incl[wid][32 * k + lane] = e;
    g_src[wid][32 * k + lane] = src[k];
    g_row[wid][32 * k + lane] = g[k] - (e - m[k]);
    if (lane == 31) sA[wid][k] = e;
  }
  __syncwarp();
  // staging row of arrival t of cell k: the first group that ends after t
  auto arrival = [&](int k, int t) {
    const int* e = g_incl[wid] + 32 * k;
    int lo = 0;
#pragma unroll
    for (int st = 16; st; st >>= 1)
      if (e[lo + st - 1] <= t) lo += st;
    return reinterpret_cast<const float4*>(a.buf) +
           ((size_t)g_src[wid][32 * k + lo] * s.cap + g_row[wid][32 * k + lo] + t) * 2;
  };
  // arrival t takes freed slot t (ascending) while there are any
  if (flat) {
    if (lane < K) {
      const uint32_t* v = freed[wid] + 4 * lane;
      sH[wid][lane] = __popc(v[0]) + __popc(v[1]) + __popc(v[2]) + __popc(v[3]);
    }
    for (int f0 = 0; f0 < F.total(); f0 += 32) {
      const int f = f0 + lane;
      if (f >= F.total()) continue;
      int sl;
      const int k = F.cell(f, &sl);
      const uint32_t* v = freed[wid] + 4 * k;
      const int w = sl >> 5;
      if (!((v[w] >> (sl & 31)) & 1u)) continue;
      int t = __popc(v[w] & ((1u << (sl & 31)) - 1u));
      for (int j = 0; j < w; ++j) t += __popc(v[j]);
      if (t < sA[wid][k]) {
        const float4* x = arrival(k, t);
        const long q = (long)(c0 + k) * s.cap + sl;
        const float4 p0 = x[0], q0 = x[1];
        s.wp[q] = p0;
        s.xyz[q] = q0;
      }
    }
  } else {
    for (int k = 0; k < K; ++k) {
      const int n = __shfl_sync(kAll, n_l, k), A = sA[wid][k];
      if (n == 0) {
        if (lane == 0) sH[wid][k] = 0;
        continue;
      }
      const uint32_t* fw = a.freed + (size_t)(c0 + k) * W;
      const long base = (long)(c0 + k) * s.cap;
      const int nw = (n + 31) >> 5;
      int tb = 0;
      for (int wb = 0; wb < nw; wb += 32) {
        const uint32_t f_l = wb + lane < nw ? fw[wb + lane] : 0u;
        for (int w = wb; w < min(wb + 32, nw); w += kPlace) {
          // kPlace words at a time, all loaded before any is stored
          float4 p[kPlace], q[kPlace];
          bool b[kPlace];
#pragma unroll
          for (int i = 0; i < kPlace; ++i) {
            const uint32_t v = __shfl_sync(kAll, f_l, w - wb + i);  // wb + 32 is a multiple of kPlace
            const int t = tb + __popc(v & lt);
            tb += __popc(v);
            b[i] = ((v >> lane) & 1u) && t < A;
            if (b[i]) {
              const float4* x = arrival(k, t);
              p[i] = x[0];
              q[i] = x[1];
            }
          }
#pragma unroll
          for (int i = 0; i < kPlace; ++i)
            if (b[i]) {
              s.wp[base + 32 * (w + i) + lane] = p[i];
              s.xyz[base + 32 * (w + i) + lane] = q[i];
            }
        }
      }
      if (lane == 0) sH[wid][k] = tb;
    }
  }
  __syncwarp();
  // then slots n + (t - H): the cells' further arrivals as one flat range
  FlatCells<K> X;
  X.off[0] = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) X.off[k + 1] = X.off[k] + max(sA[wid][k] - sH[wid][k], 0);
  for (int f0 = 0; f0 < X.total(); f0 += 32) {
    const int f = f0 + lane;
    int e;
    const int k = X.cell(f, &e);
    const int dst = __shfl_sync(kAll, n_l, k) + e;
    if (f < X.total() && dst < s.cap) {
      const float4* x = arrival(k, sH[wid][k] + e);
      const long q = (long)(c0 + k) * s.cap + dst;
      const float4 p0 = x[0], q0 = x[1];
      s.wp[q] = p0;
      s.xyz[q] = q0;
    }
  }
  __syncwarp();
  // fewer arrivals than freed slots: the freed slots left over (indices A
  // .. H - 1) below the new count ns take, in ascending order, the kept slots
  // at or beyond ns (stayers and filled slots), in ascending order
  for (int k = 0; k < K; ++k) {
    const int A = sA[wid][k], H = sH[wid][k];
    const int n = __shfl_sync(kAll, n_l, k), ns = n - (H - A);
    if (A >= H) continue;
    const uint32_t* fw = flat ? freed[wid] + 4 * k : a.freed + (size_t)(c0 + k) * W;
    const long base = (long)(c0 + k) * s.cap;
    int before = 0;  // freed slots of the words before the current one
    const int w0 = ns >> 5;
    for (int w = 0; w < w0; ++w) before += __popc(fw[w]);
    int moved = 0;
    for (int w = w0; 32 * w < n; ++w) {
      const uint32_t v = fw[w];
      const int sl = 32 * w + lane;
      const bool left = ((v >> lane) & 1u) && before + __popc(v & lt) >= A;  // freed and not filled
      const bool mv = sl >= ns && sl < n && !left;
      const unsigned mm = __ballot_sync(kAll, mv);
      if (mv) {
        int j = A + moved + __popc(mm & lt), d = 0;  // the freed slot it takes, of all freed slots
        for (int p = __popc(fw[0]); j >= p; p = __popc(fw[d])) {
          j -= p;
          ++d;
        }
        const long qf = base + sl, qt = base + 32 * d + nth_bit(fw[d], j);
        const float4 p0 = s.wp[qf], q0 = s.xyz[qf];
        s.wp[qt] = p0;
        s.xyz[qt] = q0;
      }
      moved += __popc(mm);
      before += __popc(v);
    }
  }
  if (lane < K && c0 + lane < a.ncells) {
    const int total = n_l - sH[wid][lane] + sA[wid][lane];
    s.count[c0 + lane] = min(total, s.cap);
    if (total > s.cap) {
      atomicAdd(stats_row(a) + 3, (double)(total - s.cap));
      atomicOr(a.err, ERR_CAPACITY);
    }
  }
}

template <int K>
cudaError_t launch(const StreamArgs& a, cudaStream_t st) {
  const int grid = (a.ncells + kWarps * K - 1) / (kWarps * K);
  constexpr int periodic = K == 1 ? BOX_EITHER : BOX_PERIODIC, open = K == 1 ? BOX_EITHER : BOX_OPEN;
  const cudaError_t e = launch_chained(false, a.periodic ? stream_move_kernel<K, periodic> : stream_move_kernel<K, open>,
                                       grid, kThreads, 0, st, a);
  if (e) return e;
  return launch_chained(true, stream_place_kernel<K>, grid, kThreads, 0, st, a);
}

}  // namespace

// Cells a warp: 4, so that thinly filled cells share its lanes, or 1. 4 are
// better up to about 32 axions a cell, 1 beyond; the host does not know the
// counts, only the capacities. Slabs of at most 128 slots take 4 from one
// round of resident warps on: with the usual room to grow they hold at most
// about 40. Us a call with 4 and 1 cells a warp:
//   95,000 cells of 13 in 76 slots, 3-D      63   113
//   216,000 cells of 20 in 92 slots, 3-D    179   279
//   62,500 cells of 24 in 128 slots          58    81
//   62,500 cells of 32 in 120 slots          88    94
//   62,500 cells of 60 in 128 slots         125   121
//   36,000 cells of 100 in 128 slots        106    94
// A larger slab may hold few axions too: with enough cells for 8 rounds it
// takes 4 as well (262,144 cells of about 25 in 384 slots: 250 against 345);
// with fewer, 4 cells a warp leave the last of 2 rounds nearly empty where
// the cells are full (65,536 of 128: 235 against 215).
constexpr int kRound = 152 * 48;  // the place kernel's resident warps

cudaError_t launch_stream(const StreamArgs& a, cudaStream_t st) {
  if (a.ncells <= 0) return cudaSuccess;
  const int rounds = a.s.cap <= 128 ? 1 : 8;
  return a.ncells / kGroup >= rounds * kRound ? launch<kGroup>(a, st) : launch<1>(a, st);
}

}  // namespace axpic
