// Axion merging for population control: in every cell holding more than
// n_target axions, each group of three or more axions of one momentum
// octant and |p|^2 bin becomes two, with the group's weight, momentum and
// energy (the N -> 2 merging of Vranic et al., Comput. Phys. Commun. 191, 65
// (2015), for massless particles; the method merges axions as a species of
// the PIC code, Sec. II.A, and names no algorithm).
//
// A warp per cell, persistent over the cells:
// * each slot's group (a 5-step search of its binary32 |p|^2 among the
//   thresholds, and the sign bits), its rank in the group in slot order and
//   the group sizes, from one match per 32 slots;
// * the groups of three or more in a list, and their members' slots in
//   shared memory, grouped and in slot order;
// * a lane per listed group forms the binary32 compensated sums over its
//   members in slot order, every rounding explicit (the results match the
//   oracle bit for bit), writes the two new axions into the group's first
//   two slots and marks the others freed, a bit a slot;
// * the tail fill closes the freed slots.
// Bound by instruction issue (the lanes' sums are a third of it) and latency,
// not by its bytes (a cell's axions read once, the merged ones written). With
// 16 comparisons a slot, a byte a slot in memory, a second match pass and a
// tail fill that scanned every slot with __fns it issued 2537 warp
// instructions a cell of 128 axions and took 245 us for 65,536 of them, a fifth
// of its stalls instruction fetches; now 1951 and 162 us (8 CTAs of 4 warps an
// SM at 64 registers; 10 at 48 spill and take 168 us, 12 196).
#include "merge.h"
#include "step.h"

#include <algorithm>

namespace axpic {

namespace {

constexpr int kWarpsMax = 4;
// CTAs an SM, and passes of 32 slots whose groups stay in registers: 5, or as
// many as a slab of at most 64 slots has, where fewer registers and branches pay:
// 65,536 cells of 20 axions in 32 slots 65 -> 58 us, of 30 in 48 115 -> 108 (with
// 10 and 12 CTAs an SM 115 and 127: spills), 500,000 of 10 in 20 299 -> 264.
constexpr int kCtas = 8, kHold = 5;
constexpr unsigned kAll = 0xFFFFFFFFu;
constexpr int kGroupsMax = (kMergeMaxEdges + 1) * 8;

__device__ __forceinline__ float fsum3(float a, float b, float c) {
  return __fadd_rn(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)), __fmul_rn(c, c));
}

// A compensated (Kahan) binary32 sum, every step rounded as written.
struct Kahan {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float y = __fsub_rn(v, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
  }
};

// The two axions replacing the group whose m member slots, ascending, are
// mem[0..m) of the cell at base: binary32 compensated sums in slot order,
// then p_a and p_b on either side of P at cos theta = |P| / E. Members after
// the first two are freed (their bits set).
__device__ __forceinline__ void merge_group(const SpeciesPtrs& s, long base, const uint16_t* mem, int m,
                                            uint32_t* freed) {
  Kahan W, Px, Py, Pz, E, X, Y, Z;
  // member k + 1's fields are loaded before member k's sums (m >= 3)
  int slot = mem[0];
  long q = base + slot;
  float4 r = s.wp[q], u = s.xyz[q];
  float w = r.x, px = r.y, py = r.z, pz = r.w, x = u.x, y = u.y, z = u.z;
  for (int k = 0; k < m; ++k) {
    const int next = mem[min(k + 1, m - 1)];
    const long qn = base + next;
    r = s.wp[qn];
    u = s.xyz[qn];
    const float wn = r.x, pxn = r.y, pyn = r.z, pzn = r.w, xn = u.x, yn = u.y, zn = u.z;
    W.add(w);
    Px.add(__fmul_rn(w, px));
    Py.add(__fmul_rn(w, py));
    Pz.add(__fmul_rn(w, pz));
    E.add(__fmul_rn(w, __fsqrt_rn(fsum3(px, py, pz))));
    X.add(__fmul_rn(w, x));
    Y.add(__fmul_rn(w, y));
    Z.add(__fmul_rn(w, z));
    if (k >= 2) atomicOr(&freed[slot >> 5], 1u << (slot & 31));
    slot = next, w = wn, px = pxn, py = pyn, pz = pzn, x = xn, y = yn, z = zn;
  }
  const int sa = mem[0], sb = mem[1];
  const float pm = __fdiv_rn(E.s, W.s);
  const float Pn = __fsqrt_rn(fsum3(Px.s, Py.s, Pz.s));
  float e0, e1, e2, ct;
  if (Pn > 0.f) {
    e0 = __fdiv_rn(Px.s, Pn);
    e1 = __fdiv_rn(Py.s, Pn);
    e2 = __fdiv_rn(Pz.s, Pn);
    ct = fminf(__fdiv_rn(Pn, E.s), 1.0f);
  } else {
    e0 = 0.f, e1 = 0.f, e2 = 1.f;
    ct = 0.f;
  }
  const float st = __fsqrt_rn(__fsub_rn(1.0f, __fmul_rn(ct, ct)));
  // the axis of e_P's smallest |component|, the lowest index on ties
  int k = 0;
  float amin = fabsf(e0);
  if (fabsf(e1) < amin) k = 1, amin = fabsf(e1);
  if (fabsf(e2) < amin) k = 2;
  const float ax0 = k == 0 ? 1.f : 0.f, ax1 = k == 1 ? 1.f : 0.f, ax2 = k == 2 ? 1.f : 0.f;
  const float u0 = __fsub_rn(__fmul_rn(e1, ax2), __fmul_rn(e2, ax1));
  const float u1 = __fsub_rn(__fmul_rn(e2, ax0), __fmul_rn(e0, ax2));
  const float u2 = __fsub_rn(__fmul_rn(e0, ax1), __fmul_rn(e1, ax0));
  const float un = __fsqrt_rn(fsum3(u0, u1, u2));
  const float e[3] = {e0, e1, e2};
  const float qv[3] = {__fdiv_rn(u0, un), __fdiv_rn(u1, un), __fdiv_rn(u2, un)};
  const float wh = __fmul_rn(W.s, 0.5f);
  const float mx = __fdiv_rn(X.s, W.s), my = __fdiv_rn(Y.s, W.s), mz = __fdiv_rn(Z.s, W.s);
  float pa[3], pb[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    pa[j] = __fmul_rn(pm, __fadd_rn(__fmul_rn(ct, e[j]), __fmul_rn(st, qv[j])));
    pb[j] = __fmul_rn(pm, __fsub_rn(__fmul_rn(ct, e[j]), __fmul_rn(st, qv[j])));
  }
  const long qa = base + sa, qb = base + sb;
  s.wp[qa] = make_float4(wh, pa[0], pa[1], pa[2]);
  s.xyz[qa] = make_float4(mx, my, mz, 0.f);
  s.wp[qb] = make_float4(wh, pb[0], pb[1], pb[2]);
  s.xyz[qb] = make_float4(mx, my, mz, 0.f);
}

__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

struct MergeShared {
  uint16_t cnt[kGroupsMax];   // group sizes
  uint16_t start[kGroupsMax]; // first member position of a listed group
  uint16_t run[kGroupsMax];   // members placed so far (slots beyond the registers)
  uint8_t list[kGroupsMax];
};

// Dynamic shared memory, per warp: cap slot indices (u16), then a bit a slot.
__host__ __device__ inline size_t warp_bytes(int cap) {
  return ((size_t)cap * sizeof(uint16_t) + 3) / 4 * 4 + (size_t)((cap + 31) / 32) * sizeof(uint32_t);
}

template <int HOLD>
__global__ void __launch_bounds__(kWarpsMax * 32, kCtas) merge_kernel(MergeArgs a) {
  extern __shared__ __align__(16) unsigned char smem_warps[];
  __shared__ MergeShared sh[kWarpsMax];
  __shared__ float edges[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const SpeciesPtrs& s = a.s;
  MergeShared& S = sh[wid];
  uint16_t* const mem = reinterpret_cast<uint16_t*>(smem_warps + wid * warp_bytes(s.cap));
  uint32_t* const freed = reinterpret_cast<uint32_t*>(smem_warps + (wid + 1) * warp_bytes(s.cap)) - (s.cap + 31) / 32;
  const int ngroups = (a.nedges + 1) * 8;
  const unsigned lt = (1u << lane) - 1u;
  // the thresholds, then values that no |p|^2 reaches (comparisons with NaN fail)
  if (threadIdx.x < 32) edges[threadIdx.x] = threadIdx.x < a.nedges ? a.edges[threadIdx.x] : __int_as_float(0x7FC00000);
  __syncthreads();
  // the number of thresholds at or below |p|^2, times 8, plus the octant of p
  auto group_of = [&](const float4& r) {
    const float px = r.y, py = r.z, pz = r.w;
    const float p2 = __fadd_rn(__fadd_rn(__fmul_rn(px, px), __fmul_rn(py, py)), __fmul_rn(pz, pz));
    int e = 0;
#pragma unroll
    for (int st = 16; st; st >>= 1)
      if (edges[e + st - 1] <= p2) e += st;
    return e * 8 + (px < 0.f ? 1 : 0) + (py < 0.f ? 2 : 0) + (pz < 0.f ? 4 : 0);
  };
  int total = 0;
  for (int c = blockIdx.x * nw + wid; c < a.ncells; c += gridDim.x * nw) {
    const int n = min(max(s.count[c], 0), s.cap);
    if (n <= a.n_target) continue;
    const long base = (long)c * s.cap;
    for (int g = lane; g < ngroups; g += 32) S.cnt[g] = 0;
    for (int w = lane; 32 * w < n; w += 32) freed[w] = 0u;
    float4 r[HOLD];
#pragma unroll
    for (int i = 0; i < HOLD; ++i) {
      const int slot = 32 * i + lane;
      if (slot < n) {
        r[i] = s.wp[base + slot];
        prefetch_l1(s.xyz + base + slot);  // read by the slot's group
      }
    }
    __syncwarp();
    int gr[HOLD];  // group | rank << 8, or -1
#pragma unroll
    for (int i = 0; i < HOLD; ++i) {
      gr[i] = -1;
      if (32 * i >= n) continue;
      const bool live = 32 * i + lane < n;
      const int g = live ? group_of(r[i]) : kGroupsMax + lane;
      const unsigned peers = __match_any_sync(kAll, g);
      const int rank = (live ? S.cnt[g] : 0) + __popc(peers & lt);
      __syncwarp();
      if (live) {
        if ((peers & lt) == 0) S.cnt[g] = (uint16_t)(rank + __popc(peers));
        gr[i] = g | rank << 8;
      }
      __syncwarp();
    }
    if (n > 32 * HOLD) {
      for (int g = lane; g < ngroups; g += 32) S.run[g] = S.cnt[g];
      __syncwarp();
      for (int s0 = 32 * HOLD; s0 < n; s0 += 32) {
        const bool live = s0 + lane < n;
        const int g = live ? group_of(s.wp[base + s0 + lane]) : kGroupsMax + lane;
        const unsigned peers = __match_any_sync(kAll, g);
        if (live && (peers & lt) == 0) S.cnt[g] += (uint16_t)__popc(peers);
        __syncwarp();
      }
    }
    // the groups of three or more: a list, and each one's first member
    // position (exclusive prefix of their sizes)
    int nm = 0, run = 0;
    for (int g0 = 0; g0 < ngroups; g0 += 32) {
      const int g = g0 + lane;
      const int m = g < ngroups ? S.cnt[g] : 0;
      const bool listed = m >= 3;
      const unsigned bm = __ballot_sync(kAll, listed);
      if (bm == 0) continue;
      const int v = listed ? m : 0;
      int incl = v;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(kAll, incl, d);
        if (lane >= d) incl += t;
      }
      if (listed) {
        S.start[g] = (uint16_t)(run + incl - v);
        S.list[nm + __popc(bm & lt)] = (uint8_t)g;
      }
      nm += __popc(bm);
      run += __shfl_sync(kAll, incl, 31);
    }
    if (nm == 0) continue;
    __syncwarp();
    // members of listed groups in slot order
#pragma unroll
    for (int i = 0; i < HOLD; ++i) {
      if (gr[i] < 0) continue;
      const int g = gr[i] & 255;
      if (S.cnt[g] >= 3) mem[S.start[g] + (gr[i] >> 8)] = (uint16_t)(32 * i + lane);
    }
    for (int s0 = 32 * HOLD; s0 < n; s0 += 32) {
      const bool live = s0 + lane < n;
      const int g = live ? group_of(s.wp[base + s0 + lane]) : kGroupsMax + lane;
      const unsigned peers = __match_any_sync(kAll, g);
      const int rank = (live ? S.run[g] : 0) + __popc(peers & lt);
      __syncwarp();
      if (live) {
        if ((peers & lt) == 0) S.run[g] = (uint16_t)(rank + __popc(peers));
        if (S.cnt[g] >= 3) mem[S.start[g] + rank] = (uint16_t)(s0 + lane);
      }
      __syncwarp();
    }
    __syncwarp();
    // a lane per listed group
    int removed = 0;
    for (int t = lane; t < nm; t += 32) {
      const int g = S.list[t], m = S.cnt[g];
      merge_group(s, base, mem + S.start[g], m, freed);
      removed += m - 2;
    }
    removed = __reduce_add_sync(kAll, removed);
    __syncwarp();  // the lanes' bits and new axions are visible
    // the tail fill: the freed slots below the new count ns take, in
    // ascending order, the kept slots at or beyond it, in ascending order
    const int ns = n - removed;
    int moved = 0;
    for (int w = ns >> 5; 32 * w < n; ++w) {
      const int slot = 32 * w + lane;
      const bool mv = slot >= ns && slot < n && !((freed[w] >> lane) & 1u);
      const unsigned mm = __ballot_sync(kAll, mv);
      if (mv) {
        int j = moved + __popc(mm & lt), d = 0;  // it takes freed slot j of all
        for (int p = __popc(freed[0]); j >= p; p = __popc(freed[d])) {
          j -= p;
          ++d;
        }
        const long qf = base + slot, qt = base + 32 * d + nth_bit(freed[d], j);
        const float4 x = s.wp[qf], u = s.xyz[qf];
        s.wp[qt] = x;
        s.xyz[qt] = u;
      }
      moved += __popc(mm);
    }
    if (lane == 0) s.count[c] = ns;
    total += removed;
    __syncwarp();
  }
  if (lane == 0 && total) atomicAdd(a.removed, (double)total);
}

}  // namespace

constexpr int kDynMax = 160 * 1024;  // the warps' dynamic shared memory, at most

// warps per CTA: as many as fit the shared memory, at most 4
static int merge_warps(int cap) {
  const size_t per_warp = std::max<size_t>(warp_bytes(cap), 4);
  return (int)std::max<size_t>(1, std::min<size_t>(kWarpsMax, kDynMax / per_warp));
}

using MergeKernel = void (*)(MergeArgs);
static MergeKernel merge_instance(int cap) {
  return cap <= 32 ? merge_kernel<1> : cap <= 64 ? merge_kernel<2> : merge_kernel<kHold>;
}

// as many CTAs as the device holds at once; asked for once, since the
// driver's answers take some microseconds and a merge of a thousand cells 40
cudaError_t merge_init_kernels(int cap, int* fit) {
  const auto kernel = merge_instance(cap);
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynMax);
  if (e) return e;
  const int nw = merge_warps(cap);
  *fit = resident_ctas((const void*)kernel, nw * 32, std::max<size_t>(warp_bytes(cap), 4) * nw);
  return *fit > 0 ? cudaSuccess : cudaErrorUnknown;
}

cudaError_t launch_merge(const MergeArgs& a, int fit, cudaStream_t st) {
  if (a.ncells <= 0) return cudaSuccess;
  if (a.s.cap > kMergeMaxCap) return cudaErrorInvalidValue;
  const int nw = merge_warps(a.s.cap);
  const int grid = std::min((a.ncells + nw - 1) / nw, fit);
  merge_instance(a.s.cap)<<<grid, nw * 32, std::max<size_t>(warp_bytes(a.s.cap), 4) * nw, st>>>(a);
  return cudaGetLastError();
}

}  // namespace axpic
