// Auxiliary kernels of libaxpic: the synthetic initial plasma, per-cell rate
// records and cached electron moments, deterministic rate evaluation for
// checking, and the reductions behind the tallies.
#include "common.cuh"
#include "misc.h"
#include "step.h"

namespace axpic {

constexpr unsigned kFullMask = 0xFFFFFFFFu;

// ---------------------------------------------------------------- records
__global__ void record_kernel(int ncells, int nspecies, CellConst cc, const double* __restrict__ T,
                              const double* __restrict__ n_ion, float* rec, int* err) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncells) return;
  float r[kRecLen];
#pragma unroll
  for (int i = 0; i < kRecLen; ++i) r[i] = 0.f;
  compute_composition(cc, n_ion + (size_t)c * nspecies, r);
  const float Tc = (float)T[c];
  if (!(Tc > 0.f) || !isfinite(Tc)) atomicOr(err, ERR_NUMERIC);
  compute_temperature(cc, Tc, r);
  float4* o = reinterpret_cast<float4*>(rec + (size_t)c * kRecLen);
#pragma unroll
  for (int i = 0; i < kRecLen / 4; ++i) o[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
}

cudaError_t launch_records(int ncells, int nspecies, const CellConst& cc, const double* T, const double* n_ion,
                           float* rec, int* err, cudaStream_t st) {
  if (ncells == 0) return cudaSuccess;
  record_kernel<<<(ncells + 127) / 128, 128, 0, st>>>(ncells, nspecies, cc, T, n_ion, rec, err);
  return cudaGetLastError();
}

// FP64 view of a cell's parameters (for checking): from the record, with the
// temperature-dependent extras recomputed exactly as the step kernels do.
__global__ void info_kernel(int first, int count, CellConst cc, double k_gamma, const float* __restrict__ rec_all,
                            double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int c = first + i;
  float r[kRecLen];
  for (int k = 0; k < kRecLen; ++k) r[k] = rec_all[(size_t)c * kRecLen + k];
  const CellExtras ex = compute_temperature(cc, r[R_T], r);
  double* o = out + (size_t)i * AXPIC_CELL_INFO_LEN;
  for (int k = 0; k < AXPIC_CELL_INFO_LEN; ++k) o[k] = 0.0;
  o[AXPIC_CI_RHO] = r[R_RHO];
  o[AXPIC_CI_XH] = r[R_XH];
  o[AXPIC_CI_NE] = (double)r[R_NE] * 1e24;
  o[AXPIC_CI_NEFF] = (double)r[R_NEFF] * 1e24;
  o[AXPIC_CI_SZ] = (double)r[R_SZ] * 1e24;
  o[AXPIC_CI_KAPPA] = ex.kappa;
  o[AXPIC_CI_QC] = ex.QC;
  o[AXPIC_CI_QB] = ex.QB;
  // k_gamma = 1 / (dt w_a^-1): recover Gamma from lambda per unit weight
  o[AXPIC_CI_GAMMA_C] = (double)r[R_CC] * k_gamma;
  o[AXPIC_CI_GAMMA_B] = (double)r[R_CB] * k_gamma;
  o[AXPIC_CI_ETA] = ex.eta;
  o[AXPIC_CI_T] = r[R_T];
  o[AXPIC_CI_GAMMA0_P] = (double)r[R_AP];  // Gamma_0 dt; the host divides by dt
}

cudaError_t launch_info(int first, int count, const CellConst& cc, double k_gamma, const float* rec, double* out,
                        cudaStream_t st) {
  if (count == 0) return cudaSuccess;
  info_kernel<<<(count + 127) / 128, 128, 0, st>>>(first, count, cc, k_gamma, rec, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- deposit
// Composition from the deposited electron density (Sec. II.E, Eqs. rho_def,
// qn_def): n_e = sum w / V over the cell's electron macroparticles, then
// n_i = n_e * coef_i: the host's coefficients hold coef_i / V, so the device
// does no FP64 division. One warp per cell, the
// sum kept as an unevaluated binary32 pair (hi, lo): Knuth's TwoSum gives
// the exact rounding error of each hi + w, accumulated in lo, so the pair is
// within about (terms) 2^-48 of the exact sum without the FP64 pipe. The
// lanes' pairs are combined the same way; one FP64 add per cell evaluates
// the pair.
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float w) {
  const float s = __fadd_rn(hi, w);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(w, bb));
  hi = s;
  lo = __fadd_rn(lo, e);
}

__global__ void deposit_kernel(int ncells, int nspecies, SpeciesPtrs e, DepositCoef k, double* __restrict__ n_ion) {
  constexpr int kU = 4;  // quads in flight per lane
  const int lane = threadIdx.x & 31;
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (c >= ncells) return;
  const int n = min(max(e.count[c], 0), e.cap);
  // quads of slots (cap is a multiple of 4); the weight is the first word of
  // each slot's record
  const float* wr = reinterpret_cast<const float*>(e.wp + (long)c * e.cap);
  float hi = 0.f, lo = 0.f;
  for (int q0 = lane; 4 * q0 < n; q0 += 32 * kU) {
    float4 v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int q = q0 + 32 * u;
      v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (4 * q < n) {
        const float* p = wr + 16 * q;
        v[u] = make_float4(__ldcs(p), __ldcs(p + 4), __ldcs(p + 8), __ldcs(p + 12));
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int j = 4 * (q0 + 32 * u);  // slots past the count add +0
      two_sum_add(hi, lo, v[u].x);
      two_sum_add(hi, lo, j + 1 < n ? v[u].y : 0.f);
      two_sum_add(hi, lo, j + 2 < n ? v[u].z : 0.f);
      two_sum_add(hi, lo, j + 3 < n ? v[u].w : 0.f);
    }
  }
  for (int o = 16; o; o >>= 1) {
    const float h2 = __shfl_xor_sync(kFullMask, hi, o), l2 = __shfl_xor_sync(kFullMask, lo, o);
    two_sum_add(hi, lo, h2);
    lo = __fadd_rn(lo, l2);
  }
  // lane 0's pair for every species (the lanes combined in different orders)
  hi = __shfl_sync(kFullMask, hi, 0);
  lo = __shfl_sync(kFullMask, lo, 0);
  if (lane < nspecies) {  // the FP64 work, in these lanes only
    double cf = 0.0;      // coef[lane], read with constant indices (no local copy)
#pragma unroll
    for (int i = 0; i < kMaxSpecies; ++i)
      if (lane == i) cf = k.coef[i];
    n_ion[(size_t)c * nspecies + lane] = ((double)hi + (double)lo) * cf;
  }
}

cudaError_t launch_deposit(int ncells, int nspecies, const SpeciesPtrs& e, const DepositCoef& k, double* n_ion,
                           cudaStream_t st) {
  if (ncells == 0) return cudaSuccess;
  deposit_kernel<<<(ncells + 7) / 8, 256, 0, st>>>(ncells, nspecies, e, k, n_ion);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- moments
// Cached electron moments W, P, U2 and var = U2 - |P|^2 / W (Eqs.
// cell_moments, var_unnormalized), one warp per cell.
__global__ void moments_kernel(int ncells, SpeciesPtrs e, float* mom) {
  const int lane = threadIdx.x & 31;
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (c >= ncells) return;
  const int n = min(max(e.count[c], 0), e.cap);
  const long b = (long)c * e.cap;
  float W = 0.f, Px = 0.f, Py = 0.f, Pz = 0.f, U2 = 0.f;
  float wmin = 3.0e38f, wmax = -3.0e38f;
  for (int i = lane; i < n; i += 32) {
    const float4 r = e.wp[b + i];
    const float w = r.x, px = r.y, py = r.z, pz = r.w;
    wmin = fminf(wmin, w);
    wmax = fmaxf(wmax, w);
    W += w;
    Px += w * px;
    Py += w * py;
    Pz += w * pz;
    U2 += w * (px * px + py * py + pz * pz);
  }
  for (int o = 16; o; o >>= 1) {
    W += __shfl_xor_sync(kFullMask, W, o);
    Px += __shfl_xor_sync(kFullMask, Px, o);
    Py += __shfl_xor_sync(kFullMask, Py, o);
    Pz += __shfl_xor_sync(kFullMask, Pz, o);
    U2 += __shfl_xor_sync(kFullMask, U2, o);
    wmin = fminf(wmin, __shfl_xor_sync(kFullMask, wmin, o));
    wmax = fmaxf(wmax, __shfl_xor_sync(kFullMask, wmax, o));
  }
  if (lane == 0) {
    float* m = mom + (size_t)c * kMomLen;
    m[M_W] = W;
    m[M_PX] = Px;
    m[M_PY] = Py;
    m[M_PZ] = Pz;
    m[M_U2] = U2;
    m[M_VAR] = W > 0.f ? fmaxf(0.f, U2 - (Px * Px + Py * Py + Pz * Pz) / W) : 0.f;
    m[M_WU] = (n > 0 && wmin == wmax && wmin > 0.f) ? wmin : 0.f;
    m[7] = 0.f;
  }
}

cudaError_t launch_moments(int ncells, const SpeciesPtrs& e, float* mom, cudaStream_t st) {
  if (ncells == 0) return cudaSuccess;
  moments_kernel<<<(ncells + 7) / 8, 256, 0, st>>>(ncells, e, mom);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- sampler
// Synthetic initial plasma: per cell, NR-Maxwellian electrons (Box-Muller on
// block sub 0, positions on sub 1), Planck photons and MB-equilibrium axions
// (energy from word 0 through the inverse-CDF tables, direction from words 1
// and 2, positions on sub 1). One warp per cell.
__global__ void sample_kernel(SampleArgs S) {
  const int lane = threadIdx.x & 31;
  const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (c >= S.ncells) return;
  const uint32_t gcell = S.cell_base + (uint32_t)c;
  const float* rec = S.rec + (size_t)c * kRecLen;
  const float T = rec[R_T];
  const float sigma = sqrtf(T * kInvMeC2f);
  const float we = rec[R_NE] * S.k_we;             // n_e V / n_el
  const float wg = T * T * T * S.k_wg;             // n_gamma V / n_ph
  for (int sp = 0; sp < 3; ++sp) {
    const SpeciesPtrs& P = sp == 0 ? S.e : (sp == 1 ? S.g : S.a);
    const int n = sp == 0 ? S.n_el : (sp == 1 ? S.n_ph : S.n_ax);
    const uint32_t stream = sp == 0 ? S_INIT_E : (sp == 1 ? S_INIT_G : S_INIT_A);
    const long b = (long)c * P.cap;
    for (int i = lane; i < n; i += 32) {
      const uint4 b0 = philox4x32_10(make_uint4(kInitStep, gcell, (uint32_t)i, stream << 24), S.key0, S.key1);
      const uint4 b1 = philox4x32_10(make_uint4(kInitStep, gcell, (uint32_t)i, (stream << 24) | 1u), S.key0, S.key1);
      float w, px, py, pz;
      if (sp == 0) {
        const float r1 = sqrtf(-2.0f * logf(u23(b0.x)));
        const float r2 = sqrtf(-2.0f * logf(u23(b0.z)));
        float s1, c1, s2, c2;
        sincospif(2.0f * u23(b0.y), &s1, &c1);
        sincospif(2.0f * u23(b0.w), &s2, &c2);
        px = sigma * r1 * c1;
        py = sigma * r1 * s1;
        pz = sigma * r2 * c2;
        w = we;
      } else {
        const float* tab = S.tables + (sp == 1 ? TAB_PLANCK : TAB_MBAXION) * kTableN;
        const float pm = icdf_lookup(tab, u23(b0.x)) * T * kInvMeC2f;
        const float3 d = iso_dir(u23(b0.y), u23(b0.z));
        px = pm * d.x;
        py = pm * d.y;
        pz = pm * d.z;
        w = sp == 1 ? wg : S.w_a;
      }
      P.wp[b + i] = make_float4(w, px, py, pz);
      P.xyz[b + i] = make_float4(u23(b1.x), u23(b1.y), u23(b1.z), 0.f);
    }
    if (lane == 0) P.count[c] = n;
  }
}

cudaError_t launch_sample(const SampleArgs& S, cudaStream_t st) {
  if (S.ncells == 0) return cudaSuccess;
  sample_kernel<<<(S.ncells + 7) / 8, 256, 0, st>>>(S);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- rates
__global__ void rates_kernel(const float* __restrict__ rec_all, int cell, const float* __restrict__ E, int n,
                             int eq_stats, float am3, float prim_mult, float mu2, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float rec[kRecLen];
  for (int k = 0; k < kRecLen; ++k) rec[k] = rec_all[(size_t)cell * kRecLen + k];
  const float om = E[i];
  const float x = om * rec[R_INVT];
  // gamma->a of a massive axion: beta(omega) times the rate (1 when massless)
  const float beta = mu2 > 0.f ? axion_beta(om * kInvMeC2f, mu2) : 1.0f;
  out[4 * i + 0] = prim_prob(rec, om, beta * rec[R_AP]);
  out[4 * i + 1] = prim_prob(rec, om, prim_mult * rec[R_AP]);
  out[4 * i + 2] = tau_compton(rec, x, eq_stats);
  out[4 * i + 3] = tau_brems(rec, x, am3, eq_stats);
}

cudaError_t launch_rates(const float* rec, int cell, const float* E, int n, int eq_stats, float am3, float prim_mult,
                         float mu2, float* out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  rates_kernel<<<(n + 255) / 256, 256, 0, st>>>(rec, cell, E, n, eq_stats, am3, prim_mult, mu2, out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- reductions
// Column sums: blocks [0, kNumCounters) of the per-CTA counters, blocks
// kNumCounters + j of the totals kernel's per-CTA partials (column j of 8), in
// a fixed order.
constexpr int kColThreads = 512;
__global__ void __launch_bounds__(kColThreads) columns_kernel(const unsigned long long* __restrict__ ctr, int rows,
                                                              double* out, const double* __restrict__ part, int nparts,
                                                              double* out8) {
  __shared__ unsigned long long buf[kColThreads];
  __shared__ double dbuf[kColThreads];
  const bool counters = blockIdx.x < kNumCounters;
  const int col = counters ? blockIdx.x : blockIdx.x - kNumCounters;
  unsigned long long s = 0;
  double d = 0.0;
  if (counters) {
    for (int r = threadIdx.x; r < rows; r += kColThreads) s += ctr[(size_t)r * kNumCounters + col];
  } else {
    for (int r = threadIdx.x; r < nparts; r += kColThreads) d += part[(size_t)r * 8 + col];
  }
  buf[threadIdx.x] = s;
  dbuf[threadIdx.x] = d;
  __syncthreads();
  for (int o = kColThreads / 2; o; o >>= 1) {
    if (threadIdx.x < o) {
      buf[threadIdx.x] += buf[threadIdx.x + o];
      dbuf[threadIdx.x] += dbuf[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (counters) out[col] = (double)buf[0];
    else out8[col] = dbuf[0];
  }
}

// Folds the tally rows: thread (x, y) sums rows y, y + 32, ... of entry x,
// its loads issued together; no more threads than rows (8 rows of 60,006 entries:
// a tally of 1,000 cells 184 -> 133 us without the idle ones).
constexpr int kFoldY = 32;
__global__ void __launch_bounds__(32 * kFoldY) fold_tally_kernel(double* __restrict__ rows, int nrows, long stride,
                                                                 int n, double* __restrict__ tally) {
  __shared__ double part[kFoldY][33];
  const int i = blockIdx.x * 32 + threadIdx.x;
  double s = 0.0;
  if (i < n) {
    static_assert(kTallyRows % kFoldY == 0, "row passes");
    double v[kTallyRows / kFoldY];
#pragma unroll
    for (int k = 0; k < kTallyRows / kFoldY; ++k) {
      const int r = threadIdx.y + k * kFoldY;
      v[k] = r < nrows ? rows[r * stride + i] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kTallyRows / kFoldY; ++k) {
      const int r = threadIdx.y + k * kFoldY;
      if (r < nrows) rows[r * stride + i] = 0.0;
      s += v[k];
    }
  }
  part[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && i < n) {
    double t = 0.0;
    for (int y = 0; y < (int)blockDim.y; ++y) t += part[y][threadIdx.x];
    tally[i] += t;
  }
}

cudaError_t launch_fold_tally(double* rows, int nrows, long stride, int n, double* tally, cudaStream_t st) {
  fold_tally_kernel<<<(n + 31) / 32, dim3(32, min(nrows, kFoldY)), 0, st>>>(rows, nrows, stride, n, tally);
  return cudaGetLastError();
}

// Alive totals: sum w and sum w E for axions and photons, electron NR
// kinetic energy, macroparticle counts and carried energy.
//
// Bound by the particle bytes (16 B each). FP64 runs at 1/64 of the FP32 rate
// here, so a lane sums its particles in an unevaluated triple of binary32
// numbers: TwoSum is exact, so what is lost is the rounding of the third
// member, 2^-72 of the sum a term, below the 2^-53 a term of an FP64 sum;
// a product enters as its binary32 value and the exact remainder that fma
// gives. One FP64 evaluation per lane ends the kernel. The persistent warps
// take 8 cells at a time (their counts in one load, a cell's first loads of
// all species together) and each CTA writes one row of partial sums; a second
// kernel adds the rows in a fixed order. With FP64 sums, a shuffle reduction
// and 8 atomics on one line per cell it took 2217 us for 262,144 cells of 109
// particles (457 MB); now 109 us (ncu), 4.3 TB/s with 32 warps an SM.
constexpr int kTotThreads = 256;
constexpr int kTotWarps = kTotThreads / 32;
constexpr int kTotCells = 8;  // cells a warp takes at a time

// The same five sums by FP64 over this warp's cells, for sums outside the
// triples' range.
__device__ __noinline__ void totals_fp64(int ncells, const SpeciesPtrs& e, const SpeciesPtrs& g, const SpeciesPtrs& a,
                                         int warp, int nwarps, double* v) {
  const int lane = threadIdx.x & 31;
  for (int j = 0; j < 5; ++j) v[j] = 0.0;
  for (int c0 = warp * kTotCells; c0 < ncells; c0 += nwarps * kTotCells)
    for (int c = c0; c < min(c0 + kTotCells, ncells); ++c) {
      const int na = min(max(a.count[c], 0), a.cap), ng = min(max(g.count[c], 0), g.cap),
                ne = min(max(e.count[c], 0), e.cap);
      for (int i = lane; i < na; i += 32) {
        const float4 r = a.wp[(long)c * a.cap + i];
        v[0] += r.x;
        v[1] += (double)r.x * sqrtf(sum_sq(r.y, r.z, r.w));
      }
      for (int i = lane; i < ng; i += 32) {
        const float4 r = g.wp[(long)c * g.cap + i];
        v[2] += r.x;
        v[3] += (double)r.x * sqrtf(sum_sq(r.y, r.z, r.w));
      }
      for (int i = lane; i < ne; i += 32) {
        const float4 r = e.wp[(long)c * e.cap + i];
        v[4] += 0.5 * (double)r.x * (double)sum_sq(r.y, r.z, r.w);
      }
    }
}

__global__ void __launch_bounds__(kTotThreads) totals_kernel(int ncells, SpeciesPtrs e, SpeciesPtrs g, SpeciesPtrs a,
                                                             const double* __restrict__ res,
                                                             double* __restrict__ part) {
  __shared__ double sums[kTotWarps][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int warp = blockIdx.x * kTotWarps + wid, nwarps = gridDim.x * kTotWarps;
  Sum3 aw, aE, gw, gE, eE;
  unsigned long long macro = 0;  // lanes 0..7 axions, 8..15 photons
  double carried = 0.0;          // lanes 24..31
  for (int c0 = warp * kTotCells; c0 < ncells; c0 += nwarps * kTotCells) {
    // lanes 0..7 the cells' axion counts, 8..15 photons, 16..23 electrons
    int n = 0;
    const int cl = c0 + (lane & 7);
    if (cl < ncells) {
      if (lane < 8) n = min(max(a.count[cl], 0), a.cap);
      else if (lane < 16) n = min(max(g.count[cl], 0), g.cap);
      else if (lane < 24) n = min(max(e.count[cl], 0), e.cap);
      else carried += res[(size_t)cl * 4];
    }
    if (lane < 16) macro += (unsigned long long)n;
    const int nc = min(kTotCells, ncells - c0);
    for (int k = 0; k < nc; ++k) {
      const int na = __shfl_sync(kFullMask, n, k), ng = __shfl_sync(kFullMask, n, 8 + k),
                ne = __shfl_sync(kFullMask, n, 16 + k);
      const float4* pa = a.wp + (long)(c0 + k) * a.cap;
      const float4* pg = g.wp + (long)(c0 + k) * g.cap;
      const float4* pe = e.wp + (long)(c0 + k) * e.cap;
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int i0 = 0; i0 < max(max(na, ng), (ne + 1) / 2); i0 += 32) {
        const int i = i0 + lane, j0 = 2 * i0 + lane, j1 = j0 + 32;
        const float4 ra = i < na ? pa[i] : z;
        const float4 rg = i < ng ? pg[i] : z;
        const float4 r0 = j0 < ne ? pe[j0] : z;
        const float4 r1 = j1 < ne ? pe[j1] : z;
        if (i0 < na) {
          aw.add(ra.x);
          aE.add_product(ra.x, sqrtf(sum_sq(ra.y, ra.z, ra.w)));
        }
        if (i0 < ng) {
          gw.add(rg.x);
          gE.add_product(rg.x, sqrtf(sum_sq(rg.y, rg.z, rg.w)));
        }
        if (2 * i0 < ne) {
          eE.add_product(r0.x, sum_sq(r0.y, r0.z, r0.w));
          eE.add_product(r1.x, sum_sq(r1.y, r1.z, r1.w));
        }
      }
    }
  }
  double v[8] = {aw.value(), aE.value(), gw.value(), gE.value(), 0.5 * eE.value(), 0.0, 0.0, carried};
  if (__any_sync(kFullMask, aw.unsafe() || aE.unsafe() || gw.unsafe() || gE.unsafe() || eE.unsafe()))
    totals_fp64(ncells, e, g, a, warp, nwarps, v);
  if (lane < 8) v[5] = (double)macro;
  else if (lane < 16) v[6] = (double)macro;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    double x = v[j];
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
    if (lane == 0) sums[wid][j] = x;
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    double x = 0.0;
    for (int w = 0; w < kTotWarps; ++w) x += sums[w][threadIdx.x];
    part[(size_t)blockIdx.x * 8 + threadIdx.x] = x;
  }
}

cudaError_t totals_resident_ctas(int* out) {
  *out = resident_ctas((const void*)totals_kernel, kTotThreads, 0);
  return *out > 0 ? cudaSuccess : cudaErrorUnknown;
}

cudaError_t launch_totals(int ncells, const SpeciesPtrs& e, const SpeciesPtrs& g, const SpeciesPtrs& a,
                          const double* res, const unsigned long long* ctr, int ctr_rows, double* out8,
                          double* out_ctr, double* part, int max_parts, int fit, cudaStream_t st) {
  int grid = 0;
  if (ncells > 0) {
    grid = (ncells + kTotWarps * kTotCells - 1) / (kTotWarps * kTotCells);
    grid = min(min(grid, fit), max_parts);
    totals_kernel<<<grid, kTotThreads, 0, st>>>(ncells, e, g, a, res, part);
    cudaError_t err = cudaGetLastError();
    if (err) return err;
  }
  columns_kernel<<<kNumCounters + 8, kColThreads, 0, st>>>(ctr, ctr_rows, out_ctr, part, grid, out8);
  return cudaGetLastError();
}

}  // namespace axpic
