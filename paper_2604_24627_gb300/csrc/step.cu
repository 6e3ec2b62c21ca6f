// The per-cell step: absorb -> emit -> feedback (Sec. II.D-II.J).
//
// A step is four kernels (five with an evolved temperature under the surrogate
// model, sr.cu), each started while its predecessor ends:
//  * decide_kernel: persistent warps over chunks of consecutive cells, lane
//    per quad of consecutive slots (16-byte records {w, p} of the slabs, one
//    Philox4x32-10 block per quad and stream, word j for slot 4q+j). Each
//    slot gets a cheap exact test that proves "no event this step"; slots it
//    cannot clear are flagged in a per-cell bit mask and their full decision
//    is taken from per-warp lists, 32 at a time, into slot-indexed records.
//    This kernel carries almost all the per-particle work.
//  * event_kernel: a lane per cell, 4, 8 or 32 cells a warp. It reads the bit
//    masks and the records of the flagged slots, writes products and refills
//    removed slots in the deterministic order of the method's definition, and
//    accumulates the FP64 exchange (Delta E, Delta P). Cells with more flagged
//    slots than a lane takes are listed for
//  * event_heavy_kernel: a warp per listed cell, offsets from warp prefix sums.
//  * feedback_kernel: thread per cell for the temperature update; the cells
//    whose exchange needs an affine remap are remapped by their warp.
// The separate API calls run the same kernels with a subset of the passes (the
// event kernel's warps take their own heavy cells). The exchange passes through
// an FP64 per-cell buffer; a lane adds its events in slot order and a warp by
// halves, so the two ways differ in a sum's last bits. Which way a cell takes
// depends, in a full step, on its own flagged slots alone.
#include <mutex>

#include "common.cuh"
#include "sr.h"
#include "step.h"

namespace axpic {

constexpr unsigned kFull = 0xFFFFFFFFu;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

__device__ __forceinline__ int warp_excl_scan(int v, int* total) {
  const int lane = lane_id();
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += t;
  }
  *total = __shfl_sync(kFull, x, 31);
  return x - v;
}

__device__ __forceinline__ bool bit(const uint32_t* b, int i) { return (b[i >> 5] >> (i & 31)) & 1u; }


// Lane-local FP64 exchange (Delta E keV, Delta P m_e c) and a flag that avoids
// FP64 zero tests on the common path.
struct Lane64 {
  double dE = 0.0, dPx = 0.0, dPy = 0.0, dPz = 0.0;
  bool any = false;
  __device__ void add(double w, float om, float px, float py, float pz) {
    dE += w * (double)om;
    dPx += w * (double)px;
    dPy += w * (double)py;
    dPz += w * (double)pz;
    any = true;
  }
};

// Per-CTA counters live in shared memory; events are rare, so they are
// counted with shared-memory atomics where they happen instead of holding a
// register per counter for the whole kernel.
struct Cnt {
  unsigned long long* c;
  __device__ void add(int i, unsigned v) const {
    if (v) atomicAdd(c + i, (unsigned long long)v);
  }
};

__device__ __forceinline__ void write_particle(const SpeciesPtrs& s, long idx, float w, float px, float py,
                                               float pz, float x, float y, float z) {
  s.wp[idx] = make_float4(w, px, py, pz);
  s.xyz[idx] = make_float4(x, y, z, 0.f);
}

// A slot's weight alone (the first word of its record).
__device__ __forceinline__ float& slot_w(const SpeciesPtrs& s, long idx) {
  return reinterpret_cast<float*>(s.wp + idx)[0];
}

__device__ __noinline__ void tally_add(const StepArgs& A, int ch, float w, float E) {
  const int k = (int)floorf(E * A.inv_dE_bin);
  const double wE = (double)w * (double)E;
  double* row = A.tally + (size_t)(blockIdx.x & A.tally_mask) * A.tally_stride;
  if (k >= 0 && k < A.nbins) atomicAdd(row + ch * A.nbins + k, wE);
  atomicAdd(row + 3 * A.nbins + ch, (double)w);
  atomicAdd(row + 3 * A.nbins + 3 + ch, wE);
}

// ---------------------------------------------------------------- spectral records
// Rates from a cell's spectral record (table or surrogate rate model): the
// record holds ln(dQ_c/dx) + x at unit coupling on 32 points of ln x (step
// ln(400)/29, one beyond each end of [0.05, 20]); a Catmull-Rom spline in
// ln x interpolates it, the closed factors of Eqs. prim_rate and gamma_abs
// turn it into a rate. The entries a decision needs (4 of 192 a channel) are
// interpolated from the table where they are needed (sr_table_entry, the bits
// of the stored record): about 1.5 slots a cell and step take a full decision,
// and writing every cell's 768-byte record after each temperature update took
// 287 us a step of 884,736 cells (4 steps: 2.58 -> 1.80 ms without).
// A full decision shares everything but the rates between the two sources: with
// the whole decision written out for each, a batch with both cost twice (4.1 M
// cells under the network: decisions 1.11 -> 1.04 ms a step, 4 steps 7.63 ->
// 7.55 ms; 0.9 M under the table: 1.71 -> 1.67).
struct CellSpectrum {
  SrInterp q;
  const RecordArgs* a;
  __device__ __forceinline__ float at(int o) const { return sr_table_entry(*a, q, o); }
};

__device__ __forceinline__ bool sr_in_range(float x) { return x >= 0.05f && x <= 20.0f; }

__device__ __forceinline__ float sr_lnL(const CellSpectrum& sr, int ch, float lnx) {
  float u = (lnx - kSrLnXLo) * (1.0f / kSrH) + 1.0f;
  u = fminf(fmaxf(u, 1.f), 30.f);
  const int k = min((int)u, 29);
  const float f = u - (float)k;
  const int g = ch * kSrGrid + k;
  const float p0 = sr.at(g - 1), p1 = sr.at(g), p2 = sr.at(g + 1), p3 = sr.at(g + 2);
  const float s = p1 + 0.5f * f * (p2 - p0 + f * (2.f * p0 - 5.f * p1 + 4.f * p2 - p3 + f * (3.f * (p1 - p2) + p3 - p0)));
  return s - fminf(fmaxf(__expf(lnx), 0.05f), 20.0f);  // the stored values are ln(dQ/dx) + x
}

// Gamma_{gamma->a} dt at the cell's couplings (multiplicity 1).
__device__ __forceinline__ float sr_prim_gdt(const CellSpectrum& sr, float x) {
  const float lx = logf(x);
  return expf((sr_lnL(sr, 0, lx) + sr.q.lnKP) - 3.f * lx) * expm1f(x);
}

// Absorption tau_c = Gamma_abs,c dt (c = 1 Compton-like, 2 bremsstrahlung).
__device__ __forceinline__ float sr_tau(const CellSpectrum& sr, int ch, float x, int eq_stats) {
  const float lx = logf(x);
  const float b = expf((sr_lnL(sr, ch, lx) + sr.q.lnKA) - 3.f * lx);
  return eq_stats ? b * expm1f(x) : b * expf(x);
}

// Whether a cell's full decisions and emission energies take their rates from
// its spectral record: every cell under the table model, the cells the
// network is not trusted for under the surrogate model; the others use the
// closed forms with the cell record's prefactors.
__device__ __forceinline__ bool cell_has_sr(const StepArgs& A, int cell) {
  return A.rate_model == 1 || (A.rate_model == 2 && A.ra.src[cell]);
}

__device__ __forceinline__ CellSpectrum cell_spectrum(const StepArgs& A, const float* rec) {
  CellSpectrum s{{}, &A.ra};
  sr_interp(A.ra, sr_cell_from(rec, A.ra.k_T7), &s.q);
  return s;
}

// ---------------------------------------------------------------- decisions
// One axion at the start of the step: a->gamma conversion (Sec. II.F.1, last
// paragraph) then detailed-balance absorption of the thermal-bath channels
// (Sec. II.I).
struct AxionDecision {
  int K;
  float wprod, wnew, om, w;
  bool keep, absorbed, capped, over, abs_c;
};

__device__ __forceinline__ AxionDecision axion_decide(const float* rec, bool has_sr, const StepArgs& A, int mask,
                                                      float w, float px, float py, float pz, uint32_t wP,
                                                      uint32_t wA) {
  AxionDecision d;
  d.om = sqrtf((px * px + py * py + pz * pz) + A.mu2) * kMeC2f;  // the total energy E
  d.K = 0;
  d.wprod = 0.f;
  d.capped = false;
  d.over = false;
  d.absorbed = false;
  d.abs_c = false;
  float wrem = w;
  const float xr = d.om * rec[R_INVT];
  // the spectrum's constants once, and only where a rate comes from it
  const bool use_sr = has_sr && sr_in_range(xr);
  CellSpectrum sr{{}, &A.ra};
  if (use_sr) sr = cell_spectrum(A, rec);
  if (mask & AXPIC_CH_PRIMAKOFF) {
    const float P = use_sr ? -expm1f(-A.cc.prim_mult * sr_prim_gdt(sr, xr))
                           : prim_prob(rec, d.om, A.cc.prim_mult * rec[R_AP]);
    float fac;
    const float le = cap_lambda(w * P * A.inv_w_gref, A.lam_cap, &fac, &d.capped);
    d.K = poisson_inv(u23(wP), le);
    if (d.K > 0) d.wprod = deplete(w, d.K, d.capped ? A.w_gref * fac : A.w_gref, &wrem, &d.over);
  }
  d.keep = wrem > 0.f;
  d.wnew = wrem;
  if (d.keep && (mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS))) {
    const float x = xr;
    const float tc = !(mask & AXPIC_CH_COMPTON) ? 0.f
                     : use_sr                   ? sr_tau(sr, 1, x, A.eq_stats)
                                                : tau_compton(rec, x, A.eq_stats);
    const float tb = !(mask & AXPIC_CH_BREMS) ? 0.f
                     : use_sr                 ? sr_tau(sr, 2, x, A.eq_stats)
                                              : tau_brems(rec, x, A.brems_am3, A.eq_stats);
    const float tau = tc + tb;
    if (A.absorb_mode == 0) {
      const float P = -expm1f(-tau);
      const float u = u23(wA);
      if (u < P) {
        d.absorbed = true;
        d.keep = false;
        d.abs_c = u / P < tc / tau;
      }
    } else {
      d.wnew = wrem * expf(-tau);
      d.keep = d.wnew > 0.f;
    }
  }
  return d;
}

__device__ __forceinline__ void load_rec(const StepArgs& A, int cell, float* rec) {
  const float4* r4 = reinterpret_cast<const float4*>(A.rec + (size_t)cell * kRecLen);
#pragma unroll
  for (int i = 0; i < kRecLen / 4; ++i) {
    const float4 v = r4[i];
    rec[4 * i] = v.x;
    rec[4 * i + 1] = v.y;
    rec[4 * i + 2] = v.z;
    rec[4 * i + 3] = v.w;
  }
}

// Out-of-line full decisions of slot idx: they load the slot's record and
// the cell's record together (one round trip), so that the caller's cell
// constants stay in registers.
// SR: the spectra of rate models 1 and 2, left out of the closed forms' decision
// kernels (shorter code: 262,144 cells 4.22 -> 4.17 ms, boxes 3.67 -> 3.62,
// 64 cells 17.5 -> 17.1 us).
template <bool SR>
__device__ __noinline__ AxionDecision axion_decide_slow(const StepArgs& A, int cell, int mask, long idx, uint32_t wP,
                                                        uint32_t wA) {
  const float4 v = A.a.wp[idx];
  float rec[kRecLen];
  load_rec(A, cell, rec);
  AxionDecision d = axion_decide(rec, SR && cell_has_sr(A, cell), A, mask, v.x, v.y, v.z, v.w, wP, wA);
  d.w = v.x;
  return d;
}

// One photon at the start of the step: gamma->a conversion (Sec. II.F,
// Eqs. prim_rate, prim_prob, lambda_P, depletion).
struct PhotonDecision {
  int K;
  float wprod, wrem, om;
  bool capped, over;
};

__device__ __forceinline__ PhotonDecision photon_decide(const float* rec, bool has_sr, const StepArgs& A, float w,
                                                        float px, float py, float pz, uint32_t wd) {
  PhotonDecision d;
  const float pm = sqrtf(px * px + py * py + pz * pz);
  d.om = pm * kMeC2f;
  const float xr = d.om * rec[R_INVT];
  // a massive axion: the rate times beta(omega), zero at and below m_a
  const float beta = A.mu > 0.f ? axion_beta(pm, A.mu2) : 1.0f;
  const float P = has_sr && sr_in_range(xr) ? -expm1f(-(beta * sr_prim_gdt(cell_spectrum(A, rec), xr)))
                                            : prim_prob(rec, d.om, beta * rec[R_AP]);
  float fac;
  const float le = cap_lambda(w * P * A.inv_w_a, A.lam_cap, &fac, &d.capped);
  d.K = poisson_inv(u23(wd), le);
  d.wrem = w;
  d.wprod = 0.f;
  d.over = false;
  if (d.K > 0) d.wprod = deplete(w, d.K, d.capped ? A.w_a * fac : A.w_a, &d.wrem, &d.over);
  return d;
}

template <bool SR>
__device__ __noinline__ PhotonDecision photon_decide_slow(const StepArgs& A, int cell, long idx, uint32_t wd) {
  const float4 v = A.g.wp[idx];
  float rec[kRecLen];
  load_rec(A, cell, rec);
  return photon_decide(rec, SR && cell_has_sr(A, cell), A, v.x, v.y, v.z, v.w, wd);
}

// Guards: cheap upper bounds that prove, without the transcendental chain,
// that a particle has no event this step. Whenever a guard answers true the
// full decision would give the same answer (the bounds carry margins far
// above the binary32 rounding of the full path), so results are unchanged.
//
// Conversion: P = 1 - exp(-A F(s)) <= A F(s) and F(s) <= min(s/2, ln(1+s)),
// so lambda <= w A min(s/2, ln(1+s)) / w_ref = lb, and K = 0 whenever
// u <= 1 - lb <= exp(-lambda).
// A bound at or above the Poisson-mean cap also sends the slot to the full
// decision, so that cap hits are counted exactly.
// kb is the cell's A ln 2 / w_ref with the margin 1.0001 (times the rate
// model's guard margin) folded in. Both bounds hold in binary32 on their own:
// s/2 to its rounding, and log2(1 + s + 5e-7), whose offset covers the
// rounding of the sum and the approximation's absolute error near 1
// (2^-22), the margin its relative error.
//
// These bounds are the decision kernel's arithmetic: one special-function
// instruction and 12 others per conversion, three and 8 per absorption (the
// approximations flush subnormals, so no scaling code surrounds them, and the
// uniform is one funnel shift and one addition of the draw's word). With
// 1 - lb - 1e-6 formed from u, a comparison to choose the bound and x formed
// first, the kernel issued 205 warp instructions a cell at 5 keV and took
// 1060 us for 4.1 M cells; now 170 and 933 us.
__device__ __forceinline__ float lg2_ftz(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_ftz(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 1 + (w >> 9) 2^-23 = u + 1 - 2^-24
__device__ __forceinline__ float one_plus(uint32_t w) { return __uint_as_float(__funnelshift_r(w, 0x7Fu, 9)); }
constexpr float kGuardAbs = 1.2e-6f;  // covers the roundings of u and of the bounds below 1

__device__ __forceinline__ bool no_conversion(float w, float p2, float c_s, float kb, uint32_t word, float lam_cap) {
  const float s = p2 * c_s;
  const float Fb = fminf(0.72134752f * s, lg2_ftz(s + 1.0000005f));  // F / ln 2
  const float lb = w * kb * Fb;
  return (lb < lam_cap) & (lb < (2.0f - kGuardAbs) - one_plus(word));
}
__device__ __forceinline__ float conversion_kb(float Acoef, float inv_wref, float gm) {
  return Acoef * inv_wref * (0.69314718f * 1.0001f * gm);
}

// Absorption: P_abs <= tau; x/(1-e^-x) <= 1 + x bounds the Compton-like
// factor, (1 - e^-x) <= 1 the Bose-Einstein one. With x = c |p|, c = m_e c^2
// / T, tau <= b_c x (1 + x) + b_b x^(a-3) = bc1 |p| + bc2 p^2 + bb
// (p^2)^((a-3)/2): the cell's coefficients with the margin 1.001 (times the
// guard margin) folded in, zero for a channel that is off. p2 = 0 gives NaN,
// which clears nothing.
struct AbsorbBound {
  float bc1, bc2, bb;
};
__device__ __forceinline__ AbsorbBound absorb_bound(float b_c, float b_b, float c, float am3) {
  AbsorbBound b;
  b.bc1 = b_c * c;
  b.bc2 = b.bc1 * c;
  b.bb = b_b * ex2_ftz(am3 * lg2_ftz(c));
  return b;
}
__device__ __forceinline__ bool no_absorption(const AbsorbBound& b, float half_am3, float p2, uint32_t word) {
  const float p = p2 * rsqrt_ftz(p2);
  const float tb = b.bc2 * p2 + (b.bc1 * p + b.bb * ex2_ftz(half_am3 * lg2_ftz(p2)));
  return tb <= one_plus(word) - (1.0f + kGuardAbs);
}

// ---------------------------------------------------------------- feedback
struct RemapOut {
  double applied_E, apx, apy, apz;
  float mW, mPx, mPy, mPz, mU2;
};

// Sums over the G lanes of a group (G = 8, 16, 32; lanes of the same
// lane / G) of four values: lane i of the group returns value (2 if bit G/2
// of i is set) + (1 if bit G/4 is). The first two steps halve the values
// instead of adding all of them in every lane, so four FP64 sums over a warp
// take 6 adds instead of 20; the pairs added are a butterfly's, and so are
// the bits.
template <int G, typename T>
__device__ __forceinline__ T group_sum4(T a, T b, T c, T d) {
  const int lane = lane_id();
  const bool u = lane & (G / 2), v = lane & (G / 4);
  T k0 = u ? c : a, k1 = u ? d : b;
  k0 += __shfl_xor_sync(kFull, u ? a : c, G / 2);
  k1 += __shfl_xor_sync(kFull, u ? b : d, G / 2);
  T k = v ? k1 : k0;
  k += __shfl_xor_sync(kFull, v ? k0 : k1, G / 4);
#pragma unroll
  for (int o = G / 8; o; o >>= 1) k += __shfl_xor_sync(kFull, k, o);
  return k;
}

// The affine map on one quad of electrons, p' = p + (s1 p + b) (Eq.
// affine_map with S = 1 + s1), and what the binary32 momenta actually
// received.
struct RemapSums {
  float aE = 0.f, aPx = 0.f, aPy = 0.f, aPz = 0.f;
  float mW = 0.f, mPx = 0.f, mPy = 0.f, mPz = 0.f, mU2 = 0.f;
  __device__ __forceinline__ void quad(float4* e, const float4* v, int nj, float s1, float fbx, float fby, float fbz) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j >= nj) break;
      const float w = v[j].x, px = v[j].y, py = v[j].z, pz = v[j].w;
      const float nx = px + fmaf(s1, px, fbx);
      const float ny = py + fmaf(s1, py, fby);
      const float nz = pz + fmaf(s1, pz, fbz);
      const float ddx = nx - px, ddy = ny - py, ddz = nz - pz;
      aE += w * (ddx * (2.f * px + ddx) + ddy * (2.f * py + ddy) + ddz * (2.f * pz + ddz));
      aPx += w * ddx;
      aPy += w * ddy;
      aPz += w * ddz;
      mW += w;
      mPx += w * nx;
      mPy += w * ny;
      mPz += w * nz;
      mU2 += w * (nx * nx + ny * ny + nz * nz);
      e[j] = make_float4(w, nx, ny, nz);
    }
  }
  // The sums over the lane's group, for the lanes whose cell group `own` took.
  template <int G>
  __device__ __forceinline__ RemapOut reduce(int own) {
    const double x = group_sum4<G>((double)aE, (double)aPx, (double)aPy, (double)aPz);
    const float m = group_sum4<G>(mW, mPx, mPy, mPz);
#pragma unroll
    for (int o = G / 2; o; o >>= 1) mU2 += __shfl_xor_sync(kFull, mU2, o);
    const int src = own * G;
    RemapOut o;
    o.applied_E = __shfl_sync(kFull, x, src) * 0.5 * kMeC2;
    o.apx = __shfl_sync(kFull, x, src + G / 4);
    o.apy = __shfl_sync(kFull, x, src + G / 2);
    o.apz = __shfl_sync(kFull, x, src + G / 2 + G / 4);
    o.mW = __shfl_sync(kFull, m, src);
    o.mPx = __shfl_sync(kFull, m, src + G / 4);
    o.mPy = __shfl_sync(kFull, m, src + G / 2);
    o.mPz = __shfl_sync(kFull, m, src + G / 2 + G / 4);
    o.mU2 = __shfl_sync(kFull, mU2, src);
    return o;
  }
};

// The remap of the warp's cells of `need` (a lane's bit: its own cell, with
// its electrons ne and the map s1, b). G lanes a cell, 32 / G cells side by
// side, each with at most G quads of electrons unless G is 32. A lane sums
// its quads in ascending order, so the result does not depend on G: the
// lanes beyond a cell's quads add zeros.
template <int G>
__device__ __noinline__ RemapOut remap_cells(const StepArgs& A, unsigned need, int cell, int ne, float s1, float bx,
                                             float by, float bz) {
  const int lane = lane_id(), gl = lane & (G - 1);
  RemapOut mine = {};
  // the next cell (its lane) of this lane's group; the group of this lane's cell
  auto pick = [&](int& j, int& own) {
    j = own = -1;
#pragma unroll
    for (int g = 0; g < 32 / G; ++g) {
      const int b = __ffs(need) - 1;
      if (lane / G == g) j = b;
      if (b == lane) own = g;
      need &= need - 1u;
    }
  };
  if constexpr (G == 32) {
    while (need) {
      int j, own;
      pick(j, own);
      float4* const e = A.e.wp + (long)__shfl_sync(kFull, cell, j) * A.e.cap;
      const int n = __shfl_sync(kFull, ne, j), nq = (n + 3) >> 2;
      const float t1 = __shfl_sync(kFull, s1, j), tx = __shfl_sync(kFull, bx, j), ty = __shfl_sync(kFull, by, j),
                  tz = __shfl_sync(kFull, bz, j);
      RemapSums S;
      // two quads per lane and pass, both loaded before either is stored
      for (int q0 = lane; q0 < nq; q0 += 64) {
        float4 v[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (q0 + 32 * h < nq)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[h][k] = e[4 * (q0 + 32 * h) + k];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = q0 + 32 * h;
          if (q < nq) S.quad(e + 4 * q, v[h], n - 4 * q, t1, tx, ty, tz);
        }
      }
      __syncwarp();
      const RemapOut r = S.reduce<32>(0);
      if (own >= 0) mine = r;
    }
  } else {
    // one quad a lane; the next cells' quads are loaded before these are summed
    int j, own, n = 0;
    float4* e = nullptr;
    float4 v[4];
    auto load = [&](float4*& ep, int& np, float4* vp) {
      const int src = max(j, 0);
      ep = A.e.wp + (long)__shfl_sync(kFull, cell, src) * A.e.cap + 4 * gl;
      np = __shfl_sync(kFull, ne, src) - 4 * gl;  // electrons from this lane's quad on
      if (j < 0) np = 0;
      if (np > 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) vp[k] = ep[k];
    };
    pick(j, own);
    load(e, n, v);
    while (true) {
      const int src = max(j, 0), o = own;
      const float t1 = __shfl_sync(kFull, s1, src), tx = __shfl_sync(kFull, bx, src),
                  ty = __shfl_sync(kFull, by, src), tz = __shfl_sync(kFull, bz, src);
      const bool more = need != 0;
      float4* e2 = nullptr;
      int n2 = 0;
      float4 v2[4];
      if (more) {
        pick(j, own);
        load(e2, n2, v2);
      }
      RemapSums S;
      if (n > 0) S.quad(e, v, n, t1, tx, ty, tz);
      __syncwarp();
      const RemapOut r = S.reduce<G>(max(o, 0));
      if (o >= 0) mine = r;
      if (!more) break;
      e = e2;
      n = n2;
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = v2[k];
    }
  }
  return mine;
}

__device__ __forceinline__ bool nz64(double v) { return (__double_as_longlong(v) << 1) != 0; }

// Conversions on the integer units: an FP64 instruction, a conversion
// included, takes 16 cycles of an SM for a warp, these a few each. The same
// bits as the plain conversion, which takes what is subnormal, infinite or
// not a number in binary32.
__device__ __forceinline__ float f32_of(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t m = hi & 0x7FFFFFFFu;
  if (m - 0x38100000u < 0x47F00000u - 0x38100000u) {  // 2^-126 <= |x| < 2^128: rounded to nearest even
    uint32_t u = __funnelshift_l(lo, m - 0x38000000u, 3);
    u += (lo & 0x1FFFFFFFu) + (u & 1u) > 0x10000000u;
    return __uint_as_float(u | (hi & 0x80000000u));
  }
  return (float)x;
}
__device__ __forceinline__ double f64_of(float x) {
  const uint32_t u = __float_as_uint(x), m = u & 0x7FFFFFFFu;
  if (m - 0x00800000u < 0x7F000000u)  // normal
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
  return m ? (double)x : __hiloint2double((int)u, 0);
}
// |x| from the upper half of its bits, at most 2^-20 below it; 0 below
// 2^-126, infinite from 2^128 on and where x is not a number
__device__ __forceinline__ float abs_below(double x) {
  const int m = __double2hiint(x) & 0x7FFFFFFF;
  return m < 0x38100000 ? 0.f : __int_as_float(m >= 0x47F00000 ? 0x7F800000 : (m - 0x38000000) << 3);
}

// ---------------------------------------------------------------- decision records
// A flagged slot's full decision, written by the decision kernels and read by
// the event kernel (slot-indexed arrays, touched only for flagged slots):
// x = K | flags << 8, y = product weight, z = new weight (axions) or the
// remaining weight (photons).
enum : uint32_t {
  DF_KEEP = 1u << 8, DF_ABSORBED = 1u << 9, DF_ABS_C = 1u << 10, DF_CAPPED = 1u << 11, DF_OVER = 1u << 12,
  DF_CAPPED_B = 1u << 13
};

// ---------------------------------------------------------------- decision kernels
// Bit masks: word (cell * W + s / 32), bit s % 32 flags slot s. Words are
// set by atomicOr (rare: electrons whose draw passes, axions and photons
// whose full decision changes something) and cleared by the event kernel
// after reading.

__device__ __forceinline__ void flag_quad(uint32_t* bits, int W, int cell, int q, uint32_t nib) {
  if (nib) atomicOr(bits + (size_t)cell * W + ((4 * q) >> 5), nib << ((4 * q) & 31));
}

// A persistent grid of warps. Warp i owns the chunks i, i + nwarps, ... of
// C consecutive cells and, per chunk and species, gives the chunk's quads
// to its lanes as one flat range (lane per quad, cell-major), so uneven counts
// still fill the lanes. Slots that the guards cannot clear go to the warp's
// own list in shared memory, which carries over from chunk to chunk and is
// decided 32 at a time: the out-of-line chain runs with full lanes and no CTA
// barrier is needed. List order does not matter: records are indexed by slot.
constexpr int kDecThreads = 256;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kListCap = 32 + 4 * 32;  // < 32 pending + one pass of flags

// Per-warp lists: {cell, slot, decision word(s)}.
struct DecLists {
  uint4 a[kDecWarps][kListCap];
  uint4 g[kDecWarps][kListCap];
};

// Flat quad range of a chunk: lanes < nc hold their cell's slot count n; on
// return lanes < nc hold their cell's first quad (qoff; the lanes beyond
// hold INT_MAX) and every lane the total. The starts stay in the lanes: a
// quad's cell is found by shuffles, which keeps the per-chunk state to two
// registers.
template <int C>
struct QuadRange {
  int qoff, total;
};

template <int C>
__device__ __forceinline__ QuadRange<C> quad_range(int n, int lane, int nc) {
  QuadRange<C> R;
  const int nq = lane < nc ? (n + 3) >> 2 : 0;
  R.qoff = warp_excl_scan(nq, &R.total);
  if (lane >= nc) R.qoff = 0x7fffffff;
  return R;
}

// Cell (in the chunk) of flat quad g: the last cell whose first quad is at
// or before g (binary search over the lanes' starts).
template <int C>
__device__ __forceinline__ int quad_cell(const QuadRange<C>& R, int g) {
  int lc = 0;
#pragma unroll
  for (int s = C / 2; s >= 1; s >>= 1) lc += g >= __shfl_sync(kFull, R.qoff, lc + s) ? s : 0;
  return lc;
}

// Appends this lane's flagged slots (bits of nib; words w0/w1 rotate with the
// slot) to a warp list of current length pend; returns the new length.
__device__ __forceinline__ int list_append(uint4* L, int pend, int cell, int slot0, uint32_t nib, uint4 w0, uint4 w1) {
  if (!__any_sync(kFull, nib != 0)) return pend;  // the common pass: nothing flagged
  int tot;
  int o = pend + warp_excl_scan(__popc(nib), &tot);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if ((nib >> j) & 1u) L[o++] = make_uint4((uint32_t)cell, (uint32_t)(slot0 + j), word(w0, j), word(w1, j));
  __syncwarp();
  return pend + tot;
}

// A full decision that changes nothing (no event, no cap hit, weight kept
// unchanged) leaves its slot unflagged: the event kernel never sees it.
template <bool SR>
__device__ __forceinline__ void axion_full(const StepArgs& A, uint4 it) {
  const int cell = (int)it.x;
  const long idx = (long)cell * A.a.cap + it.y;
  const AxionDecision d = axion_decide_slow<SR>(A, cell, A.mask, idx, it.z, it.w);
  const float w = d.w;
  uint32_t f = (uint32_t)d.K;
  if (d.keep) f |= DF_KEEP;
  if (d.absorbed) f |= DF_ABSORBED;
  if (d.abs_c) f |= DF_ABS_C;
  if (d.capped) f |= DF_CAPPED;
  if (d.over) f |= DF_OVER;
  const bool reduce = A.absorb_mode == 1 && (A.mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS));
  if (f == DF_KEEP && d.wnew == w && !reduce) return;
  A.recA[idx] = make_uint4(f, __float_as_uint(d.wprod), __float_as_uint(d.wnew), 0u);
  atomicOr(A.bitsA + (size_t)cell * A.Wa + (it.y >> 5), 1u << (it.y & 31));
}

template <bool SR>
__device__ __forceinline__ void photon_full(const StepArgs& A, uint4 it) {
  const int cell = (int)it.x;
  const long idx = (long)cell * A.g.cap + it.y;
  const PhotonDecision d = photon_decide_slow<SR>(A, cell, idx, it.z);
  uint32_t f = (uint32_t)d.K;
  if (d.wrem > 0.f) f |= DF_KEEP;
  if (d.capped) f |= DF_CAPPED;
  if (d.over) f |= DF_OVER;
  if (f == DF_KEEP) return;
  A.recG[idx] = make_uint4(f, __float_as_uint(d.wprod), __float_as_uint(d.wrem), 0u);
  atomicOr(A.bitsG + (size_t)cell * A.Wg + (it.y >> 5), 1u << (it.y & 31));
}

__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// Decides full batches of 32 from the top of a list; returns what is left.
template <bool AX, bool SR>
__device__ __forceinline__ int list_drain(const StepArgs& A, const uint4* L, int pend, int lane) {
  while (pend >= 32) {
    pend -= 32;
    const uint4 it = L[pend + lane];
    if (AX) axion_full<SR>(A, it);
    else photon_full<SR>(A, it);
  }
  __syncwarp();
  return pend;
}

// Electrons of a chunk (thermal-bath emission). With a common weight the
// decision is u > exp(-lambda) with lambda shared by the cell; the full
// decision of a flagged electron is a short Poisson inversion, taken here.
template <int C>
__device__ __forceinline__ void electron_chunk(const StepArgs& A, uint32_t step, int c0, int nc, int lane) {
  const int mask = A.mask;
  const bool eC = mask & AXPIC_CH_COMPTON, eB = mask & AXPIC_CH_BREMS;
  int n = 0, thr = 0;
  float wu = 0.f, lsum = 0.f, rcc = 0.f, rcb = 0.f;
  if (lane < nc) {
    const int c = c0 + lane;
    const float* rec = A.rec + (size_t)c * kRecLen;
    n = min(max(A.e.count[c], 0), A.e.cap);
    rcc = rec[R_CC];
    rcb = rec[R_CB];
    wu = A.mom[(size_t)c * kMomLen + M_WU];
    if (wu > 0.f) {
      float fac;
      bool cc = false, cb = false;
      const float lc = eC ? cap_lambda(wu * rcc, A.lam_cap, &fac, &cc) : 0.f;
      const float lb = eB ? cap_lambda(wu * rcb, A.lam_cap, &fac, &cb) : 0.f;
      lsum = lc + lb;
      // every electron of the cell has the capped mean (rare: counted here,
      // where the cap is found)
      if (cc || cb)
        atomicAdd(A.counters + (size_t)(blockIdx.x % A.ctr_rows) * kNumCounters + C_CAP,
                  (unsigned long long)n * ((unsigned)cc + (unsigned)cb));
      // u23(w) > F0 exactly when (w >> 9) > floor(F0 2^23 - 1/2): the
      // scaling and the subtraction are exact in binary32
      thr = (int)floorf(__fsub_rn(__fmul_rn(expf(-lsum), 8388608.0f), 0.5f));
    }
  }
  if (__all_sync(kFull, lane >= nc || (wu > 0.f && (((n + 3) >> 2) & 63) == 0))) {
    // every cell of the chunk has a common weight and whole passes of 64
    // quads: cell by cell, two quads per lane and pass (two independent
    // Philox chains in flight), the decision the integer compare alone
    for (int lc = 0; lc < nc; ++lc) {
      const int nn = __shfl_sync(kFull, n, lc);
      const int cthr = __shfl_sync(kFull, thr, lc);
      const float cls = __shfl_sync(kFull, lsum, lc);
      const int cell = c0 + lc;
      const uint32_t gcell = A.cell_base + (uint32_t)cell;
      const long cb = (long)cell * A.e.cap;
      const int nq = (nn + 3) >> 2;
      for (int q0 = 0; q0 < nq; q0 += 64) {
        uint4 r[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          r[h] = philox4x32_10(make_uint4(step, gcell, (uint32_t)(q0 + 32 * h + lane), S_EMIT_E << 24), A.rk);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = q0 + 32 * h + lane;
          const uint32_t m = max(max(r[h].x, r[h].y), max(r[h].z, r[h].w));
          if ((int)(m >> 9) <= cthr) continue;  // no slot of the quad emits
          const int nj = min(4, nn - 4 * q);
          uint32_t nib = 0;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t wj = word(r[h], j);
            if (j < nj && (int)(wj >> 9) > cthr) {
              A.recE[cb + 4 * q + j] = (uint32_t)poisson_inv(u23(wj), cls);
              nib |= 1u << j;
            }
          }
          flag_quad(A.bitsE, A.We, cell, q, nib);
        }
      }
    }
    return;
  }
  const QuadRange<C> R = quad_range<C>(n, lane, nc);
  if (__all_sync(kFull, lane >= nc || wu > 0.f)) {
    // every cell of the chunk has a common weight: the decision is the
    // integer compare alone. Two quads per lane and pass, so that two
    // independent Philox chains are in flight. Where the cells hold equally
    // many electrons (they never change) a quad's cell is a multiplication by
    // ceil(2^32 / nq), exact for the g < 32 nq <= 2^17 here.
    const int nq0 = __shfl_sync(kFull, (n + 3) >> 2, 0);
    const bool even = nq0 > 1 && nq0 <= 4096 && __all_sync(kFull, lane >= nc || (n + 3) >> 2 == nq0);
    const uint32_t magic = even ? 0xFFFFFFFFu / (uint32_t)nq0 + 1u : 0u;
    for (int g0 = 0; g0 < R.total; g0 += 64) {
      int lc[2], q[2];
      uint4 r[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int g = g0 + 32 * h + lane;
        if (even) {
          lc[h] = (int)__umulhi((uint32_t)g, magic);
          q[h] = g - lc[h] * nq0;
        } else {
          lc[h] = quad_cell(R, g);
          q[h] = g - __shfl_sync(kFull, R.qoff, lc[h]);
        }
        r[h] = philox4x32_10(make_uint4(step, A.cell_base + (uint32_t)(c0 + lc[h]), (uint32_t)q[h], S_EMIT_E << 24), A.rk);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int cthr = __shfl_sync(kFull, thr, lc[h]);
        const uint32_t m = max(max(r[h].x, r[h].y), max(r[h].z, r[h].w));
        const bool emits = g0 + 32 * h + lane < R.total && (int)(m >> 9) > cthr;
        if (!__any_sync(kFull, emits)) continue;  // the common pass: no slot of any quad emits
        const int nn = __shfl_sync(kFull, n, lc[h]);
        const float cls = __shfl_sync(kFull, lsum, lc[h]);
        if (!emits) continue;
        const int cell = c0 + lc[h];
        const int nj = min(4, nn - 4 * q[h]);
        const long b = (long)cell * A.e.cap + 4 * q[h];
        uint32_t nib = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t wj = word(r[h], j);
          if (j < nj && (int)(wj >> 9) > cthr) {
            A.recE[b + j] = (uint32_t)poisson_inv(u23(wj), cls);
            nib |= 1u << j;
          }
        }
        flag_quad(A.bitsE, A.We, cell, q[h], nib);
      }
    }
    return;
  }
  for (int g0 = 0; g0 < R.total; g0 += 32) {
    const int g = g0 + lane;
    const int lc = quad_cell(R, g);
    const int qb = __shfl_sync(kFull, R.qoff, lc);
    const int nn = __shfl_sync(kFull, n, lc);
    const float cwu = __shfl_sync(kFull, wu, lc);
    const int cthr = __shfl_sync(kFull, thr, lc);
    const float cls = __shfl_sync(kFull, lsum, lc);
    const float ccc = __shfl_sync(kFull, rcc, lc);
    const float ccb = __shfl_sync(kFull, rcb, lc);
    if (g >= R.total) continue;
    const int cell = c0 + lc;
    const int q = g - qb;
    const int nj = min(4, nn - 4 * q);
    const uint4 r = philox4x32_10(make_uint4(step, A.cell_base + (uint32_t)cell, (uint32_t)q, S_EMIT_E << 24), A.rk);
    const long b = (long)cell * A.e.cap + 4 * q;
    uint32_t nib = 0;
    if (cwu > 0.f) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t wj = word(r, j);
        if (j < nj && (int)(wj >> 9) > cthr) {
          A.recE[b + j] = (uint32_t)poisson_inv(u23(wj), cls);
          nib |= 1u << j;
        }
      }
    } else {
      const float rsum = ((eC ? ccc : 0.f) + (eB ? ccb : 0.f)) * 1.0001f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float wj = slot_w(A.e, b + j);
        const float lbnd = wj * rsum;
        if (j < nj && !(lbnd < A.lam_cap && u23(word(r, j)) <= 1.0f - lbnd - 1e-6f)) {
          float fac;
          bool cc = false, cb = false;
          const float l1 = eC ? cap_lambda(wj * ccc, A.lam_cap, &fac, &cc) : 0.f;
          const float l2 = eB ? cap_lambda(wj * ccb, A.lam_cap, &fac, &cb) : 0.f;
          uint32_t f = (uint32_t)poisson_inv(u23(word(r, j)), l1 + l2);
          if (cc) f |= DF_CAPPED;
          if (cb) f |= DF_CAPPED_B;
          A.recE[b + j] = f;
          nib |= 1u << j;
        }
      }
    }
    flag_quad(A.bitsE, A.We, cell, q, nib);
  }
}

// The photon and axion passes find the next pass's cells one pass ahead and
// prefetch its slots into L1: the loads were a third of the kernel's stalls,
// and held in registers instead they spill. 65,536 cells in 8 launches: 361
// -> 340 us, 196,000 cells of boxes 459 -> 417 us.

// Photons of a chunk present at the start of the step (gamma->a).
template <int C, bool SR>
__device__ __forceinline__ int photon_chunk(const StepArgs& A, uint32_t step, int c0, int nc, int lane, uint4* L,
                                            int pend) {
  int n = 0;
  float c_s = 0.f, ap = 0.f;
  if (lane < nc) {
    const int c = c0 + lane;
    const float* rec = A.rec + (size_t)c * kRecLen;
    const int cnt = min(max(A.g.count[c], 0), A.g.cap);
    n = A.use_snapshot ? min(A.photon_start[c], cnt) : cnt;
    c_s = kMeC2f * kMeC2f * rec[R_FOURK2];
    ap = conversion_kb(rec[R_AP], A.inv_w_a, A.guard_margin);
  }
  const QuadRange<C> R = quad_range<C>(n, lane, nc);
  int lcn = quad_cell(R, lane), qbn = __shfl_sync(kFull, R.qoff, lcn);
  for (int g0 = 0; g0 < R.total; g0 += 32) {
    const int g = g0 + lane;
    const int lc = lcn, qb = qbn;
    if (g0 + 32 < R.total) {
      lcn = quad_cell(R, g + 32);
      qbn = __shfl_sync(kFull, R.qoff, lcn);
      if (g + 32 < R.total) prefetch_l1(A.g.wp + (long)(c0 + lcn) * A.g.cap + 4 * (g + 32 - qbn));
    }
    const int nn = __shfl_sync(kFull, n, lc);
    const float cs = __shfl_sync(kFull, c_s, lc);
    const float ca = __shfl_sync(kFull, ap, lc);
    const int cell = c0 + lc;
    const int q = g - qb;
    uint32_t nib = 0;
    uint4 r = make_uint4(0, 0, 0, 0);
    if (g < R.total) {
      const int nj = min(4, nn - 4 * q);
      const long b = (long)cell * A.g.cap + 4 * q;
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = A.g.wp[b + j];
      r = philox4x32_10(make_uint4(step, A.cell_base + (uint32_t)cell, (uint32_t)q, S_PRIM_FWD << 24), A.rk);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float px = v[j].y, py = v[j].z, pz = v[j].w;
        const float p2 = px * px + py * py + pz * pz;
        nib |= (uint32_t)!no_conversion(v[j].x, p2, cs, ca, word(r, j), A.lam_cap) << j;
      }
      nib &= (1u << nj) - 1u;
    }
    pend = list_append(L, pend, cell, 4 * q, nib, r, r);
    pend = list_drain<false, SR>(A, L, pend, lane);
  }
  return pend;
}

// Axions of a chunk present at the start of the step: a->gamma and absorption.
template <int C, bool SR>
__device__ __forceinline__ int axion_chunk(const StepArgs& A, uint32_t step, int c0, int nc, int lane, uint4* L,
                                           int pend) {
  const int mask = A.mask;
  const bool prim = mask & AXPIC_CH_PRIMAKOFF;
  const bool bath = mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS);
  const bool all = A.absorb_mode == 1 && bath;  // weight reduction changes every axion
  int n = 0;
  const float half_am3 = 0.5f * A.brems_am3;
  float c_s = 0.f, apinv = 0.f;
  AbsorbBound ab = {0.f, 0.f, 0.f};
  if (lane < nc) {
    const int c = c0 + lane;
    const float* rec = A.rec + (size_t)c * kRecLen;
    n = min(max(A.a.count[c], 0), A.a.cap);
    c_s = kMeC2f * kMeC2f * rec[R_FOURK2];
    apinv = conversion_kb(A.cc.prim_mult * rec[R_AP], A.inv_w_gref, A.guard_margin);
    const float gm = 1.001f * A.guard_margin;
    ab = absorb_bound((mask & AXPIC_CH_COMPTON) ? rec[R_BC] * gm : 0.f,
                      (mask & AXPIC_CH_BREMS) ? rec[R_BB] * gm : 0.f, kMeC2f * rec[R_INVT],
                      A.brems_am3);
  }
  const QuadRange<C> R = quad_range<C>(n, lane, nc);
  int lcn = quad_cell(R, lane), qbn = __shfl_sync(kFull, R.qoff, lcn);
  for (int g0 = 0; g0 < R.total; g0 += 32) {
    const int g = g0 + lane;
    const int lc = lcn, qb = qbn;
    if (g0 + 32 < R.total) {
      lcn = quad_cell(R, g + 32);
      qbn = __shfl_sync(kFull, R.qoff, lcn);
      if (g + 32 < R.total) prefetch_l1(A.a.wp + (long)(c0 + lcn) * A.a.cap + 4 * (g + 32 - qbn));
    }
    const int nn = __shfl_sync(kFull, n, lc);
    const float cs = __shfl_sync(kFull, c_s, lc);
    const float cap_inv = __shfl_sync(kFull, apinv, lc);
    const AbsorbBound cab = {__shfl_sync(kFull, ab.bc1, lc), __shfl_sync(kFull, ab.bc2, lc),
                             __shfl_sync(kFull, ab.bb, lc)};
    const int cell = c0 + lc;
    const int q = g - qb;
    uint32_t nib = 0;
    uint4 rP = make_uint4(0, 0, 0, 0), rA = make_uint4(0, 0, 0, 0);
    if (g < R.total) {
      const int nj = min(4, nn - 4 * q);
      const uint32_t gcell = A.cell_base + (uint32_t)cell;
      const long b = (long)cell * A.a.cap + 4 * q;
      if (prim) rP = philox4x32_10(make_uint4(step, gcell, (uint32_t)q, S_PRIM_INV << 24), A.rk);
      if (bath) rA = philox4x32_10(make_uint4(step, gcell, (uint32_t)q, S_ABSORB << 24), A.rk);
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = A.a.wp[b + j];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float px = v[j].y, py = v[j].z, pz = v[j].w;
        const float p2 = (px * px + py * py + pz * pz) + A.mu2;  // E^2 (m_e c^2 units)
        bool fast = !all;
        if (prim) fast &= no_conversion(v[j].x, p2, cs, cap_inv, word(rP, j), A.lam_cap);
        if (bath) fast &= no_absorption(cab, half_am3, p2, word(rA, j));
        nib |= (uint32_t)!fast << j;
      }
      nib &= (1u << nj) - 1u;
    }
    pend = list_append(L, pend, cell, 4 * q, nib, rP, rA);
    pend = list_drain<true, SR>(A, L, pend, lane);
  }
  return pend;
}

// All decisions of a call in one launch. The photon decisions read the
// photons present at the start of the step: the absorb phase appends a->gamma
// products only in the event kernel.
enum : int { DK_ELECTRON = 1, DK_PHOTON = 2, DK_AXION = 4 };

#ifndef AXPIC_DEC_MIN_CTAS
#define AXPIC_DEC_MIN_CTAS 4
#endif

// The step index of this call: from the device counter when the step runs
// inside a replayed graph, else the launch argument.
__device__ __forceinline__ uint32_t step_of(const StepArgs& A) { return A.step_dev ? *A.step_dev : A.step; }

template <int C, bool SR>
__global__ void __launch_bounds__(kDecThreads, AXPIC_DEC_MIN_CTAS) decide_kernel(StepArgs A, int kinds) {
  wait_predecessor();
  __shared__ DecLists L;
  const int lane = lane_id(), wid = threadIdx.x >> 5;
  const uint32_t step = step_of(A);
  const int nwarps = gridDim.x * kDecWarps;
  const int nchunks = (A.ncells + C - 1) / C;
  const int cend = A.cell0 + A.ncells;
  int pa = 0, pg = 0;
  for (int ch = blockIdx.x * kDecWarps + wid; ch < nchunks; ch += nwarps) {
    const int c0 = A.cell0 + ch * C;
    const int nc = min(C, cend - c0);
    if (kinds & DK_ELECTRON) electron_chunk<C>(A, step, c0, nc, lane);
    if (kinds & DK_PHOTON) pg = photon_chunk<C, SR>(A, step, c0, nc, lane, L.g[wid], pg);
    if (kinds & DK_AXION) pa = axion_chunk<C, SR>(A, step, c0, nc, lane, L.a[wid], pa);
  }
  if (lane < pg) photon_full<SR>(A, L.g[wid][lane]);
  if (lane < pa) axion_full<SR>(A, L.a[wid][lane]);
}

// ---------------------------------------------------------------- feedback kernel
// Per cell: the exchange of this step plus the carried part; when it is
// representable in binary32 momenta the cell's electrons get the affine remap
// (Eqs. delta_def to b_def, affine_map) by a whole warp, measuring what was
// applied; then the temperature update (Eqs. Te_est, Te_relax) and the
// record's temperature half.

struct FbCell {
  double dE, dPx, dPy, dPz;  // this step's exchange
  double rE, rPx, rPy, rPz;  // carried exchange
  double T;
  double qE, qPx, qPy, qPz, s1d, bx, by, bz, vnd;
  float W, Px, Py, Pz, U2, var;
  float4 rc[4];
  int ne;
  bool has_x, has_res, need;
};

// What the feedback of a cell reads besides the exchange.
__device__ __forceinline__ void fb_load(const StepArgs& A, int cell, FbCell& f) {
  const double* rs = A.res + (size_t)cell * 4;
  f.rE = rs[0];
  f.rPx = rs[1];
  f.rPy = rs[2];
  f.rPz = rs[3];
  const float4* mom = reinterpret_cast<const float4*>(A.mom + (size_t)cell * kMomLen);
  const float4 m0 = mom[0], m1 = mom[1];
  static_assert(M_W == 0 && M_PZ == 3 && M_U2 == 4 && M_VAR == 5, "two loads");
  f.W = m0.x;
  f.Px = m0.y;
  f.Py = m0.z;
  f.Pz = m0.w;
  f.U2 = m1.x;
  f.var = m1.y;
  f.ne = min(max(A.e.count[cell], 0), A.e.cap);
  f.T = 0.0;
  f.rc[0] = f.rc[1] = f.rc[2] = f.rc[3] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (A.T_mode == 2) {
    f.T = A.T[cell];
    const float4* r4 = reinterpret_cast<const float4*>(A.rec + (size_t)cell * kRecLen);
    f.rc[0] = r4[0];
    f.rc[1] = r4[1];
    f.rc[2] = r4[2];
    f.rc[3] = r4[3];
  }
}

// The pending exchange and, when it needs a remap now, the map's s - 1 and b.
__device__ __forceinline__ void fb_prepare(FbCell& f) {
  f.has_x = nz64(f.dE) || nz64(f.dPx) || nz64(f.dPy) || nz64(f.dPz);
  f.has_res = nz64(f.rE) || nz64(f.rPx) || nz64(f.rPy) || nz64(f.rPz);
  f.need = false;
  f.qE = f.qPx = f.qPy = f.qPz = f.s1d = f.bx = f.by = f.bz = f.vnd = 0.0;
  if (!(f.has_x || f.has_res)) return;
  f.qE = f.rE;
  f.qPx = f.rPx;
  f.qPy = f.rPy;
  f.qPz = f.rPz;
  if (f.has_x) {
    f.qE += f.dE;
    f.qPx += f.dPx;
    f.qPy += f.dPy;
    f.qPz += f.dPz;
  }
  // Exchanges below 2^-22 of the cell's kinetic energy (or momentum spread)
  // cannot be represented by binary32 momenta; they stay pending.
  const float ekin = 0.5f * f.U2 * kMeC2f;
  const float prms = sqrtf(fmaxf(f.U2 * f.W, 0.f));
  const float tE = 2.384185791015625e-07f * ekin, tP = 2.384185791015625e-07f * prms;
  // Most are far below: told in binary32 with a margin of 1e-4 for the cut
  // magnitudes and the roundings, thresholds so small that a square could
  // underflow left to the test itself.
  const float aE = abs_below(f.qE), ax = abs_below(f.qPx), ay = abs_below(f.qPy), az = abs_below(f.qPz);
  if (tE >= 1e-30f && tP >= 1e-15f && 1.0001f * aE < tE && 1.0001f * sqrtf(ax * ax + ay * ay + az * az) < tP) return;
  f.need = f.W > 0.f && (fabsf((float)f.qE) >= tE ||
                         sqrtf((float)(f.qPx * f.qPx + f.qPy * f.qPy + f.qPz * f.qPz)) >= tP);
  if (!f.need) return;
  // Eqs. delta_def, dE_bulk, dE_th, var_new, s_def, b_def (mu = 1). Three
  // FP64 divisions and one square root (FP64 runs at a small fraction of the
  // FP32 rate): 1/W once, and S - 1 = t / (S + 1) with t = var_new / var - 1
  // formed from 2 dE_th without cancellation.
  const double Wd = f.W;
  const double iW = 1.0 / Wd;
  const double dx = f.qPx * iW, dy = f.qPy * iW, dz = f.qPz * iW;
  const double dEb = (2.0 * (dx * f.Px + dy * f.Py + dz * f.Pz) + Wd * (dx * dx + dy * dy + dz * dz)) * 0.5;
  const double dEth = f.qE * (1.0 / kMeC2) - dEb;
  f.vnd = f.var;
  if (f.var > 0.f) {
    const double var = f.var;
    f.vnd = fmax(0.0, var + 2.0 * dEth);
    const double t = (f.vnd > 0.0 ? 2.0 * dEth : -var) / var;
    const double S = sqrt(1.0 + t);
    f.s1d = t / (S + 1.0);
  }
  f.bx = -f.s1d * f.Px * iW + dx;
  f.by = -f.s1d * f.Py * iW + dy;
  f.bz = -f.s1d * f.Pz * iW + dz;
}

// Carry, moments, diagnostics, temperature and record once the remap (r;
// null when the cell was not remapped) is done. The record gets the
// closed-form prefactors of the new temperature; under the surrogate rate
// model the network's kernel, launched next, replaces them where it is
// trusted.
__device__ __forceinline__ void fb_finish(const StepArgs& A, int cell, const FbCell& f, const RemapOut* r) {
  double nrE = f.qE, nrPx = f.qPx, nrPy = f.qPy, nrPz = f.qPz, applied_E = 0.0;
  float var_new = f.var;
  if (r) {
    applied_E = r->applied_E;
    nrE = f.qE - r->applied_E;
    nrPx = f.qPx - r->apx;
    nrPy = f.qPy - r->apy;
    nrPz = f.qPz - r->apz;
    var_new = (float)f.vnd;
    float* mom = A.mom + (size_t)cell * kMomLen;
    mom[M_W] = r->mW;
    mom[M_PX] = r->mPx;
    mom[M_PY] = r->mPy;
    mom[M_PZ] = r->mPz;
    mom[M_U2] = r->mU2;
    mom[M_VAR] = fmaxf(0.f, r->mU2 - sum_sq(r->mPx, r->mPy, r->mPz) / r->mW);
  }
  if (f.has_x || r) {  // else the carried exchange is as it was
    double* rs = A.res + (size_t)cell * 4;
    rs[0] = nrE;
    rs[1] = nrPx;
    rs[2] = nrPy;
    rs[3] = nrPz;
  }
  if (A.diag_enable) {
    double* dg = A.diag + (size_t)cell * AXPIC_CELL_DIAG_LEN;
    dg[AXPIC_CD_DE] = f.dE;
    dg[AXPIC_CD_DPX] = f.dPx;
    dg[AXPIC_CD_DPY] = f.dPy;
    dg[AXPIC_CD_DPZ] = f.dPz;
    dg[AXPIC_CD_S_MINUS_1] = f.s1d;
    dg[AXPIC_CD_BX] = f.bx;
    dg[AXPIC_CD_BY] = f.by;
    dg[AXPIC_CD_BZ] = f.bz;
    dg[AXPIC_CD_VAR] = f.var;
    dg[AXPIC_CD_VAR_NEW] = f.need ? f.vnd : (double)f.var;
    dg[AXPIC_CD_W] = f.W;
    dg[AXPIC_CD_APPLIED_E] = applied_E;
    dg[AXPIC_CD_RES_E] = f.has_x || f.has_res ? nrE : 0.0;
    dg[AXPIC_CD_RES_PX] = f.has_x || f.has_res ? nrPx : 0.0;
    dg[AXPIC_CD_RES_PY] = f.has_x || f.has_res ? nrPy : 0.0;
    dg[AXPIC_CD_RES_PZ] = f.has_x || f.has_res ? nrPz : 0.0;
  }
  // temperature (Eqs. Te_est, Te_relax), then the record's temperature half;
  // T stays FP64, the relaxation step is formed in binary32 and added once
  if (A.T_mode == 2 && f.W > 0.f) {
    const float Tf = f32_of(f.T);
    const float Test = (kMeC2f / 3.0f) * var_new / f.W;
    const float dT = A.relax_r * (Test - Tf);
    double Tn = f.T + f64_of(dT);
    const float Tnf = Tf + dT;
    if (Tnf <= A.T_floor_f || Tnf >= A.T_ceil_f) Tn = fmin(fmax(Tn, A.T_floor), A.T_ceil);
    float rec[kRecLen];
    const float4* rc = f.rc;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      rec[4 * i] = rc[i].x;
      rec[4 * i + 1] = rc[i].y;
      rec[4 * i + 2] = rc[i].z;
      rec[4 * i + 3] = rc[i].w;
    }
    compute_temperature(A.cc, f32_of(Tn), rec);
    A.T[cell] = Tn;
    // the closed-form Primakoff prefactor (the network's may be there)
    if (A.rate_model == 2) rec[R_AP] = A.cc.k_AP * rec[R_SZ];
    float4* r4 = reinterpret_cast<float4*>(A.rec + (size_t)cell * kRecLen);
    r4[0] = make_float4(rec[0], rec[1], rec[2], rec[3]);
    r4[1] = make_float4(rec[4], rec[5], rec[6], rec[7]);
  }
}

// Thread per cell, every load issued first; a warp remaps the cells among
// its 32 whose exchange needs an affine remap, then each thread finishes its
// cell. No CTA barrier: the warps of a CTA never wait for one another's
// remaps. Bound by its loads where few cells are remapped (about one warp in
// twelve has one at 5 keV), by the FP64 sums and the chain of remaps where
// all are.
// * DENSE = false: a remap takes the whole warp; five CTAs an SM (96
//   registers; the remap path spills a little). 4.1 M cells at 5 keV: 217 us
//   with 20 FP64 adds a remap, 202 with the 6 of group_sum4; 224 with the
//   groups below in the same kernel (more spills). The FP64 units were busy
//   two thirds of the time: the test whether to remap first in binary32, the
//   conversions on the integer units, an unchanged carry not written and
//   16-byte loads take four steps of 4.1 M cells from 7.79 to 7.63 ms and of
//   0.9 M from 1.74 to 1.71 (conversions of the remap too: 7.66, spills).
// * DENSE = true (absorption by weight reduction, which takes energy from
//   every axion): cells of at most 64 electrons are remapped two or four side
//   by side, the next ones' electrons loaded meanwhile; four CTAs an SM
//   without spills. 112,095 cells of 64 electrons, all remapped: 306 us ->
//   125 us.
constexpr int kFeedbackThreads = 128;

template <bool DENSE>
__global__ void __launch_bounds__(kFeedbackThreads, DENSE ? 4 : 5) feedback_kernel(StepArgs A) {
  wait_predecessor();
  // a replayed graph takes its step index from the device counter: the last
  // kernel of the step advances it (no kernel of this launch reads it)
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (A.step_dev) *A.step_dev += 1u;
    *A.heavy_n = 0;  // the heavy cells' list of the next step
  }
  const int lane = threadIdx.x & 31;
  const int cell = A.cell0 + blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = cell < A.cell0 + A.ncells;
  FbCell f = {};
  if (valid) {
    double2* xb = reinterpret_cast<double2*>(A.xbuf + (size_t)cell * 4);
    const double2 x0 = xb[0], x1 = xb[1];
    f.dE = x0.x;
    f.dPx = x0.y;
    f.dPy = x1.x;
    f.dPz = x1.y;
    fb_load(A, cell, f);
    fb_prepare(f);
    if (f.has_x) xb[0] = xb[1] = make_double2(0.0, 0.0);
  }
  // the warp remaps its cells that need it: as many side by side as have a
  // lane for every quad of electrons
  RemapOut mine;
  const unsigned need = __ballot_sync(kFull, f.need);
  if (need) {
    const float s1 = (float)f.s1d, bx = (float)f.bx, by = (float)f.by, bz = (float)f.bz;
    const int nq = DENSE ? __reduce_max_sync(kFull, f.need ? (f.ne + 3) >> 2 : 0) : 32;
    if (DENSE && nq <= 8) mine = remap_cells<8>(A, need, cell, f.ne, s1, bx, by, bz);
    else if (DENSE && nq <= 16) mine = remap_cells<16>(A, need, cell, f.ne, s1, bx, by, bz);
    else mine = remap_cells<32>(A, need, cell, f.ne, s1, bx, by, bz);
  }
  if (valid) {
    fb_finish(A, cell, f, f.need ? &mine : nullptr);
    if (f.need) {
      atomicAdd(A.counters + C_REMAP, 1ull);
      atomicAdd(A.counters + C_REMAP_E, (unsigned long long)f.ne);
    }
  }
}


// ---------------------------------------------------------------- event kernel
// A warp takes consecutive cells, one a lane (32; 4 or 8 in a full step of few
// cells). Most cells have a handful of flagged slots: the lane then takes the
// cell alone, so the per-cell scans, counts and stores are shared by the warp's
// cells per instruction. A cell with more flagged slots in a phase than a lane
// takes is done by the whole warp: in a separate call after the lanes, in a full
// step by event_heavy_kernel.
//
// Per-warp shared scratch:
//   flagged-slot lists of one heavy cell (u16, full capacities; the removed
//   lists reuse them) and its removed-slot bits;
//   the lanes' lists: kLight entries per species and lane, entry i of lane l
//   at [32 i + l] (the removed list reuses it in place);
//   the 32 cells' mask rows, copied in by cp.async (row stride W | 1 words,
//   so that lanes reading their own rows hit distinct banks).

// Flagged slots per species up to which one lane takes a cell's phase
// (electrons: kLightE, each event with its own Philox block). Cells beyond go
// to a kernel of their own in a full step, whose chain of a few long cells
// every step waits for: with 8 and 4 a handful of 65,536 dense cells went
// there, with 16 and 8 hardly any (32 replayed steps: 6.60 -> 6.13 ms; 16,384
// cells, 8 steps: 1.14 -> 0.91 ms). The lists take 3 KB a warp.
constexpr int kLight = 16;
constexpr int kLightE = 8;
constexpr size_t kLaneListBytes = 3 * kLight * 32 * sizeof(uint16_t);

struct EvScratch {
  uint16_t *flA, *flG, *flE, *rmA, *rmG;
  uint32_t *rbA, *rbG;
  uint16_t* lt;
  uint32_t *rowA, *rowG, *rowE;  // null when some row is longer than 32 words
  double2* xs;                    // the lanes' exchange buffers, copied in by cp.async
  int sA, sG, sE;
};

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~size_t(15); }
__host__ __device__ inline int row_words(int cap) { return (cap + 31) / 32; }
__host__ __device__ inline bool rows_staged(int acap, int gcap, int ecap) {
  return row_words(acap) <= 32 && row_words(gcap) <= 32 && row_words(ecap) <= 32;
}

// What a kernel's warps keep there: the heavy cells' lists and bits, the lanes'
// lists, the mask rows with the exchange buffers. Lanes take cells only where
// the rows are staged, so there are no lanes' lists without them.
enum { EV_LISTS = 1, EV_LANES = 2, EV_ROWS = 4 };
__host__ __device__ constexpr int ev_parts(int phases) {
  return phases == PH_ABSORB ? EV_LISTS | EV_ROWS              // its lanes read the rows themselves
         : phases == PH_EMIT ? EV_LISTS | EV_LANES | EV_ROWS
                             : EV_LANES | EV_ROWS;             // heavy cells: event_heavy_kernel, EV_LISTS
}
__host__ __device__ inline size_t ev_list_bytes(int acap, int gcap, int ecap) {
  const size_t b = align16(2 * ((size_t)acap + (size_t)gcap + (size_t)ecap));
  return align16(b + 4 * (size_t)(row_words(acap) + row_words(gcap)));
}
__host__ __device__ inline size_t ev_row_bytes(int acap, int gcap, int ecap) {
  size_t b = 32 * 2 * sizeof(double2);
  if (rows_staged(acap, gcap, ecap))
    b += align16(4 * 32 * (size_t)((row_words(acap) | 1) + (row_words(gcap) | 1) + (row_words(ecap) | 1)));
  return b;
}
__host__ __device__ inline size_t ev_scratch_bytes(int acap, int gcap, int ecap, int parts) {
  return ((parts & EV_LISTS) ? ev_list_bytes(acap, gcap, ecap) : 0) +
         ((parts & EV_LANES) && rows_staged(acap, gcap, ecap) ? kLaneListBytes : 0) +
         ((parts & EV_ROWS) ? ev_row_bytes(acap, gcap, ecap) : 0);
}

template <int PARTS>
__device__ inline EvScratch ev_carve(unsigned char* base, int acap, int gcap, int ecap) {
  EvScratch s;
  uint16_t* h = reinterpret_cast<uint16_t*>(base);
  s.flA = h; h += acap;
  s.flG = h; h += gcap;
  s.flE = h; h += ecap;
  s.rmA = s.flA;
  s.rmG = s.flG;
  uint32_t* u = reinterpret_cast<uint32_t*>(base + align16(2 * ((size_t)acap + gcap + ecap)));
  s.rbA = u; u += row_words(acap);
  s.rbG = u;
  const bool staged = rows_staged(acap, gcap, ecap);
  size_t off = (PARTS & EV_LISTS) ? ev_list_bytes(acap, gcap, ecap) : 0;
  s.lt = reinterpret_cast<uint16_t*>(base + off);
  if ((PARTS & EV_LANES) && staged) off += kLaneListBytes;
  s.sA = row_words(acap) | 1;
  s.sG = row_words(gcap) | 1;
  s.sE = row_words(ecap) | 1;
  if ((PARTS & EV_ROWS) && staged) {
    s.rowA = reinterpret_cast<uint32_t*>(base + off);
    s.rowG = s.rowA + 32 * s.sA;
    s.rowE = s.rowG + 32 * s.sG;
    off += align16(4 * 32 * (size_t)(s.sA + s.sG + s.sE));
  } else {
    s.rowA = s.rowG = s.rowE = nullptr;
  }
  s.xs = reinterpret_cast<double2*>(base + off);
  return s;
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
// Waits for this thread's copies; the warp then synchronises to see all.
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Turns one bit-mask word per lane (words [w0, w0 + 32) of a row covering
// [0, n)) into the ascending list of flagged slots; returns the new length.
__device__ __forceinline__ int list_flags(uint32_t v, int wi, int nw, int n, uint16_t* list, int total) {
  if (wi == nw - 1 && (n & 31)) v &= (1u << (n & 31)) - 1u;  // bits beyond n never count
  int tot;
  int at = total + warp_excl_scan(__popc(v), &tot);
  while (v) {
    const int bpos = __ffs(v) - 1;
    v &= v - 1u;
    list[at++] = (uint16_t)(32 * wi + bpos);
  }
  return total + tot;
}

// Writes the flagged slots of a mask row covering [0, n) to `list` in
// ascending order (warp-wide) and returns their number. The row is the
// staged copy, or the global row itself, which is then cleared (clr).
__device__ __noinline__ int gather_row(const uint32_t* row, uint32_t* clr, int n, uint16_t* list) {
  const int lane = lane_id();
  const int nw = (n + 31) >> 5;
  int total = 0;
  for (int w0 = 0; w0 < nw; w0 += 32) {
    const int wi = w0 + lane;
    const uint32_t v = wi < nw ? row[wi] : 0u;
    if (clr && v) clr[wi] = 0u;
    total = list_flags(v, wi, nw, n, list, total);
  }
  return total;
}

// Tail fill by the warp with the ascending removed list: holes are the
// removed slots below n_surv, movers the kept slots at or beyond it, matched
// in order.
__device__ __noinline__ void compact_tail(const SpeciesPtrs& s, long base, const uint16_t* rm, const uint32_t* rb,
                                          int n_surv, int n) {
  const int lane = lane_id();
  const unsigned lt = (1u << lane) - 1u;
  int run = 0;
  for (int b0 = n_surv; b0 < n; b0 += 32) {
    const int i = b0 + lane;
    const bool mv = i < n && !bit(rb, i);
    const unsigned m = __ballot_sync(kFull, mv);
    if (mv) {
      const long src = base + i;
      const long dst = base + rm[run + __popc(m & lt)];
      s.wp[dst] = s.wp[src];
      s.xyz[dst] = s.xyz[src];
    }
    run += __popc(m);
  }
}

// A flagged slot with its decision record and the fields its outcome may
// need, loaded in one round trip.
struct AxItem {
  uint4 r;
  float w, px, py, pz, x, y, z;
  int slot;
};
struct PhItem {
  uint4 r;
  float px, py, pz, x, y, z;
  int slot;
};
struct ElItem {
  uint32_t f;
  float w, x, y, z;
  int slot;
};

__device__ __forceinline__ AxItem ax_load(const StepArgs& A, long base, int slot) {
  AxItem t;
  t.slot = slot;
  t.r = make_uint4(0, 0, 0, 0);
  t.w = t.px = t.py = t.pz = t.x = t.y = t.z = 0.f;
  if (slot >= 0) {
    const long src = base + slot;
    t.r = A.recA[src];
    const float4 v = A.a.wp[src];
    t.w = v.x;
    t.px = v.y;
    t.py = v.z;
    t.pz = v.w;
    const float4 r = A.a.xyz[src];
    t.x = r.x;
    t.y = r.y;
    t.z = r.z;
  }
  return t;
}

__device__ __forceinline__ PhItem ph_load(const StepArgs& A, long base, int slot) {
  PhItem t;
  t.slot = slot;
  t.r = make_uint4(0, 0, 0, 0);
  t.px = t.py = t.pz = t.x = t.y = t.z = 0.f;
  if (slot >= 0) {
    const long src = base + slot;
    t.r = A.recG[src];
    const float4 v = A.g.wp[src];
    t.px = v.y;
    t.py = v.z;
    t.pz = v.w;
    const float4 r = A.g.xyz[src];
    t.x = r.x;
    t.y = r.y;
    t.z = r.z;
  }
  return t;
}

__device__ __forceinline__ ElItem el_load(const StepArgs& A, long base, int slot, float wu) {
  ElItem t;
  t.slot = slot;
  t.f = 0u;
  t.w = wu;
  t.x = t.y = t.z = 0.f;
  if (slot >= 0) {
    const long src = base + slot;
    t.f = A.recE[src];
    const float4 r = A.e.xyz[src];
    t.x = r.x;
    t.y = r.y;
    t.z = r.z;
    if (wu <= 0.f) t.w = slot_w(A.e, src);
  }
  return t;
}

// ---------------------------------------------------------------- per-slot outcomes
// Shared by the lane and warp paths. Output order is the method's: photon
// products of a->gamma after the photons present, axion products of gamma->a
// after the surviving axions, then the thermal-bath products in electron then
// event order; removed slots are refilled from the tail.

// A flagged axion: counters, exchange, new weight. Returns K; *removed tells
// whether the slot leaves the slab.
// The momentum of an a->gamma photon: the axion's direction with the axion's
// total energy E (its own momentum when massless).
__device__ __forceinline__ float3 photon_from_axion(const StepArgs& A, float px, float py, float pz) {
  if (A.mu <= 0.f) return make_float3(px, py, pz);
  const float p2 = px * px + py * py + pz * pz;
  const float f = __fdiv_rn(sqrtf(p2 + A.mu2), sqrtf(p2));
  return make_float3(px * f, py * f, pz * f);
}

__device__ __forceinline__ int axion_outcome(const StepArgs& A, const AxItem& t, long abase, bool bath,
                                             const Cnt& cnt, Lane64& x64, bool* removed) {
  const int K = t.r.x & 0xFF;
  const float wprod = __uint_as_float(t.r.y);
  const float wnew = __uint_as_float(t.r.z);
  const float om = sqrtf((t.px * t.px + t.py * t.py + t.pz * t.pz) + A.mu2) * kMeC2f;  // E
  cnt.add(C_CAP, (t.r.x & DF_CAPPED) ? 1u : 0u);
  cnt.add(C_CLAMP, (t.r.x & DF_OVER) ? 1u : 0u);
  cnt.add(C_EV_PINV, (unsigned)K);
  if (t.r.x & DF_ABSORBED) {
    x64.add((double)wnew, om, t.px, t.py, t.pz);
    cnt.add((t.r.x & DF_ABS_C) ? C_ABS_C : C_ABS_B, 1);
  } else if (A.absorb_mode == 1 && bath) {
    // weight reduction: the lost weight's energy goes to the plasma
    float wrem = t.w;
    if (K > 0) wrem = (t.r.x & DF_OVER) ? 0.f : __fsub_rn(t.w, __fmul_rn((float)K, wprod));
    x64.add((double)wrem - (double)wnew, om, t.px, t.py, t.pz);
  }
  *removed = !(t.r.x & DF_KEEP);
  if (!*removed && wnew != t.w) slot_w(A.a, abase + t.slot) = wnew;
  return K;
}

// A flagged photon: counters and the remaining weight. Returns K.
__device__ __forceinline__ int photon_outcome(const StepArgs& A, const PhItem& t, long gbase, const Cnt& cnt,
                                              bool* removed) {
  const int K = t.r.x & 0xFF;
  cnt.add(C_CAP, (t.r.x & DF_CAPPED) ? 1u : 0u);
  cnt.add(C_CLAMP, (t.r.x & DF_OVER) ? 1u : 0u);
  cnt.add(C_EV_P, (unsigned)K);
  *removed = !(t.r.x & DF_KEEP);
  if (K && !*removed) slot_w(A.g, gbase + t.slot) = __uint_as_float(t.r.z);
  return K;
}

// Slot of the i-th new axion of an emit phase: the freed slots holes[0,
// nholes) (ascending, entries `stride` apart) first, then from base on. A
// separate emit call has no freed slots (base: the axion count); a full step
// reuses the slots its absorb phase freed (base: the count at its start).
struct AxDest {
  const uint16_t* holes;
  int nholes, stride, base;
  __device__ __forceinline__ int at(int i) const {
    return i < nholes ? (int)holes[stride * i] : base + (i - nholes);
  }
};

// The K axion products of a gamma->a event, new axions i0 .. i0 + K - 1.
__device__ __forceinline__ void gamma_products(const StepArgs& A, const PhItem& t, long abase, const AxDest& D,
                                               int i0, int K, const Cnt& cnt) {
  const float wprod = __uint_as_float(t.r.y);
  const float pm = sqrtf(sum_sq(t.px, t.py, t.pz));
  const float om = pm * kMeC2f;
  // a massive axion takes E = omega and momentum beta p_gamma
  const float beta = A.mu > 0.f ? axion_beta(pm, A.mu2) : 1.0f;
  const float ax = A.mu > 0.f ? t.px * beta : t.px, ay = A.mu > 0.f ? t.py * beta : t.py,
              az = A.mu > 0.f ? t.pz * beta : t.pz;
  for (int k = 0; k < K; ++k) {
    const int dst = D.at(i0 + k);
    if (dst < A.a.cap) {
      write_particle(A.a, abase + dst, wprod, ax, ay, az, t.x, t.y, t.z);
      if (A.tally_enable) tally_add(A, 0, wprod, om);
    } else {
      cnt.add(C_DROP, 1);
    }
  }
}

// x from the 31 quantiles of channel c (end points 0.05 and 20), linear
// between quantiles: the cell's spectral record's, or the network's for every
// cell. Rate models 1 and 2 have their own instances of the event kernels: out
// of line in one instance for all it cost 60 bytes of spills and 15 % of the
// kernel (450 -> 517 us at 4.1 M cells).
__device__ __forceinline__ float sr_sample_x(const StepArgs& A, int cell, int ch, float u) {
  const float t = u * 32.f;
  const int j = min((int)t, 31);
  const float f = t - (float)j;
  const int o = 96 + ch * kSrKnots + j;
  float x0, x1;
  if (cell_has_sr(A, cell)) {
    float rec[kRecLen];
    load_rec(A, cell, rec);
    const CellSpectrum sr = cell_spectrum(A, rec);
    x0 = j == 0 ? 0.05f : sr.at(o - 1);
    x1 = j == 31 ? 20.0f : sr.at(o);
  } else {
    x0 = j == 0 ? 0.05f : A.ra.uni[o - 1];
    x1 = j == 31 ? 20.0f : A.ra.uni[o];
  }
  return fmaf(f, x1 - x0, x0);
}

// The events of a flagged electron (thermal-bath emission), new axions i0
// on: event k takes cos theta, phi, energy and channel from one Philox
// block. A massive axion's event is kept when the channel uniform, rescaled
// inside its channel's interval, is below beta(E) (thinning; every event is
// kept when massless). Returns the kept events; WRITE = false only counts
// them (the warp path's offsets need the counts first).
template <bool WRITE, bool SR>
__device__ __forceinline__ int electron_events(const StepArgs& A, uint32_t step, int cell, const ElItem& t,
                                               long abase, const AxDest& D, int i0, float r_cc, float r_cb,
                                               float r_T, float wu, const Cnt& cnt, Lane64& x64) {
  const int K = t.f & 0xFF;
  if (WRITE && wu <= 0.f) cnt.add(C_CAP, ((t.f & DF_CAPPED) ? 1u : 0u) + ((t.f & DF_CAPPED_B) ? 1u : 0u));
  if (!K) return 0;
  const bool eC = A.mask & AXPIC_CH_COMPTON, eB = A.mask & AXPIC_CH_BREMS;
  float facC = 1.f, facB = 1.f;
  bool cc = false, cb = false;
  const float lc = eC ? cap_lambda(t.w * r_cc, A.lam_cap, &facC, &cc) : 0.f;
  const float lb = eB ? cap_lambda(t.w * r_cb, A.lam_cap, &facB, &cb) : 0.f;
  const float fracC = lc / (lc + lb);
  const float wvC = cc ? A.w_a * facC : A.w_a;
  const float wvB = cb ? A.w_a * facB : A.w_a;
  const uint32_t gcell = A.cell_base + (uint32_t)cell;
  // the energies: the exact inverse CDFs (closed forms), the cell's spectral
  // record, or the network's cell-independent quantiles
  int kept = 0;
  for (int k = 0; k < K; ++k) {
    const uint4 r = philox4x32_10(make_uint4(step, gcell, (uint32_t)t.slot, (S_EV_E << 24) | (uint32_t)k), A.rk);
    const float uc = u23(r.w);
    const bool isC = uc < fracC;
    const float E = (SR ? sr_sample_x(A, cell, isC ? 1 : 2, u23(r.z))
                        : icdf_lookup(A.tables + (isC ? TAB_COMPTON : TAB_BREMS) * kTableN, u23(r.z))) *
                    r_T;
    float pm = E * kInvMeC2f;
    if (A.mu > 0.f) {
      const float ut = isC ? __fdiv_rn(uc, fracC) : __fdiv_rn(__fsub_rn(uc, fracC), __fsub_rn(1.0f, fracC));
      const float beta = axion_beta(pm, A.mu2);
      if (!(ut < beta)) continue;  // thinned: below the threshold always
      pm = pm * beta;               // |p| = sqrt(E^2 - m_a^2)
    }
    if (WRITE) {
      const float3 dv = iso_dir(u23(r.x), u23(r.y));
      const float wv = isC ? wvC : wvB;
      const float px = pm * dv.x, py = pm * dv.y, pz = pm * dv.z;
      const int dst = D.at(i0 + kept);
      if (dst < A.a.cap) {
        write_particle(A.a, abase + dst, wv, px, py, pz, t.x, t.y, t.z);
        if (A.tally_enable) tally_add(A, isC ? 1 : 2, wv, E);
      } else {
        cnt.add(C_DROP, 1);
      }
      x64.add(-(double)wv, E, px, py, pz);
      cnt.add(isC ? C_EV_C : C_EV_B, 1);
    }
    ++kept;
  }
  return kept;
}

// ---------------------------------------------------------------- warp path
struct PhaseOut {
  int na, ng, np;  // axion and photon counts, new axions
  double x[4];
  bool any;
};

__device__ __forceinline__ void reduce_out(const Lane64& x64, PhaseOut* out) {
  out->any = __any_sync(kFull, x64.any);
  out->x[0] = out->x[1] = out->x[2] = out->x[3] = 0.0;
  if (out->any) {
    out->x[0] = warp_sum_d(x64.dE);
    out->x[1] = warp_sum_d(x64.dPx);
    out->x[2] = warp_sum_d(x64.dPy);
    out->x[3] = warp_sum_d(x64.dPz);
  }
}

// Absorb phase of one cell by the warp: a->gamma products, absorption and
// weight reduction, then (fill) the axion tail fill; without it the freed
// slots stay listed, ascending, in S.rmA (marked in S.rbA). sb is the warp's
// scratch, carved here again: a scratch descriptor passed by reference to an
// out-of-line call would live in local memory, written by every thread of
// the kernel.
__device__ __noinline__ void absorb_warp(const StepArgs& A, int cell, unsigned char* sb, const uint32_t* row,
                                         uint32_t* clr, const Cnt cnt, int na_start, int ng_start, bool fill,
                                         PhaseOut* out) {
  const EvScratch S = ev_carve<EV_LISTS>(sb, A.a.cap, A.g.cap, A.e.cap);
  const int lane = lane_id();
  const unsigned lt = (1u << lane) - 1u;
  const bool bath = A.mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS);
  const long abase = (long)cell * A.a.cap;
  const long gbase = (long)cell * A.g.cap;
  const int nfl = gather_row(row, clr, na_start, S.flA);
  for (int i = lane; i < (na_start + 31) / 32; i += 32) S.rbA[i] = 0u;
  __syncwarp();
  Lane64 x64;
  int run = 0, nrm = 0;
  for (int i0 = 0; i0 < nfl; i0 += 32) {
    const AxItem t = ax_load(A, abase, i0 + lane < nfl ? (int)S.flA[i0 + lane] : -1);
    int K = 0;
    bool removed = false;
    if (t.slot >= 0) K = axion_outcome(A, t, abase, bath, cnt, x64, &removed);
    int tot;
    int off = run + warp_excl_scan(K, &tot);
    const float wprod = __uint_as_float(t.r.y);
    const float3 pg = photon_from_axion(A, t.px, t.py, t.pz);
    for (int k = 0; k < K; ++k, ++off) {
      const int dst = ng_start + off;
      if (dst < A.g.cap) write_particle(A.g, gbase + dst, wprod, pg.x, pg.y, pg.z, t.x, t.y, t.z);
      else cnt.add(C_DROP, 1);
    }
    run += tot;
    const unsigned m = __ballot_sync(kFull, removed);
    if (removed) {
      S.rmA[nrm + __popc(m & lt)] = (uint16_t)t.slot;
      atomicOr(&S.rbA[t.slot >> 5], 1u << (t.slot & 31));
    }
    nrm += __popc(m);
  }
  reduce_out(x64, out);
  __syncwarp();
  if (fill && nrm > 0) compact_tail(A.a, abase, S.rmA, S.rbA, na_start - nrm, na_start);
  out->na = na_start - nrm;
  out->ng = min(ng_start + run, A.g.cap);
  out->np = 0;
}

// Emit phase of one cell by the warp: gamma->a, the thermal-bath events (new
// axions placed by D), then the photon tail fill (a->gamma products
// included).
template <bool SR>
__device__ __noinline__ void emit_warp(const StepArgs& A, uint32_t step, int cell, unsigned char* sb,
                                       const uint32_t* rowG, uint32_t* clrG, const uint32_t* rowE, uint32_t* clrE,
                                       const Cnt cnt, AxDest D, int ng_tot, int ng0, int ne, float wu, float r_cc,
                                       float r_cb, float r_T, PhaseOut* out) {
  const EvScratch S = ev_carve<EV_LISTS>(sb, A.a.cap, A.g.cap, A.e.cap);
  const int lane = lane_id();
  const unsigned lt = (1u << lane) - 1u;
  const long abase = (long)cell * A.a.cap;
  const long gbase = (long)cell * A.g.cap;
  const long ebase = (long)cell * A.e.cap;
  const int nflG = rowG ? gather_row(rowG, clrG, ng0, S.flG) : 0;
  const int nflE = rowE ? gather_row(rowE, clrE, ne, S.flE) : 0;
  for (int i = lane; i < (ng_tot + 31) / 32; i += 32) S.rbG[i] = 0u;
  __syncwarp();
  int run = 0, nrm = 0;
  for (int i0 = 0; i0 < nflG; i0 += 32) {
    const PhItem t = ph_load(A, gbase, i0 + lane < nflG ? (int)S.flG[i0 + lane] : -1);
    int K = 0;
    bool removed = false;
    if (t.slot >= 0) K = photon_outcome(A, t, gbase, cnt, &removed);
    int tot;
    const int off = run + warp_excl_scan(K, &tot);
    if (K) gamma_products(A, t, abase, D, off, K, cnt);
    run += tot;
    const unsigned m = __ballot_sync(kFull, removed);
    if (removed) {
      S.rmG[nrm + __popc(m & lt)] = (uint16_t)t.slot;
      atomicOr(&S.rbG[t.slot >> 5], 1u << (t.slot & 31));
    }
    nrm += __popc(m);
  }
  Lane64 x64;
  for (int i0 = 0; i0 < nflE; i0 += 32) {
    const ElItem t = el_load(A, ebase, i0 + lane < nflE ? (int)S.flE[i0 + lane] : -1, wu);
    int K = t.slot >= 0 ? (int)(t.f & 0xFF) : 0;
    if (A.mu > 0.f && K > 0)  // massive axions: the kept events, before the offsets
      K = electron_events<false, SR>(A, step, cell, t, abase, D, 0, r_cc, r_cb, r_T, wu, cnt, x64);
    int tot;
    const int off = run + warp_excl_scan(K, &tot);
    if (t.slot >= 0) electron_events<true, SR>(A, step, cell, t, abase, D, off, r_cc, r_cb, r_T, wu, cnt, x64);
    run += tot;
  }
  reduce_out(x64, out);
  __syncwarp();
  if (nrm > 0) compact_tail(A.g, gbase, S.rmG, S.rbG, ng_tot - nrm, ng_tot);
  out->na = min(D.base - D.nholes + run, A.a.cap);
  out->ng = ng_tot - nrm;
  out->np = run;
}

// ---------------------------------------------------------------- lane path
// Counts the flagged slots of a staged mask row in [0, n) and lists the
// first kLight of them (ascending, stride 32); *nz gets the nonzero words.
__device__ __forceinline__ int scan_row(const uint32_t* row, int n, uint16_t* list, uint32_t* nz) {
  const int nw = (n + 31) >> 5;
  int c = 0;
  uint32_t m = 0u;
  for (int w = 0; w < nw; ++w) {
    uint32_t v = row[w];
    if (v) {
      m |= 1u << w;
      if (w == nw - 1 && (n & 31)) v &= (1u << (n & 31)) - 1u;
      while (v) {
        if (c < kLight) list[32 * c] = (uint16_t)(32 * w + __ffs(v) - 1);
        ++c;
        v &= v - 1u;
      }
    }
  }
  *nz = m;
  return c;
}

// The flagged slots of a staged mask row in [0, n), and its nonzero words.
__device__ __forceinline__ int count_row(const uint32_t* row, int n, uint32_t* nz) {
  const int nw = (n + 31) >> 5;
  int c = 0;
  uint32_t m = 0u;
  for (int w = 0; w < nw; ++w) {
    uint32_t v = row[w];
    if (v) m |= 1u << w;
    if (w == nw - 1 && (n & 31)) v &= (1u << (n & 31)) - 1u;
    c += __popc(v);
  }
  *nz = m;
  return c;
}

// Clears the nonzero words of a cell's global mask row.
__device__ __forceinline__ void clear_row(uint32_t* bits, int W, int cell, uint32_t nz) {
  uint32_t* row = bits + (size_t)cell * W;
  while (nz) {
    row[__ffs(nz) - 1] = 0u;
    nz &= nz - 1u;
  }
}

// Tail fill by one lane: the removed slots rm[0, nrm) (ascending) below
// n_surv are refilled, in order, by the kept slots of [n_surv, n). The first
// mover can be loaded ahead and written later; fill_rest moves the others.
struct FillIt {
  int h, j, i, m;  // holes, next removed entry at or past the scan, scan position, movers done
};
struct Mover {
  float w, px, py, pz, x, y, z;
  int dst;
};

__device__ __forceinline__ FillIt fill_begin(const uint16_t* rm, int nrm, int n_surv) {
  FillIt it;
  it.h = 0;
  while (it.h < nrm && rm[32 * it.h] < n_surv) ++it.h;
  it.j = it.h;
  it.i = n_surv;
  it.m = 0;
  return it;
}

// Source slot of the next mover (the caller checks it.m < it.h).
__device__ __forceinline__ int fill_next(const uint16_t* rm, int nrm, FillIt& it) {
  while (it.j < nrm && rm[32 * it.j] == it.i) {
    ++it.j;
    ++it.i;
  }
  return it.i++;
}

__device__ __forceinline__ Mover mover_load(const SpeciesPtrs& sp, long base, int src, int dst) {
  Mover v;
  v.dst = dst;
  if (dst >= 0) {
    const long q = base + src;
    const float4 r = sp.wp[q];
    v.w = r.x;
    v.px = r.y;
    v.py = r.z;
    v.pz = r.w;
    const float4 u = sp.xyz[q];
    v.x = u.x;
    v.y = u.y;
    v.z = u.z;
  }
  return v;
}

__device__ __forceinline__ void mover_store(const SpeciesPtrs& sp, long base, const Mover& v) {
  if (v.dst >= 0) write_particle(sp, base + v.dst, v.w, v.px, v.py, v.pz, v.x, v.y, v.z);
}

__device__ __forceinline__ void fill_rest(const SpeciesPtrs& sp, long base, const uint16_t* rm, int nrm, FillIt& it) {
  while (it.m < it.h) {
    Mover v[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      int src = 0, dst = -1;
      if (it.m < it.h) {
        src = fill_next(rm, nrm, it);
        dst = rm[32 * it.m++];
      }
      v[t] = mover_load(sp, base, src, dst);
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) mover_store(sp, base, v[t]);
  }
}

// One cell by one lane: its emit phase, or the full step (doA: the new axions
// of the emit phase reuse the axion slots the absorb phase freed). Round
// trips: the first flagged axion and photon together; the first photon tail
// mover under the thermal-bath events. Longer lists take further round trips.
// Each loop stands once: with the first items and
// movers handled apart from the rest the kernel's code was half again as
// large and stalled on instruction fetches (4.1 M cells at 5 keV: 569 us, now
// 450; two tail movers at a time there, 529 with four). Every flagged axion is read before a new axion is written over
// a freed slot.
struct LaneCell {
  int na, ng;       // in: counts at the start of the phase(s); out: final counts
  int ng0, ne;      // photons eligible for gamma->a, electrons
  int nflA, nflG, nflE;
  float wu, r_cc, r_cb, r_T;
};

template <bool SR>
__device__ __forceinline__ void cell_lane(const StepArgs& A, uint32_t step, int cell, bool doA, uint16_t* lA,
                                          uint16_t* lG, const uint16_t* lE, LaneCell& L, const Cnt& cnt, Lane64& xa,
                                          Lane64& xe) {
  const bool bath = A.mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS);
  const long abase = (long)cell * A.a.cap;
  const long gbase = (long)cell * A.g.cap;
  const long ebase = (long)cell * A.e.cap;
  const int nA = doA ? L.nflA : 0;
  const int nG = L.nflG;
  const int nE = L.nflE;
  AxItem ta = ax_load(A, abase, nA > 0 ? (int)lA[0] : -1);
  PhItem tg = ph_load(A, gbase, nG > 0 ? (int)lG[0] : -1);

  // absorb: a->gamma products after the photons present
  int ng = L.ng, nrmA = 0;
  for (int i = 0; i < nA; ++i) {
    bool removed;
    const int K = axion_outcome(A, ta, abase, bath, cnt, xa, &removed);
    if (K > 0) {
      const float wprod = __uint_as_float(ta.r.y);
      const float3 pg = photon_from_axion(A, ta.px, ta.py, ta.pz);
      for (int k = 0; k < K; ++k) {
        const int dst = ng + k;
        if (dst < A.g.cap) write_particle(A.g, gbase + dst, wprod, pg.x, pg.y, pg.z, ta.x, ta.y, ta.z);
        else cnt.add(C_DROP, 1);
      }
      ng += K;
    }
    if (removed) lA[32 * nrmA++] = (uint16_t)ta.slot;
    if (i + 1 < nA) ta = ax_load(A, abase, lA[32 * (i + 1)]);
  }
  ng = min(ng, A.g.cap);

  // emit: new axions, first the gamma->a products
  const AxDest D{lA, nrmA, 32, L.na};
  int NP = 0, nrmG = 0;
  for (int i = 0; i < nG; ++i) {
    bool removed;
    const int K = photon_outcome(A, tg, gbase, cnt, &removed);
    if (K) gamma_products(A, tg, abase, D, NP, K, cnt);
    NP += K;
    if (removed) lG[32 * nrmG++] = (uint16_t)tg.slot;
    if (i + 1 < nG) tg = ph_load(A, gbase, lG[32 * (i + 1)]);
  }
  // the first photon tail mover (a->gamma products included), loaded under
  // the thermal-bath events
  FillIt fg = fill_begin(lG, nrmG, ng - nrmG);
  Mover mg;
  {
    int src = 0, dst = -1;
    if (fg.h > 0) {
      src = fill_next(lG, nrmG, fg);
      dst = lG[0];
      fg.m = 1;
    }
    mg = mover_load(A.g, gbase, src, dst);
  }
  for (int i = 0; i < nE; ++i) {
    const ElItem t = el_load(A, ebase, lE[32 * i], L.wu);
    NP += electron_events<true, SR>(A, step, cell, t, abase, D, NP, L.r_cc, L.r_cb, L.r_T, L.wu, cnt, xe);
  }
  const int na = min(D.base - D.nholes + NP, A.a.cap);
  if (NP < nrmA) {
    // freed slots left over: closed from the tail (their movers lie beyond
    // every slot a new axion took)
    FillIt fr = fill_begin(lA + 32 * NP, nrmA - NP, na);
    fill_rest(A.a, abase, lA + 32 * NP, nrmA - NP, fr);
  }
  mover_store(A.g, gbase, mg);
  fill_rest(A.g, gbase, lG, nrmG, fg);
  ng -= nrmG;
  L.na = na;
  L.ng = ng;
}

// The absorb phase of a separate call by one lane: the cell's flagged axions
// in slot order straight from its staged mask row (any number of them, so no
// list is needed), the next one's record and momentum loaded while one is
// decided. Its position is loaded with them where most flagged axions convert
// (AHEAD), else only if it converts. Words of the row are cleared as they are
// read and take the removed slots' bits, which the tail fill then follows.
//
// Which cells (by the cell's own count and the launch's cells, so that the sums'
// order does not depend on the cells beside it):
// * Weight reduction flags every axion of every cell. A lane takes 0.7 to 0.9 us
//   an axion, the warp 4 us a cell, 6 beyond 32 axions: 5 axions a cell of
//   the warp, at most kManyAbsorb. A call of absorption, us, all cells by the
//   warp / with a limit of 64 / with this one:
//     cells   axions 24            60             70             140
//     1        20   29   17     24   56   19    26   20   20     35   25   25
//     16       73   35   36    101   71   72   120  112   83    167  155  155
//     4,000   137   41   41    193   83   84   231  225   96    326  314  179
//     112,000 423  154  155    650  359  359   762  741  412   1156 1119  798
//   (without kManyAbsorb 4,000 cells of 1,000 axions with conversions take
//   1865 instead of 1855 and 64 cells of 300 427 instead of 515.)
// * Otherwise only axions with an event are flagged, and lanes that write
//   products at places of their own take 3.7 us an axion in a full warp: up to
//   kFewAbsorb, as many as the lists held at first (20,000 cells of 120 axions,
//   a third of them flagged: 205 us by lists of 8, 331 with a limit of 64, 186
//   now; limits of 4 and 12 lose 5 to 50 % where most cells have 5 to 8).
constexpr int kFewAbsorb = 8, kManyAbsorb = 256, kWarpAxions = 5;

__host__ __device__ constexpr int absorb_limit(bool all, int ncells) {
  const int few = ncells < kManyAbsorb ? kWarpAxions * ncells : kManyAbsorb;
  return !all || few < kFewAbsorb ? kFewAbsorb : few < kManyAbsorb ? few : kManyAbsorb;
}

template <bool AHEAD>
__device__ __forceinline__ void absorb_lane(const StepArgs& A, int cell, uint32_t* row, LaneCell& L, const Cnt& cnt,
                                            Lane64& xa) {
  const bool bath = A.mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS);
  const long abase = (long)cell * A.a.cap, gbase = (long)cell * A.g.cap;
  const int n = L.na, nw = (n + 31) >> 5;
  int w = -1;
  uint32_t v = 0u;
  auto next = [&]() {  // the next flagged slot, or -1
    while (v == 0u) {
      if (++w >= nw) return -1;
      v = row[w];
      row[w] = 0u;
      if (w == nw - 1 && (n & 31)) v &= (1u << (n & 31)) - 1u;  // bits beyond n never count
    }
    const int b = __ffs(v) - 1;
    v &= v - 1u;
    return 32 * w + b;
  };
  AxItem t;
  float4 q, u;
  t.slot = next();
  t.x = t.y = t.z = 0.f;
  if (t.slot >= 0) {
    t.r = A.recA[abase + t.slot];
    q = A.a.wp[abase + t.slot];
    if (AHEAD) u = A.a.xyz[abase + t.slot];
  }
  int run = 0, nrm = 0;
  while (t.slot >= 0) {
    t.w = q.x;
    t.px = q.y;
    t.py = q.z;
    t.pz = q.w;
    const int slot2 = next();
    uint4 r2 = make_uint4(0, 0, 0, 0);
    float4 u2;
    if (slot2 >= 0) {
      r2 = A.recA[abase + slot2];
      q = A.a.wp[abase + slot2];
      if (AHEAD) u2 = A.a.xyz[abase + slot2];
    }
    bool removed;
    const int K = axion_outcome(A, t, abase, bath, cnt, xa, &removed);
    if (K > 0) {
      if (!AHEAD) u = A.a.xyz[abase + t.slot];
      const float wprod = __uint_as_float(t.r.y);
      const float3 pg = photon_from_axion(A, t.px, t.py, t.pz);
      for (int k = 0; k < K; ++k) {
        const int dst = L.ng + run + k;
        if (dst < A.g.cap) write_particle(A.g, gbase + dst, wprod, pg.x, pg.y, pg.z, u.x, u.y, u.z);
        else cnt.add(C_DROP, 1);
      }
      run += K;
    }
    if (removed) {
      row[t.slot >> 5] |= 1u << (t.slot & 31);
      ++nrm;
    }
    t.slot = slot2;
    t.r = r2;
    u = u2;
  }
  L.ng = min(L.ng + run, A.g.cap);
  if (nrm == 0) return;
  // tail fill: removed slots below ns, ascending, take the kept slots from ns
  // on, four at a time, all loaded before any is stored
  const int ns = n - nrm;
  int src = ns, wd = -1;
  uint32_t h = 0u;
  auto hole = [&]() {  // the next removed slot below ns, or -1
    while (h == 0u) {
      if (32 * ++wd >= ns) return -1;
      h = row[wd];
      if (32 * wd + 32 > ns) h &= (1u << (ns & 31)) - 1u;
    }
    const int b = __ffs(h) - 1;
    h &= h - 1u;
    return 32 * wd + b;
  };
  int dst;
  do {
    Mover m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      dst = hole();
      if (dst >= 0)
        while ((row[src >> 5] >> (src & 31)) & 1u) ++src;
      m[i] = mover_load(A.a, abase, src, dst);
      if (dst >= 0) ++src;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) mover_store(A.a, abase, m[i]);
  } while (dst >= 0);
  L.na = ns;
}

#ifndef AXPIC_EVENT_MIN_CTAS
#define AXPIC_EVENT_MIN_CTAS 4
#endif
// the full-step kernel, without the warp paths (event_heavy_kernel takes
// them), fits more CTAs an SM
#ifndef AXPIC_EVENT_FULL_MIN_CTAS
#define AXPIC_EVENT_FULL_MIN_CTAS 6
#endif

// Round trip 1: counts and the mask rows (staged by cp.async; cleared for
// the next step as soon as they are read). Only the cells that have an
// electron event read the cell constants; only those with a flagged slot
// read their exchange buffer (while their events run), and only those with
// an exchange write it. Each phase runs first in the lanes whose cell is
// light for it, then warp-wide for the heavy cells one by one (in a full
// step, by event_heavy_kernel: without the warp paths, and with one load of
// each kind in flight, this kernel holds 6 CTAs an SM instead of 4); a
// cell's absorb phase ends before its emit phase starts. The absorb and emit
// exchanges are added to the cell's buffer in that order, whichever way the
// step was called.
template <int PH, bool SR>
__global__ void __launch_bounds__(128, PH == 3 ? AXPIC_EVENT_FULL_MIN_CTAS : AXPIC_EVENT_MIN_CTAS)
    event_kernel(StepArgs A) {
  wait_predecessor();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long warp_cnt[4][kNumCounters];
  const int wid = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  const int lane = threadIdx.x & 31;
  // a full step's launch may give a warp fewer cells than lanes
  const int cells = PH == (PH_ABSORB | PH_EMIT) ? A.ev_cells : 32;
  const int cell = A.cell0 + (blockIdx.x * nw + wid) * cells + lane;
  const bool valid = lane < cells && cell < A.cell0 + A.ncells;
  if (lane < kNumCounters) warp_cnt[wid][lane] = 0ull;
  __syncwarp();
  const Cnt cnt{warp_cnt[wid]};
  unsigned char* const sbase = smem + wid * ev_scratch_bytes(A.a.cap, A.g.cap, A.e.cap, ev_parts(PH));
  const EvScratch S = ev_carve<ev_parts(PH)>(sbase, A.a.cap, A.g.cap, A.e.cap);
  uint16_t* lA = S.lt + lane;
  uint16_t* lG = lA + 32 * kLight;
  uint16_t* lE = lG + 32 * kLight;
  const uint32_t step = step_of(A);
  const int mask = A.mask;
  const bool emitG = (PH & PH_EMIT) && (mask & AXPIC_CH_PRIMAKOFF);
  const bool emitE = (PH & PH_EMIT) && (mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS));
  const bool staged = S.rowA != nullptr;
  uint32_t* rA = staged ? S.rowA + lane * S.sA : nullptr;
  uint32_t* rG = staged ? S.rowG + lane * S.sG : nullptr;
  uint32_t* rE = staged ? S.rowE + lane * S.sE : nullptr;

  // ------------------------------------------------------------ round trip 1
  LaneCell L;
  L.na = L.ng = L.ng0 = L.ne = 0;
  L.nflA = L.nflG = L.nflE = 0;
  L.wu = L.r_cc = L.r_cb = L.r_T = 0.f;
  int pstart = 0;
  double xb[4] = {0.0, 0.0, 0.0, 0.0};
  bool xload = false;
  if (valid) {
    if (staged) {
      if (PH & PH_ABSORB)
        for (int w = 0; w < A.Wa; ++w) cp_async4(rA + w, A.bitsA + (size_t)cell * A.Wa + w);
      if (emitG)
        for (int w = 0; w < A.Wg; ++w) cp_async4(rG + w, A.bitsG + (size_t)cell * A.Wg + w);
      if (emitE)
        for (int w = 0; w < A.We; ++w) cp_async4(rE + w, A.bitsE + (size_t)cell * A.We + w);
    }
    L.ne = min(max(A.e.count[cell], 0), A.e.cap);
    L.ng = min(max(A.g.count[cell], 0), A.g.cap);
    L.na = min(max(A.a.count[cell], 0), A.a.cap);
    if (!(PH & PH_ABSORB) && A.use_snapshot) pstart = A.photon_start[cell];
  }
  const int ne = L.ne, ng_start = L.ng, na_start = L.na;
  L.ng0 = (PH & PH_ABSORB) ? ng_start : (A.use_snapshot ? min(pstart, ng_start) : ng_start);
  // particles present at the start of the step: counted by the absorb phase,
  // or by the emit phase when no absorb ran this step
  if ((PH & PH_ABSORB) || ((PH & PH_EMIT) && !A.use_snapshot)) {
    const int sne = warp_sum_i(ne), sng = warp_sum_i(ng_start), sna = warp_sum_i(na_start);
    const unsigned nv = __popc(__ballot_sync(kFull, valid));
    if (lane == 0) {
      cnt.add(C_NE, (unsigned)sne);
      cnt.add(C_NG, (unsigned)sng);
      cnt.add(C_NA, (unsigned)sna);
      cnt.add(C_CELLS, nv);
    }
  }
  if (staged) cp_async_wait_all();
  __syncwarp();

  bool hA = false, hE = false;
  // a full step leaves a cell heavy in either phase, rows uncleared, to
  // event_heavy_kernel
  bool defer = false;
  if (valid) {
    if (staged) {
      uint32_t nzA = 0u, nzG = 0u, nzE = 0u;
      if (PH == PH_ABSORB) L.nflA = count_row(rA, na_start, &nzA);
      else if (PH & PH_ABSORB) L.nflA = scan_row(rA, na_start, lA, &nzA);
      if (emitG) L.nflG = scan_row(rG, L.ng0, lG, &nzG);
      if (emitE) L.nflE = scan_row(rE, ne, lE, &nzE);
      hA = L.nflA > kLight;
      hE = L.nflG > kLight || L.nflE > kLightE;
      defer = PH == (PH_ABSORB | PH_EMIT) && (hA || hE);
      if (!defer) {
        if (PH & PH_ABSORB) clear_row(A.bitsA, A.Wa, cell, nzA);
        if (emitG) clear_row(A.bitsG, A.Wg, cell, nzG);
        if (emitE) clear_row(A.bitsE, A.We, cell, nzE);
      }
    } else {
      hA = (PH & PH_ABSORB) != 0;
      hE = (PH & PH_EMIT) != 0;
      defer = PH == (PH_ABSORB | PH_EMIT);
    }
    if (PH == PH_ABSORB) A.photon_start[cell] = ng_start;  // read by the emit call of this step
    // the cell constants of the thermal-bath events, for the cells that
    // have one (the capped means of common-weight cells are counted by the
    // decision kernel)
    if (!defer && emitE && (!staged || L.nflE > 0)) {
      const float* rec = A.rec + (size_t)cell * kRecLen;
      L.wu = A.mom[(size_t)cell * kMomLen + M_WU];
      L.r_cc = rec[R_CC];
      L.r_cb = rec[R_CB];
      L.r_T = rec[R_T];
    }
    // the exchange buffer of a cell with an event, loaded while its events run
    if (!defer && (!staged || (L.nflA | L.nflG | L.nflE))) {
      xload = true;
      const double2* x2 = reinterpret_cast<const double2*>(A.xbuf + (size_t)cell * 4);
      cp_async16(S.xs + 2 * lane, x2);
      cp_async16(S.xs + 2 * lane + 1, x2 + 1);
    }
  }

  Lane64 xa, xe;
  if (PH == (PH_ABSORB | PH_EMIT)) {
    // full step: a cell light in both phases is taken by its lane, any other
    // by event_heavy_kernel after this kernel (a warp per cell); either way
    // the new axions reuse the freed slots
    if (valid && !defer && (L.nflA | L.nflG | L.nflE))
      cell_lane<SR>(A, step, cell, true, lA, lG, lE, L, cnt, xa, xe);
    // the heavy cells are listed for event_heavy_kernel, from index cell0
    const unsigned hm = __ballot_sync(kFull, defer);
    if (hm) {
      int base = 0;
      if (lane == 0) base = atomicAdd(A.heavy_n, __popc(hm));
      base = __shfl_sync(kFull, base, 0);
      if (defer) A.heavy[A.cell0 + base + __popc(hm & ((1u << lane) - 1u))] = cell;
    }
  } else if (PH == PH_ABSORB) {
    const bool all = A.absorb_mode == 1 && (mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS));  // every axion is flagged
    if (staged) hA = L.nflA > absorb_limit(all, A.ncells);
    if (valid && !hA && L.nflA) {
      if (all) absorb_lane<false>(A, cell, rA, L, cnt, xa);
      else absorb_lane<true>(A, cell, rA, L, cnt, xa);
    }
    __syncwarp();
    for (unsigned hm = __ballot_sync(kFull, valid && hA); hm; hm &= hm - 1u) {
      const int j = __ffs(hm) - 1;
      const int c = __shfl_sync(kFull, cell, j);
      PhaseOut o;
      absorb_warp(A, c, sbase, staged ? S.rowA + j * S.sA : A.bitsA + (size_t)c * A.Wa,
                  staged ? nullptr : A.bitsA + (size_t)c * A.Wa, cnt, __shfl_sync(kFull, na_start, j),
                  __shfl_sync(kFull, ng_start, j), true, &o);
      if (lane == j) {
        L.na = o.na;
        L.ng = o.ng;
        xa.dE = o.x[0];
        xa.dPx = o.x[1];
        xa.dPy = o.x[2];
        xa.dPz = o.x[3];
        xa.any = o.any;
      }
    }
  } else {
    if (valid && !hE && (L.nflG | L.nflE)) cell_lane<SR>(A, step, cell, false, lA, lG, lE, L, cnt, xa, xe);
    __syncwarp();
    for (unsigned hm = __ballot_sync(kFull, valid && hE); hm; hm &= hm - 1u) {
      const int j = __ffs(hm) - 1;
      const int c = __shfl_sync(kFull, cell, j);
      PhaseOut o;
      const uint32_t* gG = emitG ? (staged ? S.rowG + j * S.sG : A.bitsG + (size_t)c * A.Wg) : nullptr;
      const uint32_t* gE = emitE ? (staged ? S.rowE + j * S.sE : A.bitsE + (size_t)c * A.We) : nullptr;
      emit_warp<SR>(A, step, c, sbase, gG, (emitG && !staged) ? A.bitsG + (size_t)c * A.Wg : nullptr, gE,
                (emitE && !staged) ? A.bitsE + (size_t)c * A.We : nullptr, cnt,
                AxDest{nullptr, 0, 1, __shfl_sync(kFull, L.na, j)}, __shfl_sync(kFull, L.ng, j),
                __shfl_sync(kFull, L.ng0, j), __shfl_sync(kFull, ne, j), __shfl_sync(kFull, L.wu, j),
                __shfl_sync(kFull, L.r_cc, j), __shfl_sync(kFull, L.r_cb, j), __shfl_sync(kFull, L.r_T, j), &o);
      if (lane == j) {
        L.na = o.na;
        L.ng = o.ng;
        xe.dE = o.x[0];
        xe.dPx = o.x[1];
        xe.dPy = o.x[2];
        xe.dPz = o.x[3];
        xe.any = o.any;
      }
    }
  }
  if (valid && !defer) {
    A.a.count[cell] = L.na;
    A.g.count[cell] = L.ng;
    if (xa.any || xe.any) {
      {
        const double2* x2 = xload ? S.xs + 2 * lane : reinterpret_cast<const double2*>(A.xbuf + (size_t)cell * 4);
        if (xload) cp_async_wait_all();
        const double2 a = x2[0], b = x2[1];
        xb[0] = a.x;
        xb[1] = a.y;
        xb[2] = b.x;
        xb[3] = b.y;
      }
      if (xa.any) {
        xb[0] += xa.dE;
        xb[1] += xa.dPx;
        xb[2] += xa.dPy;
        xb[3] += xa.dPz;
      }
      if (xe.any) {
        xb[0] += xe.dE;
        xb[1] += xe.dPx;
        xb[2] += xe.dPy;
        xb[3] += xe.dPz;
      }
      double2* xo = reinterpret_cast<double2*>(A.xbuf + (size_t)cell * 4);
      xo[0] = make_double2(xb[0], xb[1]);
      xo[1] = make_double2(xb[2], xb[3]);
    }
  }
  __syncwarp();
  if (lane < kNumCounters) {
    const unsigned long long v = warp_cnt[wid][lane];
    if (v) atomicAdd(A.counters + (size_t)(blockIdx.x % A.ctr_rows) * kNumCounters + lane, v);
    if (lane == C_DROP && v) atomicOr(A.err, ERR_CAPACITY);
  }
}


// The full step of the cells the event kernel listed as heavy (more flagged
// slots in a phase than a lane takes): a warp per cell, persistent over the
// list, with the mask rows read and cleared in global memory. Cells are
// independent within a step, so each gets what the warp path inside the
// event kernel gave it; the list order does not matter.
constexpr int kHeavyGrid = 152;  // one CTA on each of the 152 SMs

template <bool SR>
__global__ void __launch_bounds__(128) event_heavy_kernel(StepArgs A) {
  wait_predecessor();
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long warp_cnt[4][kNumCounters];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  if (lane < kNumCounters) warp_cnt[wid][lane] = 0ull;
  __syncwarp();
  const Cnt cnt{warp_cnt[wid]};
  unsigned char* const sbase = smem + wid * ev_scratch_bytes(A.a.cap, A.g.cap, A.e.cap, EV_LISTS);
  const EvScratch S = ev_carve<EV_LISTS>(sbase, A.a.cap, A.g.cap, A.e.cap);
  const uint32_t step = step_of(A);
  const bool emitG = (A.mask & AXPIC_CH_PRIMAKOFF) != 0;
  const bool emitE = (A.mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS)) != 0;
  const int n = *A.heavy_n;
  for (int k = blockIdx.x * nw + wid; k < n; k += gridDim.x * nw) {
    const int c = A.heavy[A.cell0 + k];
    const int na0 = min(max(A.a.count[c], 0), A.a.cap);
    const int ng0 = min(max(A.g.count[c], 0), A.g.cap);
    const int ne = min(max(A.e.count[c], 0), A.e.cap);
    float wu = 0.f, r_cc = 0.f, r_cb = 0.f, r_T = 0.f;
    if (emitE) {
      const float* rec = A.rec + (size_t)c * kRecLen;
      wu = A.mom[(size_t)c * kMomLen + M_WU];
      r_cc = rec[R_CC];
      r_cb = rec[R_CB];
      r_T = rec[R_T];
    }
    uint32_t* rowA = A.bitsA + (size_t)c * A.Wa;
    uint32_t* rowG = emitG ? A.bitsG + (size_t)c * A.Wg : nullptr;
    uint32_t* rowE = emitE ? A.bitsE + (size_t)c * A.We : nullptr;
    PhaseOut oa, oe;
    absorb_warp(A, c, sbase, rowA, rowA, cnt, na0, ng0, false, &oa);
    const int nrmA = na0 - oa.na;
    emit_warp<SR>(A, step, c, sbase, rowG, rowG, rowE, rowE, cnt, AxDest{S.rmA, nrmA, 1, na0}, oa.ng, ng0, ne, wu, r_cc,
              r_cb, r_T, &oe);
    // freed slots left over: closed from the tail
    if (oe.np < nrmA) compact_tail(A.a, (long)c * A.a.cap, S.rmA + oe.np, S.rbA, oe.na, na0);
    if (lane == 0) {
      A.a.count[c] = oe.na;
      A.g.count[c] = oe.ng;
      if (oa.any || oe.any) {
        double* xb = A.xbuf + (size_t)c * 4;
        double x0 = xb[0], x1 = xb[1], x2 = xb[2], x3 = xb[3];
        if (oa.any) {
          x0 += oa.x[0];
          x1 += oa.x[1];
          x2 += oa.x[2];
          x3 += oa.x[3];
        }
        if (oe.any) {
          x0 += oe.x[0];
          x1 += oe.x[1];
          x2 += oe.x[2];
          x3 += oe.x[3];
        }
        xb[0] = x0;
        xb[1] = x1;
        xb[2] = x2;
        xb[3] = x3;
      }
    }
    __syncwarp();
  }
  __syncwarp();
  if (lane < kNumCounters) {
    const unsigned long long v = warp_cnt[wid][lane];
    if (v) atomicAdd(A.counters + (size_t)(blockIdx.x % A.ctr_rows) * kNumCounters + lane, v);
    if (lane == C_DROP && v) atomicOr(A.err, ERR_CAPACITY);
  }
}

// ---------------------------------------------------------------- launchers
size_t step_smem_per_warp(int acap, int gcap, int ecap) {
  return ev_scratch_bytes(acap, gcap, ecap, EV_LISTS | EV_LANES | EV_ROWS);
}
size_t step_smem_accepted(int acap, int gcap, int ecap) {
  return ev_list_bytes(acap, gcap, ecap) + 1536 + ev_row_bytes(acap, gcap, ecap);
}

int resident_ctas(const void* fn, int threads, size_t dyn_smem, int max_per_sm) {
  int dev = 0, sms = 0, regs_sm = 0, smem_sm = 0, reserved = 0, threads_sm = 0, blocks_sm = 0;
  cudaFuncAttributes fa;
  if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) ||
      cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) ||
      cudaDeviceGetAttribute(&threads_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) ||
      cudaDeviceGetAttribute(&blocks_sm, cudaDevAttrMaxBlocksPerMultiprocessor, dev) ||
      cudaFuncGetAttributes(&fa, fn))
    return 0;
  const int warps = (threads + 31) / 32;
  const int regs_cta = warps * ((max(1, fa.numRegs) * 32 + 255) / 256 * 256);
  const int smem_cta = (int)((fa.sharedSizeBytes + dyn_smem + reserved + 127) / 128 * 128);
  const int nb = min(min(regs_sm / regs_cta, smem_sm / smem_cta), min(threads_sm / (warps * 32), blocks_sm));
  return max(1, min(nb, max_per_sm)) * max(1, sms);
}

// Cells per warp of a full step's event kernel. A lane takes a cell, and a
// warp as long as its lane with the most flagged slots: 32 cells a warp issue
// the least, fewer end sooner and spread over more warps. By the cells that
// run side by side; a pass, us, with 32, 16, 8 and 4 cells a warp:
//   4,096 dense cells (512 e, 256 g), 8 steps:    646   587   553   529
//   9,200 cells of 24 boxes, 16 steps:            1074  990   935   899
//   16,384 dense cells, 8 steps:                  909   835   800   869
//   46,000 cells of 120 boxes, 16 steps:          2050  1829  1693
//   65,536 dense cells, 32 steps:                 6129  6146  6915
//   64,000 thin cells (64 e, 32 g), 4 steps:      260   267   279
//   884,736 thin cells, 4 steps:                  1747  1977  2392
static int event_cells(const StepArgs& A) {
  const int n = max(A.ncells, A.dec_cells);
  return n < 12288 ? 4 : n < 49152 ? 8 : 32;
}

template <int PH>
static cudaError_t launch_events(const StepArgs& A, int warps, cudaStream_t st, bool chained) {
  constexpr bool full = PH == (PH_ABSORB | PH_EMIT);
  const size_t per = ev_scratch_bytes(A.a.cap, A.g.cap, A.e.cap, ev_parts(PH));
  StepArgs B = A;
  B.ev_cells = full ? event_cells(A) : 32;
  const int grid = (A.ncells + B.ev_cells * warps - 1) / (B.ev_cells * warps);
  const bool sr = A.rate_model != 0;
  const cudaError_t e = launch_chained(chained, sr ? event_kernel<PH, true> : event_kernel<PH, false>, grid, warps * 32,
                                       per * warps, st, B);
  if (e || !full) return e;
  // persistent over the heavy list: a warp per cell, at most one warp per
  // cell of the launch and kHeavyGrid CTAs
  const int hgrid = max(1, min((A.ncells + warps - 1) / warps, kHeavyGrid));
  // in a replay the branches' kernels share the SMs, and an SM that splits its
  // memory otherwise for one of them waits for the others to end: as much shared
  // memory as the event kernel where that is more (65,536 dense cells in 8
  // branches: 133 us a step, 141 with the lists alone, 137 with lists and event
  // scratch). A launch of its own leaves the rest to L1 (20,000 hot cells, all
  // heavy: 612 us a step, 650 with the event kernel's size).
  size_t lists = ev_scratch_bytes(A.a.cap, A.g.cap, A.e.cap, EV_LISTS);
  if (A.dec_cells) lists = max(lists, per);
  return launch_chained(chained, sr ? event_heavy_kernel<true> : event_heavy_kernel<false>, hgrid, warps * 32, lists * warps, st, A);
}

// Cells per chunk of a decision warp: asked for, or by the launch. A chunk
// should hold enough work for the warp's lanes and for full batches of full
// decisions, not so much that the last chunks are waited for, and the chunks
// should fill the resident warps (rounds: chunks over resident warps, over
// all the branches that a replayed step runs side by side). The work of a
// cell is taken from its capacities, u = e/2 + g + a slots. Times of a pass,
// us, by chunk size (the one taken first):
//   4,096 cells of 512 e, 256 g (u 1024):       1: 720   2: 746   4: 794   8: 898
//   16,384 of the same:                         4: 1015  2: 1197  8: 1098  1: 1290
//   196,000 of 128 e, 64 g (u 704), replayed:   8: 3700  16: 3884 4: 3926  32: 4515
//   262,144 of 256 e, 128 g (u 1280):           8: 4593  16: 4655 4: 4727  32: 5047
//   6,000 of 64 e, 48 g (u 384):                4: 41.5  2: 41.8  8: 43.8  1: 45.8
//   64,000 of 64 e, 32 g (u 160), replayed:     16: 285  8: 293   32: 318  4: 312
//   262,144 of the same, replayed:              32: 563  16: 581  8: 660   4: 711
//   262,144 of the same, a launch of its own:   16: 294  32: 312  8: 328   4: 347
//   64 of 128 g, latency (u 1154):              1: 23.7  4: 26.0  8: 28.7  32: 42.8
int decide_chunk(const StepArgs& A) {
  if (A.dec_chunk) return A.dec_chunk;
  const long u = A.e.cap / 2 + A.g.cap + A.a.cap;
  const long warps = (long)A.dec_grid * kDecWarps;
  const long n = max(A.ncells, A.dec_cells);
  int lo = 1, hi = 32;
  while (lo < 32 && lo * u < 1000) lo *= 2;
  while (hi > lo && hi * u > 10400) hi /= 2;
  for (int c = hi; c > lo; c /= 2) {
    // one launch of less than two rounds of the largest chunks waits for its second
    const long tenths = c == 32 && A.dec_cells == 0 ? 20 : 8;
    if (10 * (n / c) >= tenths * warps) return c;
  }
  return lo;
}

// The decision passes a phase set needs, as DK_* bits.
static int decide_kinds(const StepArgs& A, int phases) {
  int k = 0;
  if ((phases & PH_EMIT) && (A.mask & (AXPIC_CH_COMPTON | AXPIC_CH_BREMS)) && A.e.cap > 0) k |= DK_ELECTRON;
  if ((phases & PH_EMIT) && (A.mask & AXPIC_CH_PRIMAKOFF) && A.g.cap > 0) k |= DK_PHOTON;
  if ((phases & PH_ABSORB) && A.a.cap > 0) k |= DK_AXION;
  return k;
}

static cudaError_t launch_decide(const StepArgs& A, int phases, cudaStream_t st, bool chained) {
  const int kinds = decide_kinds(A, phases);
  if (kinds == 0) return cudaSuccess;
  // persistent: as many CTAs as the device holds at once, at most one warp
  // per chunk
  const int chunk = decide_chunk(A);
  const int nchunks = (A.ncells + chunk - 1) / chunk;
  const int grid = max(1, min((nchunks + kDecWarps - 1) / kDecWarps, A.dec_grid));
  const bool sr = A.rate_model != 0;
  auto kernel = sr ? decide_kernel<32, true> : decide_kernel<32, false>;
  switch (chunk) {
    case 1: kernel = sr ? decide_kernel<1, true> : decide_kernel<1, false>; break;
    case 2: kernel = sr ? decide_kernel<2, true> : decide_kernel<2, false>; break;
    case 4: kernel = sr ? decide_kernel<4, true> : decide_kernel<4, false>; break;
    case 8: kernel = sr ? decide_kernel<8, true> : decide_kernel<8, false>; break;
    case 16: kernel = sr ? decide_kernel<16, true> : decide_kernel<16, false>; break;
    default: break;
  }
  return launch_chained(chained, kernel, grid, kDecThreads, 0, st, A, kinds);
}

static cudaError_t launch_feedback(const StepArgs& A, cudaStream_t st, bool chained) {
  const int grid = (A.ncells + kFeedbackThreads - 1) / kFeedbackThreads;
  // absorption by weight reduction takes energy from every axion: most cells
  // are remapped every step
  return launch_chained(chained, A.absorb_mode == 1 ? feedback_kernel<true> : feedback_kernel<false>, grid,
                        kFeedbackThreads, 0, st, A);
}

const char* step_kernel_names(int rate_model, int T_mode) {
  if (T_mode == 2 && rate_model == 2) return "decide_kernel,event_kernel,feedback_kernel,sr_cells_kernel";
  return "decide_kernel,event_kernel,feedback_kernel";
}

__global__ void set_step_kernel(uint32_t* p, uint32_t v, int n) {
  for (int i = 0; i < n; ++i) p[i] = v;
}

cudaError_t launch_set_step(uint32_t* p, uint32_t v, int n, cudaStream_t st) {
  set_step_kernel<<<1, 1, 0, st>>>(p, v, n);
  return cudaGetLastError();
}

cudaError_t decide_resident_ctas(int* out) {
  int dev = 0, sms = 0, nb = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)))
    return e;
  // every chunk size is bound to the same registers and shared memory
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, decide_kernel<32, true>, kDecThreads, 0))) return e;
  *out = max(1, nb) * max(1, sms);
  return cudaSuccess;
}

// After the temperature update of an evolved-T step the surrogate network's
// prefactors follow the new T (the table's entries are interpolated where
// they are needed).
static cudaError_t launch_records_update(const StepArgs& A, const SrArgs* sra, cudaStream_t st, bool chained) {
  if (!sra || A.T_mode != 2 || A.rate_model != 2) return cudaSuccess;
  return launch_sr_cells(*sra, st, chained);
}

cudaError_t launch_step(int phases, const StepArgs& A, int warps, cudaStream_t st, cudaEvent_t* ev,
                        const SrArgs* sra, bool after_step) {
  if (A.ncells == 0) return cudaSuccess;
  cudaError_t e;
  // optional measurement: events between the kernels of a full step, which
  // then run one by one
  auto mark = [&](int i) { return ev ? cudaEventRecord(ev[i], st) : cudaSuccess; };
  const bool chain = !ev;
  switch (phases) {
    case PH_ABSORB:
      if ((e = launch_decide(A, PH_ABSORB, st, false))) return e;
      return launch_events<PH_ABSORB>(A, warps, st, true);
    case PH_EMIT:
      if ((e = launch_decide(A, PH_EMIT, st, false))) return e;
      return launch_events<PH_EMIT>(A, warps, st, true);
    case PH_FEEDBACK:
      if ((e = launch_feedback(A, st, false))) return e;
      return launch_records_update(A, sra, st, true);
    case PH_ALL:
      if ((e = mark(0)) || (e = launch_decide(A, PH_ABSORB | PH_EMIT, st, chain && after_step)) || (e = mark(1)))
        return e;
      // (with nothing to decide the events are the first kernel)
      if ((e = launch_events<PH_ABSORB | PH_EMIT>(A, warps, st,
                                                  chain && (after_step || decide_kinds(A, PH_ABSORB | PH_EMIT)))) ||
          (e = mark(2)))
        return e;
      if ((e = launch_feedback(A, st, chain)) || (e = mark(3)) || (e = launch_records_update(A, sra, st, chain)) ||
          (e = mark(4)))
        return e;
      return cudaSuccess;
    default:
      return cudaErrorInvalidValue;
  }
}

// The dynamic shared-memory limit of the event kernels is a process-wide
// attribute of each function: contexts with smaller slabs share it with
// larger ones, so it is only ever raised (per device, under a lock), never
// lowered under a context that needs more.
cudaError_t set_step_smem_limits(size_t bytes) {
  static std::mutex mu;
  static size_t set_for[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t* cur = dev >= 0 && dev < 64 ? &set_for[dev] : nullptr;
  if (cur && bytes <= *cur) return cudaSuccess;
  const int b = (int)bytes;
  for (const void* k :
       {(const void*)event_kernel<PH_ABSORB, false>, (const void*)event_kernel<PH_EMIT, false>,
        (const void*)event_kernel<PH_ABSORB | PH_EMIT, false>, (const void*)event_heavy_kernel<false>,
        (const void*)event_kernel<PH_ABSORB, true>, (const void*)event_kernel<PH_EMIT, true>,
        (const void*)event_kernel<PH_ABSORB | PH_EMIT, true>, (const void*)event_heavy_kernel<true>})
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, b))) return e;
  if (cur) *cur = bytes;
  return cudaSuccess;
}

}  // namespace axpic
