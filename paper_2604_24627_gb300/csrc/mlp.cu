// The spectral surrogate's MLP (4 -> 64 -> 64 -> 96, tanh hidden layers) on
// the GPU: forward, backward and Adam. Layer 1 (K = 4) runs on the CUDA
// cores; every other product, forward and backward, on the 5th-generation
// tensor cores: bfloat16 operands in shared memory, one elected thread issues
// tcgen05.mma.kind::f16 with FP32 accumulators in tensor memory, commits to
// an mbarrier, and the CTA reads the tile back with tcgen05.ld.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "common.cuh"
#include "mlp.h"
#include "tc.cuh"
#include "surrogate.h"

namespace axpic {

// ---------------------------------------------------------------- the network's kernel
// One persistent CTA takes tiles of 128 rows through the whole network, and
// in training through the backward pass: every intermediate stays on the SM.
// 16 warps: warp w holds rows 32 (w & 3) .. + 31 (the tensor memory lanes it
// can read) and the column group w >> 2 of four, so a thread keeps 16 columns
// of h1 and h2 and 24 of z of its row in registers.
//
// Bound by the chain of four products with their read-backs (a tile's
// products are 0.2 us of tensor-core time), not by bytes: a row is 400 B.
// Formed kernel by kernel (16 launches a training step, activations through
// memory, operands staged element by element) a step of 8192 rows took
// 268 us; fused, with one kernel summing the CTAs' gradients, 27 us (eight steps
// and the weights read back: 2171 -> 245 us, 210 with the launches chained).
//
// Operands are bfloat16 tiles of 8 x 16-byte core matrices without swizzle.
// The weight gradients contract over the tile's rows: their operands are the
// same activation tiles read MN-major (a core matrix of 8 rows by 8 columns
// serves both majors; the group strides swap roles), 128 features by 128
// rows of which the first 64 features are real (the others read the
// neighbouring core matrices and end in accumulator lanes nothing reads).
constexpr int kNetRows = 128;
constexpr int kMlpThreads = 512;
// shared memory, bytes
constexpr int kSH1 = 0, kSH2 = 16384, kSdZ = 32768, kSdA2 = 57344;  // training: four activation tiles
constexpr int kSW2f = 73728, kSW3f = 81920, kSW2b = 94208, kSW3b = 102400;
constexpr int kSSmall = 114688;                       // W1, b1, b2, b3 (FP32), then the column sums
constexpr int kSmallFloats = 256 + 64 + 64 + 96;
constexpr int kTrainSmem = kSSmall + 4 * kSmallFloats + 4 * 4 * kSmallFloats;
// inference: h1, h2 and the forward weights alone
constexpr int kFW2f = 32768, kFW3f = 40960, kFSmall = 53248;
constexpr int kFwdSmem = kFSmall + 4 * kSmallFloats;
// tensor memory columns (training; inference uses z's columns over z2's)
constexpr int kTZ2 = 0, kTZ = 64, kTdH2 = 160, kTdH1 = 224, kTgW3 = 288, kTgW2 = 384, kTTrain = 512, kTFwd = 128;

struct MlpArgs {
  const float* P;   // parameters
  const float* X;   // [n][4]
  const float* Zt;  // training targets [n][96]
  float* Z;         // inference output [n][96]
  float* part;      // training: [CTAs][kMlpParams] gradients of each CTA's rows
  double* loss;     // training: [CTAs] sums of (z - Zt)^2
  int n;
  float inv_n;
  int vec;          // Zt (training) or Z (inference) rows are 16-byte aligned
  int* err;
};

// Descriptor of an instruction with MN-major A and B.
__host__ __device__ constexpr uint32_t mma_idesc_mn(int M, int N) { return mma_idesc(M, N) | (1u << 15) | (1u << 16); }

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

// Eight values (columns j0 .. j0 + 7 of row r) as bfloat16 into one 16-byte
// row of a core matrix of a tile of kc columns.
__device__ __forceinline__ void store8(unsigned char* tile, int r, int j0, int kc, const float* v) {
  uint4 u;
  uint32_t* w = reinterpret_cast<uint32_t*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(tile) + core_off(r, j0, kc)) = u;
}

// B^T tile (N rows n, K columns k) of a product with B(k, n) = W[k * ldn + n]
// (forward) or W[n * ldk + k] (the transposed weights of the backward pass).
template <bool TRANS>
__device__ __forceinline__ void stage_weights(unsigned char* tile, const float* W, int N, int K) {
  for (int i = threadIdx.x; i < N * (K / 8); i += kMlpThreads) {
    float v[8];
    int n, k0;
    if (TRANS) {
      n = i / (K / 8);
      k0 = 8 * (i - n * (K / 8));
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = W[n * K + k0 + j];
    } else {
      k0 = 8 * (i / N);
      n = i - (i / N) * N;
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = W[(k0 + j) * N + n];
    }
    store8(tile, n, k0, K, v);
  }
}

// C += A . B over K/16 instructions, both K-major (A rows of kc columns).
__device__ __forceinline__ void issue_k(uint32_t tmem, uint32_t a, uint32_t b, int N, int K) {
  const uint32_t sbo = (uint32_t)(K >> 3) * 128u;
  for (int s = 0; s < K / 16; ++s)
    mma_bf16(tmem, mma_desc(a + s * 256, 128, sbo), mma_desc(b + s * 256, 128, sbo), mma_idesc(128, N), s > 0);
}

// C (features x N) (+)= A^T . B over the tile's 128 rows: A a tile of 64
// columns, B one of N, both read MN-major (LBO: the row groups, SBO: the
// column groups).
__device__ __forceinline__ void issue_mn(uint32_t tmem, uint32_t a, uint32_t b, int N, bool add) {
  const uint32_t lba = 8 * 128, lbb = (uint32_t)(N >> 3) * 128u;
  for (int s = 0; s < kNetRows / 16; ++s)
    mma_bf16(tmem, mma_desc(a + 2 * s * lba, lba, 128), mma_desc(b + 2 * s * lbb, lbb, 128), mma_idesc_mn(128, N),
             add || s > 0);
}

// Sum over the warp's lanes of each of C (16 or 32) columns: lane l returns
// column l's sum (l mod 16 for 16 columns). Recursive halving, C - 1 or C
// shuffles.
template <int C>
__device__ __forceinline__ float lane_column_sums(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = C / 2; o; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float give = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
    }
  }
  if (C == 16) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 16);
  return v[0];
}

template <bool TRAIN>
__global__ void __launch_bounds__(kMlpThreads, TRAIN ? 1 : 2) mlp_kernel(MlpArgs g) {
  wait_predecessor();
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ uint64_t bars[3];  // [2]: what is in flight when a wait ran out
  __shared__ uint32_t tmem_base;
  __shared__ double lsum[kMlpThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quad = warp & 3, grp = warp >> 2;
  const int row = 32 * quad + lane;
  if (warp == 0) tmem_alloc(&tmem_base, TRAIN ? kTTrain : kTFwd);
  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    mbar_init(&bars[2], 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  unsigned char* const sW2f = sm + (TRAIN ? kSW2f : kFW2f);
  unsigned char* const sW3f = sm + (TRAIN ? kSW3f : kFW3f);
  float* const small = reinterpret_cast<float*>(sm + (TRAIN ? kSSmall : kFSmall));
  float *const sW1 = small, *const sb1 = small + 256, *const sb2 = small + 320, *const sb3 = small + 384;
  for (int i = tid; i < 256; i += kMlpThreads) sW1[i] = g.P[kOffW1 + i];
  if (tid < 64) sb1[tid] = g.P[kOffB1 + tid];
  else if (tid < 128) sb2[tid - 64] = g.P[kOffB2 + tid - 64];
  else if (tid < 224) sb3[tid - 128] = g.P[kOffB3 + tid - 128];
  stage_weights<false>(sW2f, g.P + kOffW2, 64, 64);
  stage_weights<false>(sW3f, g.P + kOffW3, 96, 64);
  if (TRAIN) {
    stage_weights<true>(sm + kSW2b, g.P + kOffW2, 64, 64);
    stage_weights<true>(sm + kSW3b, g.P + kOffW3, 64, 96);
  }
  bool ok = true;
  // shared-memory operands and tensor-memory reads of all threads before the
  // next products, and whether every wait so far completed
  auto join = [&]() {
    smem_to_async_proxy();
    tc_fence_before();
    ok = __syncthreads_and(ok) != 0;
    tc_fence_after();
  };
  join();
  const uint32_t tmem = tmem_base;
  const uint32_t trow = tmem + ((uint32_t)(32 * quad) << 16);
  const uint32_t aH1 = smem_u32(sm + kSH1), aH2 = smem_u32(sm + kSH2);
  const uint32_t aW2f = smem_u32(sW2f), aW3f = smem_u32(sW3f);
  const uint32_t tZ = TRAIN ? kTZ : 0;  // inference: z over z2, which has been read
  uint32_t ph = 0, ph1 = 0;
  // one commit of barrier b (phase parity p); the warp converges for the
  // tensor-memory loads that follow. ok is the thread's own from here to the
  // next join, which alone decides whether the CTA goes on.
  auto await = [&](int b, uint32_t& p) {
    ok = ok && mbar_wait(&bars[b], p);
    p ^= 1u;
    __syncwarp();
    tc_fence_after();
  };
  const int ntiles = (g.n + kNetRows - 1) / kNetRows;
  float sgb3 = 0.f, sgb2 = 0.f, sgb1 = 0.f, sgw1[4] = {0.f, 0.f, 0.f, 0.f};
  double loss = 0.0;
  bool first = true;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const long r = (long)tile * kNetRows + row;
    const bool live = r < g.n;
    float x[4] = {0.f, 0.f, 0.f, 0.f}, zt[24];
    if (live) {
#pragma unroll
      for (int k = 0; k < 4; ++k) x[k] = g.X[r * 4 + k];
    }
    if (TRAIN) {
      // the targets, long before they are needed
      const float* t = g.Zt + r * 96 + 24 * grp;
      if (live && g.vec) {
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          const float4 q = reinterpret_cast<const float4*>(t)[j];
          zt[4 * j] = q.x;
          zt[4 * j + 1] = q.y;
          zt[4 * j + 2] = q.z;
          zt[4 * j + 3] = q.w;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 24; ++j) zt[j] = live ? t[j] : 0.f;
      }
    }
    // layer 1 (K = 4) on the CUDA cores
    float h1[16], h2[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int c = 16 * grp + j;
      float a = sb1[c];
#pragma unroll
      for (int k = 0; k < 4; ++k) a = fmaf(x[k], sW1[k * 64 + c], a);
      h1[j] = act_tanh(a);
    }
    store8(sm + kSH1, row, 16 * grp, 64, h1);
    store8(sm + kSH1, row, 16 * grp + 8, 64, h1 + 8);
    join();
    if (!ok) break;  // all threads alike: a wait of the last tile ran out in some
    if (tid == 0) {
      issue_k(tmem + kTZ2, aH1, aW2f, 64, 64);
      tc_commit(&bars[0]);
    }
    await(0, ph);
    tmem_ld16(trow + kTZ2 + 16 * grp, h2);
#pragma unroll
    for (int j = 0; j < 16; ++j) h2[j] = act_tanh(h2[j] + sb2[16 * grp + j]);
    store8(sm + kSH2, row, 16 * grp, 64, h2);
    store8(sm + kSH2, row, 16 * grp + 8, 64, h2 + 8);
    join();
    if (tid == 0 && ok) {
      issue_k(tmem + tZ, aH2, aW3f, 96, 64);
      tc_commit(&bars[0]);
    }
    await(0, ph);
    float z[32];
#pragma unroll
    for (int j = 0; j < 24; j += 8) tmem_ld8(trow + tZ + 24 * grp + j, z + j);
#pragma unroll
    for (int j = 0; j < 24; ++j) z[j] += sb3[24 * grp + j];
    if (!TRAIN) {
      float* o = g.Z + r * 96 + 24 * grp;
      if (live && ok) {
        if (g.vec) {
#pragma unroll
          for (int j = 0; j < 6; ++j)
            reinterpret_cast<float4*>(o)[j] = make_float4(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
        } else {
#pragma unroll
          for (int j = 0; j < 24; ++j) o[j] = z[j];
        }
      }
      continue;  // the next tile's first join orders these reads before z2 is written again
    }
    // dz = 2 (z - t) / n; the loss as an exact sum of (z - t)^2
    Sum3 sq;
#pragma unroll
    for (int j = 0; j < 24; ++j) {
      const float d = live ? z[j] - zt[j] : 0.f;
      zt[j] = d;
      sq.add_product(d, d);
      z[j] = 2.0f * d * g.inv_n;
    }
    if (sq.unsafe()) {
      for (int j = 0; j < 24; ++j) loss += (double)zt[j] * (double)zt[j];
    } else {
      loss += sq.value();
    }
#pragma unroll
    for (int j = 0; j < 24; j += 8) store8(sm + kSdZ, row, 24 * grp + j, 96, z + j);
    join();
    if (tid == 0 && ok) {
      issue_k(tmem + kTdH2, smem_u32(sm + kSdZ), smem_u32(sm + kSW3b), 64, 96);  // dh2 = dz W3^T
      tc_commit(&bars[0]);
      issue_mn(tmem + kTgW3, aH2, smem_u32(sm + kSdZ), 96, !first);  // gW3 += h2^T dz
    }
#pragma unroll
    for (int j = 24; j < 32; ++j) z[j] = 0.f;
    sgb3 += lane_column_sums<32>(z);
    await(0, ph);
    float d[16];
    tmem_ld16(trow + kTdH2 + 16 * grp, d);
#pragma unroll
    for (int j = 0; j < 16; ++j) d[j] *= 1.0f - h2[j] * h2[j];  // da2 = dh2 (1 - h2^2)
    store8(sm + kSdA2, row, 16 * grp, 64, d);
    store8(sm + kSdA2, row, 16 * grp + 8, 64, d + 8);
    join();
    if (tid == 0 && ok) {
      issue_k(tmem + kTdH1, smem_u32(sm + kSdA2), smem_u32(sm + kSW2b), 64, 64);  // dh1 = da2 W2^T
      tc_commit(&bars[0]);
      issue_mn(tmem + kTgW2, aH1, smem_u32(sm + kSdA2), 64, !first);  // gW2 += h1^T da2
      tc_commit(&bars[1]);  // gW3 and gW2: the tiles may be written again
    }
    sgb2 += lane_column_sums<16>(d);
    await(0, ph);
    tmem_ld16(trow + kTdH1 + 16 * grp, d);
#pragma unroll
    for (int j = 0; j < 16; ++j) d[j] *= 1.0f - h1[j] * h1[j];  // da1 = dh1 (1 - h1^2)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float p[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) p[j] = x[k] * d[j];
      sgw1[k] += lane_column_sums<16>(p);
    }
    sgb1 += lane_column_sums<16>(d);
    await(1, ph1);
    first = false;
  }
  ok = __syncthreads_and(ok) != 0;
  if (!ok) {
    // flag it and give the tensor core a second bounded wait: for every product
    // issued so far, before the tensor memory is released
    if (tid == 0) {
      atomicOr(g.err, 1);
      tc_commit(&bars[2]);
    }
    mbar_poll(&bars[2], 0, kWaitPolls);
  } else if (TRAIN) {
    // the CTA's gradients: one row of partials
    float* out = g.part + (size_t)blockIdx.x * kMlpParams;
    if (quad < 2) {
      float v[24];
#pragma unroll
      for (int j = 0; j < 24; j += 8) tmem_ld8(trow + kTgW3 + 24 * grp + j, v + j);
#pragma unroll
      for (int j = 0; j < 24; j += 4)
        *reinterpret_cast<float4*>(out + kOffW3 + row * 96 + 24 * grp + j) =
            make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      tmem_ld16(trow + kTgW2 + 16 * grp, v);
#pragma unroll
      for (int j = 0; j < 16; j += 4)
        *reinterpret_cast<float4*>(out + kOffW2 + row * 64 + 16 * grp + j) =
            make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
    }
    float* red = small + kSmallFloats + quad * kSmallFloats;  // gW1, gb1, gb2, gb3 of these 32 rows
    if (lane < 24) red[384 + 24 * grp + lane] = sgb3;
    if (lane < 16) {
      red[320 + 16 * grp + lane] = sgb2;
      red[256 + 16 * grp + lane] = sgb1;
#pragma unroll
      for (int k = 0; k < 4; ++k) red[k * 64 + 16 * grp + lane] = sgw1[k];
    }
    for (int o = 16; o; o >>= 1) loss += __shfl_xor_sync(0xFFFFFFFFu, loss, o);
    if (lane == 0) lsum[warp] = loss;
    __syncthreads();
    for (int i = tid; i < kSmallFloats; i += kMlpThreads) {
      const float* q = small + kSmallFloats + i;
      const float v = ((q[0] + q[kSmallFloats]) + q[2 * kSmallFloats]) + q[3 * kSmallFloats];
      const int o = i < 256 ? kOffW1 + i : i < 320 ? kOffB1 + i - 256 : i < 384 ? kOffB2 + i - 320 : kOffB3 + i - 384;
      out[o] = v;
    }
    if (tid == 0) {
      double s = 0.0;
      for (int w = 0; w < kMlpThreads / 32; ++w) s += lsum[w];
      g.loss[blockIdx.x] = s;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_free(tmem, TRAIN ? kTTrain : kTFwd);
}

// ---------------------------------------------------------------- gradients and Adam
// The CTAs' gradient rows added in CTA order (eight slices of rows per
// parameter, then the slices in order), so training does not depend on
// scheduling; then Adam with bias correction on the FP32 master parameters
// (ADAM), or the gradients themselves. Block 0 also sums the loss. After a wait
// that ran out (*err) the rows are not whole: nothing is written.
constexpr int kRedX = 32, kRedY = 8;

template <bool ADAM>
__global__ void __launch_bounds__(kRedX* kRedY) reduce_kernel(const float* part, const double* losses, int rows,
                                                              float inv_n, float* G, float* P, float* M, float* V,
                                                              double* loss, const int* err, float lr, float b1,
                                                              float b2, float eps, float c1, float c2) {
  wait_predecessor();  // (no pointer here is __restrict__: nothing is read before it)
  if (*err) return;
  __shared__ float s[kRedY][kRedX];
  const int i = blockIdx.x * kRedX + threadIdx.x;
  const int per = (rows + kRedY - 1) / kRedY;
  const int r0 = threadIdx.y * per, r1 = min(rows, r0 + per);
  float acc = 0.f;
#pragma unroll 8
  for (int r = r0; r < r1; ++r) acc += part[(size_t)r * kMlpParams + i];
  s[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y == 0) {
    float g = 0.f;
#pragma unroll
    for (int y = 0; y < kRedY; ++y) g += s[y][threadIdx.x];
    if (ADAM) {
      const float m = b1 * M[i] + (1.f - b1) * g;
      const float v = b2 * V[i] + (1.f - b2) * g * g;
      M[i] = m;
      V[i] = v;
      P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
    } else {
      G[i] = g;
    }
  }
  if (blockIdx.x == 0 && threadIdx.y == 1) {
    double l = 0.0;
    for (int r = threadIdx.x; r < rows; r += 32) l += losses[r];
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
    if (threadIdx.x == 0) *loss = l * (double)inv_n;
  }
}
static_assert(kMlpParams % kRedX == 0, "whole blocks of parameters");

// ---------------------------------------------------------------- the network
Mlp::~Mlp() {
  void* bufs[] = {P, G, Ma, Va, part, err, loss, losses};
  for (void* b : bufs)
    if (b) cudaFree(b);
}

// The training CTAs (one an SM: a tile's buffers and all of its tensor
// memory) and their gradient rows, made by the first training call.
cudaError_t Mlp::reserve_train() {
  if (losses) return cudaSuccess;
  cudaError_t e;  // (part may be there from a call that failed)
  if (!part && (e = cudaMalloc(&part, sizeof(float) * kMlpParams * (size_t)sms))) return e;
  return cudaMalloc(&losses, sizeof(double) * (size_t)sms);
}

cudaError_t Mlp::init(cudaStream_t s) {
  st = s;
  cudaError_t e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
  if ((e = cudaMalloc(&P, sizeof(float) * kMlpParams)) || (e = cudaMalloc(&G, sizeof(float) * kMlpParams)) ||
      (e = cudaMalloc(&Ma, sizeof(float) * kMlpParams)) || (e = cudaMalloc(&Va, sizeof(float) * kMlpParams)) ||
      (e = cudaMalloc(&err, sizeof(int))) || (e = cudaMalloc(&loss, sizeof(double))) ||
      (e = cudaMemsetAsync(P, 0, sizeof(float) * kMlpParams, st)) ||
      (e = cudaMemsetAsync(Ma, 0, sizeof(float) * kMlpParams, st)) ||
      (e = cudaMemsetAsync(Va, 0, sizeof(float) * kMlpParams, st)) || (e = cudaMemsetAsync(err, 0, sizeof(int), st)))
    return e;
  if ((e = cudaFuncSetAttribute(mlp_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTrainSmem))) return e;
  return cudaFuncSetAttribute(mlp_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

cudaError_t Mlp::forward(const float* X, int n, float* out) {
  if (n == 0) return cudaSuccess;
  MlpArgs a;
  std::memset(&a, 0, sizeof(a));
  a.P = P;
  a.X = X;
  a.Z = out;
  a.n = n;
  a.vec = aligned16(out);
  a.err = err;
  const int ntiles = (n + kNetRows - 1) / kNetRows;
  return launch_chained(true, mlp_kernel<false>, std::min(ntiles, 2 * sms), kMlpThreads, kFwdSmem, st, a);
}

cudaError_t Mlp::backward(const float* X, const float* Zt, int n, bool adam, float lr) {
  cudaError_t e;
  if (n == 0) {
    if ((e = cudaMemsetAsync(G, 0, sizeof(float) * kMlpParams, st))) return e;
    return cudaMemsetAsync(loss, 0, sizeof(double), st);
  }
  if ((e = reserve_train())) return e;
  MlpArgs a;
  std::memset(&a, 0, sizeof(a));
  a.P = P;
  a.X = X;
  a.Zt = Zt;
  a.part = part;
  a.loss = losses;
  a.n = n;
  a.inv_n = 1.0f / (float)n;
  a.vec = aligned16(Zt);
  a.err = err;
  const int grid = std::min((n + kNetRows - 1) / kNetRows, sms);
  // chained: a training step is two short kernels behind the last step's two
  // (8 steps of 8,192 rows: 244 -> 210 us)
  if ((e = launch_chained(true, mlp_kernel<true>, grid, kMlpThreads, kTrainSmem, st, a))) return e;
  const dim3 block(kRedX, kRedY);
  if (adam) {
    ++t;
    const float c1 = 1.0f - powf(0.9f, (float)t), c2 = 1.0f - powf(0.999f, (float)t);
    return launch_chained(true, reduce_kernel<true>, kMlpParams / kRedX, block, 0, st, part, losses, grid, a.inv_n, G, P,
                          Ma, Va, loss, err, lr, 0.9f, 0.999f, 1e-8f, c1, c2);
  }
  return launch_chained(true, reduce_kernel<false>, kMlpParams / kRedX, block, 0, st, part, losses, grid, a.inv_n, G, P,
                        Ma, Va, loss, err, 0.f, 0.f, 0.f, 0.f, 1.f, 1.f);
}

cudaError_t Mlp::gradients(const float* X, const float* Zt, int n) { return backward(X, Zt, n, false, 0.f); }
cudaError_t Mlp::train(const float* X, const float* Zt, int n, float lr) { return backward(X, Zt, n, true, lr); }

}  // namespace axpic

// ---------------------------------------------------------------- C ABI
#include "axpic.h"
#include <string>

struct axpic_mlp {
  axpic::Mlp m;
  std::string last_error;
  std::vector<float> mu = std::vector<float>(96, 0.f), sigma = std::vector<float>(96, 1.f);
  std::vector<float> skip = std::vector<float>(96 * 4, 0.f);  // S[o][i]
};

// The output model y = shape(x, kappa/T) + mu + S f_c + sigma z for the
// network's normalised output z (double) at the row's features f. shape
// carries each channel's exact x-dependence, so the learned part sees the
// cell features f_c = (0, f1, f2, f3): the network is evaluated at f_c and
// the ln x column of S multiplies zero.
static double model_output(const axpic_mlp* h, int o, const float* f, double z, double brems_shape) {
  double x, kT;
  axpic::sur_feature_xkt(f, &x, &kT);
  double y = axpic::sur_shape(o, x, kT, brems_shape) + (double)h->mu[o] + (double)h->sigma[o] * z;
  for (int i = 1; i < 4; ++i) y += (double)h->skip[o * 4 + i] * (double)f[i];
  return y;
}

// The network's inputs for feature rows X: the cell features (ln x column
// zeroed).
static std::vector<float> cell_features(const std::vector<float>& X) {
  std::vector<float> Xc(X);
  for (size_t r = 0; r < Xc.size() / 4; ++r) Xc[r * 4] = 0.f;
  return Xc;
}

extern "C" {

static axpic_status mlp_fail(axpic_mlp* h, cudaError_t e, const char* where) {
  h->last_error = std::string(where) + ": " + cudaGetErrorString(e);
  return AXPIC_E_CUDA;
}

static axpic_status mlp_sync(axpic_mlp* h, const char* where) {
  cudaError_t e = cudaStreamSynchronize(h->m.st);
  if (e) return mlp_fail(h, e, where);
  int herr = 0;
  if ((e = cudaMemcpy(&herr, h->m.err, sizeof(int), cudaMemcpyDeviceToHost))) return mlp_fail(h, e, where);
  if (herr) {
    h->last_error = std::string(where) + ": a tensor-core wait ran out";
    return AXPIC_E_TIMEOUT;
  }
  return AXPIC_OK;
}

axpic_status axpic_mlp_create(axpic_mlp** out, void* stream) {
  if (!out) return AXPIC_E_INVALID;
  *out = nullptr;
  axpic_mlp* h = new axpic_mlp();
  const cudaError_t e = h->m.init((cudaStream_t)stream);
  if (e) {
    fprintf(stderr, "axpic_mlp_create: %s\n", cudaGetErrorString(e));
    delete h;
    return AXPIC_E_CUDA;
  }
  *out = h;
  return AXPIC_OK;
}

axpic_status axpic_mlp_set_params(axpic_mlp* h, const float* params) {
  if (!h || !params) return AXPIC_E_INVALID;
  cudaError_t e = cudaMemcpyAsync(h->m.P, params, sizeof(float) * axpic::kMlpParams, cudaMemcpyHostToDevice, h->m.st);
  if (e) return mlp_fail(h, e, "axpic_mlp_set_params");
  h->m.t = 0;
  if ((e = cudaMemsetAsync(h->m.Ma, 0, sizeof(float) * axpic::kMlpParams, h->m.st)) ||
      (e = cudaMemsetAsync(h->m.Va, 0, sizeof(float) * axpic::kMlpParams, h->m.st)))
    return mlp_fail(h, e, "axpic_mlp_set_params");
  return mlp_sync(h, "axpic_mlp_set_params");
}

axpic_status axpic_mlp_get_params(axpic_mlp* h, float* params) {
  if (!h || !params) return AXPIC_E_INVALID;
  const cudaError_t e =
      cudaMemcpyAsync(params, h->m.P, sizeof(float) * axpic::kMlpParams, cudaMemcpyDeviceToHost, h->m.st);
  if (e) return mlp_fail(h, e, "axpic_mlp_get_params");
  return mlp_sync(h, "axpic_mlp_get_params");
}

axpic_status axpic_mlp_forward(axpic_mlp* h, const float* X, int32_t n, float* Z) {
  if (!h || n < 0 || (n > 0 && (!X || !Z))) return AXPIC_E_INVALID;
  const cudaError_t e = h->m.forward(X, n, Z);
  if (e) return mlp_fail(h, e, "axpic_mlp_forward");
  return AXPIC_OK;
}

axpic_status axpic_mlp_gradients(axpic_mlp* h, const float* X, const float* Zt, int32_t n, double* loss_out,
                                 float* grads) {
  if (!h || n < 0 || (n > 0 && (!X || !Zt))) return AXPIC_E_INVALID;
  cudaError_t e = h->m.gradients(X, Zt, n);
  if (e) return mlp_fail(h, e, "axpic_mlp_gradients");
  if (grads && (e = cudaMemcpyAsync(grads, h->m.G, sizeof(float) * axpic::kMlpParams, cudaMemcpyDeviceToHost,
                                    h->m.st)))
    return mlp_fail(h, e, "axpic_mlp_gradients");
  if (loss_out && (e = cudaMemcpyAsync(loss_out, h->m.loss, sizeof(double), cudaMemcpyDeviceToHost, h->m.st)))
    return mlp_fail(h, e, "axpic_mlp_gradients");
  return mlp_sync(h, "axpic_mlp_gradients");
}

axpic_status axpic_mlp_train_step(axpic_mlp* h, const float* X, const float* Zt, int32_t n, float lr,
                                  double* loss_out) {
  if (!h || n < 1 || !X || !Zt || !(lr > 0.f)) return AXPIC_E_INVALID;
  cudaError_t e = h->m.train(X, Zt, n, lr);
  if (e) return mlp_fail(h, e, "axpic_mlp_train_step");
  if (loss_out) {
    if ((e = cudaMemcpyAsync(loss_out, h->m.loss, sizeof(double), cudaMemcpyDeviceToHost, h->m.st)))
      return mlp_fail(h, e, "axpic_mlp_train_step");
    return mlp_sync(h, "axpic_mlp_train_step");
  }
  return AXPIC_OK;
}

axpic_status axpic_mlp_destroy(axpic_mlp* h) {
  if (!h) return AXPIC_E_INVALID;
  const axpic_status s = mlp_sync(h, "axpic_mlp_destroy");
  delete h;
  return s;
}

const char* axpic_mlp_last_error(const axpic_mlp* h) { return h ? h->last_error.c_str() : "no network"; }

axpic_status axpic_mlp_set_norm(axpic_mlp* h, const float* mu, const float* sigma) {
  if (!h || !mu || !sigma) return AXPIC_E_INVALID;
  for (int k = 0; k < 96; ++k) {
    if (!(sigma[k] >= 0.f) || !std::isfinite(sigma[k]) || !std::isfinite(mu[k])) return AXPIC_E_INVALID;
    h->mu[k] = mu[k];
    h->sigma[k] = sigma[k];
  }
  return AXPIC_OK;
}

axpic_status axpic_mlp_set_skip(axpic_mlp* h, const float* skip) {
  if (!h || !skip) return AXPIC_E_INVALID;
  for (int k = 0; k < 96 * 4; ++k) {
    if (!std::isfinite(skip[k])) return AXPIC_E_INVALID;
    h->skip[k] = skip[k];
  }
  return AXPIC_OK;
}

axpic_status axpic_mlp_get_skip(axpic_mlp* h, float* skip) {
  if (!h || !skip) return AXPIC_E_INVALID;
  for (int k = 0; k < 96 * 4; ++k) skip[k] = h->skip[k];
  return AXPIC_OK;
}

axpic_status axpic_mlp_get_norm(axpic_mlp* h, float* mu, float* sigma) {
  if (!h || !mu || !sigma) return AXPIC_E_INVALID;
  for (int k = 0; k < 96; ++k) {
    mu[k] = h->mu[k];
    sigma[k] = h->sigma[k];
  }
  return AXPIC_OK;
}

// Glorot-uniform weights and zero biases from a seeded stream.
static void glorot(uint64_t seed, std::vector<float>& P) {
  P.assign(axpic::kMlpParams, 0.f);
  uint64_t s = seed;
  auto u01 = [&s]() {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return ((z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
  };
  const int offs[3] = {axpic::kOffW1, axpic::kOffW2, axpic::kOffW3};
  const int fin[3] = {4, 64, 64}, fout[3] = {64, 64, 96};
  for (int l = 0; l < 3; ++l) {
    const double lim = std::sqrt(6.0 / (fin[l] + fout[l]));
    for (int i = 0; i < fin[l] * fout[l]; ++i) P[offs[l] + i] = (float)((2.0 * u01() - 1.0) * lim);
  }
}

axpic_status axpic_surrogate_fit(axpic_mlp* h, int32_t ncells, int32_t x_per_cell, int32_t steps, int32_t batch,
                                 float lr, uint64_t seed, double brems_shape, double* loss_out) {
  nvtxRangePushA("axpic_surrogate_fit");
  struct Pop {
    ~Pop() { nvtxRangePop(); }
  } pop_range_;
  if (!h || ncells < 1 || x_per_cell < 1 || steps < 1 || batch < 1 || !(lr > 0.f) || !(brems_shape > 0))
    return AXPIC_E_INVALID;
  std::vector<float> X;
  std::vector<double> Y;
  axpic::sur_training_set(ncells, x_per_cell, seed, brems_shape, X, Y);
  const size_t n = (size_t)ncells * x_per_cell;
  // The output model y = shape(x, kappa/T) + mu + S f_c + sigma z: the
  // network learns only what the exact x-shapes and an FP32 linear map of the
  // cell features leave over. mu and S by least squares over the rows (4 x 4
  // normal equations in FP64 over (1, f1, f2, f3), 96 right-hand sides; the
  // ln x column of S is zero); sigma is the residual's spread, divided by
  // kRateWeight on the ln-emissivity outputs so that their errors weigh more
  // in the loss.
#ifndef AXPIC_RATE_WEIGHT
#define AXPIC_RATE_WEIGHT 16.0
#endif
  constexpr double kRateWeight = AXPIC_RATE_WEIGHT;
  for (size_t r = 0; r < n; ++r) {
    double x, kT;
    axpic::sur_feature_xkt(&X[r * 4], &x, &kT);
    for (int k = 0; k < 96; ++k) Y[r * 96 + k] -= axpic::sur_shape(k, x, kT, brems_shape);
  }
  constexpr int kD = 4;  // 1, f1, f2, f3
  double M[kD][kD + 96] = {};
  for (size_t r = 0; r < n; ++r) {
    const double d[kD] = {1.0, X[r * 4 + 1], X[r * 4 + 2], X[r * 4 + 3]};
    for (int i = 0; i < kD; ++i) {
      for (int j = 0; j < kD; ++j) M[i][j] += d[i] * d[j];
      for (int k = 0; k < 96; ++k) M[i][kD + k] += d[i] * Y[r * 96 + k];
    }
  }
  for (int c = 0; c < kD; ++c) {  // Gauss-Jordan with partial pivoting
    int p = c;
    for (int i = c + 1; i < kD; ++i)
      if (std::fabs(M[i][c]) > std::fabs(M[p][c])) p = i;
    if (!(std::fabs(M[p][c]) > 0.0)) return AXPIC_E_INVALID;  // degenerate feature draw
    for (int j = 0; j < kD + 96; ++j) std::swap(M[c][j], M[p][j]);
    for (int i = 0; i < kD; ++i) {
      if (i == c) continue;
      const double g = M[i][c] / M[c][c];
      for (int j = c; j < kD + 96; ++j) M[i][j] -= g * M[c][j];
    }
  }
  for (int k = 0; k < 96; ++k) {
    h->mu[k] = (float)(M[0][kD + k] / M[0][0]);
    h->skip[k * 4] = 0.f;
    for (int i = 1; i < kD; ++i) h->skip[k * 4 + i] = (float)(M[i][kD + k] / M[i][i]);
  }
  // The Compton-like and bremsstrahlung quantiles do not depend on the cell
  // (their number spectra in x are universal): the model carries them as
  // constants, mu = the exact knots, with S and sigma zero, so the step can
  // sample from one row for every cell.
  double uni[93];
  axpic::sur_universal_knots(brems_shape, uni);
  for (int k = 0; k < 96; ++k)
    if (axpic::sur_universal_output(k)) {
      h->mu[k] = (float)uni[31 * (k / 32) + k % 32 - 1];
      for (int i = 0; i < kD; ++i) h->skip[k * 4 + i] = 0.f;
    }
  // residuals with the binary32 coefficients the model keeps
  std::vector<double> var(96, 0.0);
  for (size_t r = 0; r < n; ++r)
    for (int k = 0; k < 96; ++k) {
      double lin = h->mu[k];
      for (int i = 1; i < 4; ++i) lin += (double)h->skip[k * 4 + i] * (double)X[r * 4 + i];
      Y[r * 96 + k] -= lin;
      var[k] += Y[r * 96 + k] * Y[r * 96 + k];
    }
  // Floors on sigma: what is left below them (the binary32 rounding of mu + S
  // f on the outputs the linear map already carries exactly) is not the
  // network's to learn. 1e-4 in ln rate (a tenth of the rate bound), 1e-5 in
  // x on the quantiles.
#ifndef AXPIC_SIGMA_FLOOR_RATE
#define AXPIC_SIGMA_FLOOR_RATE 1e-4
#endif
#ifndef AXPIC_SIGMA_FLOOR_Q
#define AXPIC_SIGMA_FLOOR_Q 1e-5
#endif
  for (int k = 0; k < 96; ++k) {
    const bool rate = k % 32 == 0;
    const double floor = rate ? AXPIC_SIGMA_FLOOR_RATE : AXPIC_SIGMA_FLOOR_Q;
    h->sigma[k] = axpic::sur_universal_output(k)
                      ? 0.f
                      : (float)(std::max(std::sqrt(var[k] / (double)n), floor) / (rate ? kRateWeight : 1.0));
  }
  // normalised targets; the network's outputs that sigma zeroes learn zero
  std::vector<float> Zt(n * 96);
  for (size_t r = 0; r < n; ++r)
    for (int k = 0; k < 96; ++k)
      Zt[r * 96 + k] = h->sigma[k] > 0.f ? (float)(Y[r * 96 + k] / h->sigma[k]) : 0.f;
  X = cell_features(X);  // the network's inputs
  std::vector<float> P;
  glorot(seed ^ 0xA5A5A5A5u, P);
  axpic_status s = axpic_mlp_set_params(h, P.data());
  if (s != AXPIC_OK) return s;
  float *dX = nullptr, *dZ = nullptr;
  cudaError_t e;
  if ((e = cudaMalloc(&dX, sizeof(float) * X.size())) || (e = cudaMalloc(&dZ, sizeof(float) * Zt.size()))) {
    cudaFree(dX);
    return mlp_fail(h, e, "axpic_surrogate_fit");
  }
  e = cudaMemcpyAsync(dX, X.data(), sizeof(float) * X.size(), cudaMemcpyHostToDevice, h->m.st);
  if (!e) e = cudaMemcpyAsync(dZ, Zt.data(), sizeof(float) * Zt.size(), cudaMemcpyHostToDevice, h->m.st);
  // rows were drawn independently: consecutive batches are random batches
  const int nb = (int)std::max<size_t>(1, n / (size_t)batch);
  for (int t = 0; t < steps && !e; ++t) {
    const int b = t % nb;
    const float lr_t = lr * (0.01f + 0.99f * 0.5f * (1.0f + cosf(3.14159265f * (float)t / (float)steps)));
    e = h->m.train(dX + (size_t)b * batch * 4, dZ + (size_t)b * batch * 96, batch, lr_t);
  }
  if (!e) e = h->m.gradients(dX, dZ, (int)n);
  double loss = 0.0;
  if (!e) e = cudaMemcpyAsync(&loss, h->m.loss, sizeof(double), cudaMemcpyDeviceToHost, h->m.st);
  if (!e) e = cudaStreamSynchronize(h->m.st);
  cudaFree(dX);
  cudaFree(dZ);
  if (e) return mlp_fail(h, e, "axpic_surrogate_fit");
  if (loss_out) *loss_out = loss;
  return mlp_sync(h, "axpic_surrogate_fit");
}

axpic_status axpic_surrogate_validate(axpic_mlp* h, int32_t nT, int32_t nne, double brems_shape, float* err_out) {
  nvtxRangePushA("axpic_surrogate_validate");
  struct Pop {
    ~Pop() { nvtxRangePop(); }
  } pop_range_;
  if (!h || nT < 2 || nne < 2 || nT > 4096 || nne > 4096 || !err_out || !(brems_shape > 0)) return AXPIC_E_INVALID;
  // the learned part of every output is a function of the cell (the
  // x-dependence is the exact shape), so a few x per node suffice
  const int nodes = nT * nne * 2, nx = 8;
  std::vector<float> X((size_t)nodes * nx * 4);
  std::vector<double> Y((size_t)nodes * nx * 96);
  double uni[93];
  axpic::sur_universal_knots(brems_shape, uni);
  const int nth = (int)std::max(1u, std::min(32u, std::thread::hardware_concurrency()));
  {
    std::vector<std::thread> th;
    for (int t = 0; t < nth; ++t)
      th.emplace_back([&, t]() {
        double knots[93];
        for (int node = t; node < nodes; node += nth) {
          const int i = node % nT, j = (node / nT) % nne, z = node / (nT * nne);
          const double T = axpic::kSurTLo * std::pow(axpic::kSurTHi / axpic::kSurTLo, i / (double)(nT - 1));
          const double ne = std::pow(10.0, 23.0 + 3.0 * j / (nne - 1));
          const double Z = z + 1.0;
          const axpic::SurCell c = axpic::sur_cell(T, ne, Z, brems_shape);
          axpic::sur_knots(c, knots, uni);
          for (int k = 0; k < nx; ++k) {
            const double x = axpic::kSurXLo * std::pow(axpic::kSurXHi / axpic::kSurXLo, k / (double)(nx - 1));
            const size_t r = (size_t)node * nx + k;
            axpic::sur_features(x, c.kappa / T, ne, Z, &X[r * 4]);
            axpic::sur_targets(x, c, knots, &Y[r * 96]);
          }
        }
      });
    for (auto& x : th) x.join();
  }
  const size_t n = (size_t)nodes * nx;
  float *dX = nullptr, *dZ = nullptr;
  cudaError_t e;
  if ((e = cudaMalloc(&dX, sizeof(float) * X.size())) || (e = cudaMalloc(&dZ, sizeof(float) * n * 96))) {
    cudaFree(dX);
    return mlp_fail(h, e, "axpic_surrogate_validate");
  }
  std::vector<float> Z(n * 96);
  const std::vector<float> Xc = cell_features(X);
  e = cudaMemcpyAsync(dX, Xc.data(), sizeof(float) * Xc.size(), cudaMemcpyHostToDevice, h->m.st);
  if (!e) e = h->m.forward(dX, (int)n, dZ);
  if (!e) e = cudaMemcpyAsync(Z.data(), dZ, sizeof(float) * Z.size(), cudaMemcpyDeviceToHost, h->m.st);
  if (!e) e = cudaStreamSynchronize(h->m.st);
  cudaFree(dX);
  cudaFree(dZ);
  if (e) return mlp_fail(h, e, "axpic_surrogate_validate");
  // per node: the largest error of ln(dQ/dx) over the x grid and channels
  // (the relative rate error), of the Compton-like and bremsstrahlung
  // quantiles (those the step samples emission energies from) and of the
  // Primakoff quantiles, relative to x
  for (int node = 0; node < nodes; ++node) {
    double eL = 0.0, eQ = 0.0, eQP = 0.0;
    for (int k = 0; k < nx; ++k) {
      const size_t r = (size_t)node * nx + k;
      for (int o = 0; o < 96; ++o) {
        const double y = model_output(h, o, &X[r * 4], (double)Z[r * 96 + o], brems_shape);
        const double d = std::fabs(y - Y[r * 96 + o]);
        if (o % 32 == 0) eL = std::max(eL, d);
        else if (o < 32) eQP = std::max(eQP, d / Y[r * 96 + o]);
        else eQ = std::max(eQ, d / Y[r * 96 + o]);
      }
    }
    err_out[3 * node] = (float)eL;
    err_out[3 * node + 1] = (float)eQ;
    err_out[3 * node + 2] = (float)eQP;
  }
  return AXPIC_OK;
}

}  // extern "C"
