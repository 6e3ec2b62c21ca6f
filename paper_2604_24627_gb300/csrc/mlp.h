// The surrogate MLP on the GPU (internal to libaxpic).
#pragma once
#include <cuda_runtime.h>

namespace axpic {

// Parameter layout (FP32): W1[4][64], b1[64], W2[64][64], b2[64], W3[64][96], b3[96].
constexpr int kOffW1 = 0, kOffB1 = 256, kOffW2 = 320, kOffB2 = 4416, kOffW3 = 4480, kOffB3 = 10624;
constexpr int kMlpParams = 10720;

struct Mlp {
  cudaStream_t st = nullptr;
  float *P = nullptr, *G = nullptr, *Ma = nullptr, *Va = nullptr;  // params, grads, Adam moments
  float* part = nullptr;     // each training CTA's gradients
  double* losses = nullptr;  // and its sum of squares
  int* err = nullptr;
  double* loss = nullptr;
  int sms = 1;
  long t = 0;  // Adam steps taken

  ~Mlp();
  cudaError_t init(cudaStream_t s);
  cudaError_t reserve_train();
  // out[n][96] = network(X[n][4]) (normalised outputs)
  cudaError_t forward(const float* X, int n, float* out);
  // G = d loss / d P and *loss, loss = sum (z - Zt)^2 / n
  cudaError_t gradients(const float* X, const float* Zt, int n);
  // the same gradients applied by one Adam step (G is not written)
  cudaError_t train(const float* X, const float* Zt, int n, float lr);

 private:
  cudaError_t backward(const float* X, const float* Zt, int n, bool adam, float lr);
};

}  // namespace axpic
