// Axion merging for population control (internal to libaxpic).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace axpic {

constexpr int kMergeMaxEdges = 30;  // |p|^2 thresholds: (30 + 1) bins x 8 octants = 248 groups
constexpr int kMergeMaxCap = 65535; // slots per cell, u16 member indices (slabs hold at most 65532)

struct MergeArgs {
  SpeciesPtrs s;     // the axion slabs
  int ncells;
  int n_target;      // cells holding more axions than this are merged
  int nedges;
  float edges[kMergeMaxEdges];  // ascending binary32 thresholds of |p|^2 (m_e c)^2
  double* removed;   // [1]: axions removed so far
};

// Sets the merge kernel's shared-memory limit and works out its largest grid
// for slabs of cap slots; called before a context's first launch.
cudaError_t merge_init_kernels(int cap, int* fit);
cudaError_t launch_merge(const MergeArgs& a, int fit, cudaStream_t st);

}  // namespace axpic
