// Axion free streaming and cell migration (internal to libaxpic).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace axpic {

// Direction of an axion after a move: the cell shift (sx, sy, sz) in {-1, 0, 1}^3
// as (sz + 1) 9 + (sy + 1) 3 + (sx + 1); 13 stays.
constexpr int kStreamDirs = 27, kStreamStay = 13;
// 16-bit entries a cell of the staging offsets: entry d the leavers with a
// direction below d, entry 27 all of them (64 bytes, two sectors)
constexpr int kStreamOffs = 32;

// rows of the escape and drop sums, added up when they are read, and doubles per
// row (a 128-byte line)
constexpr int kStreamRows = 128, kStreamRow = 16;

struct StreamArgs {
  SpeciesPtrs s;       // the axion slabs (positions rewritten, slots re-binned)
  int ncells, nx, ny, nz;
  float kappa;         // binary32(c dt / h): the cell fraction moved at |v| = c
  float mu;            // binary32(m_a c^2 / m_e c^2): the axion mass in units of the momenta
  int periodic;        // 1 periodic, 0 open
  uint32_t* freed;     // [ncells * ceil(cap / 32)]: a bit per slot whose axion does not stay
  uint16_t* goff;      // [ncells * kStreamOffs]: each direction's first row in the cell's staging rows
  float* buf;          // [ncells * cap * 8]: the cell's leaving axions, grouped by direction
  double* stats;       // [kStreamRows * kStreamRow], each row's first 4: escaped number, weight, weight x energy [keV]; dropped number
  int* err;            // latched error flags (ERR_CAPACITY)
};

cudaError_t launch_stream(const StreamArgs& a, cudaStream_t st);

}  // namespace axpic
