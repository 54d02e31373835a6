// One-sided evaluation of an i set against another j set: launch arguments
// and entry points of rows_kernel (cn_rows.cuh).
#pragma once

#include "cn_kernels.h"

namespace cn {

// A row is one tile of i-particles against all j records, in blocks of 32.
// The rows' blocks lie one after the other on a line, which is split evenly
// over the CTAs.
constexpr int kRowBlock = 32;

struct RowArgs {
  const float4* pos_i;
  const float4* pos_j;
  float* acc_out;
  float* pot_out;          // or NULL
  float* segs;             // [2 grid][sums][tile]: a CTA's sums of a row that began before its part, and of its last row
  int* status;
  int64_t n_i, n_j;
  int64_t units;           // blocks of all rows
  int32_t n_rows;
  int32_t blocks;          // per row
  int32_t grid;
  int32_t tile;            // i-particles per row: 32 K x warps along i
  int32_t wi;              // warps along i (the others split the j records)
  int32_t chunk;           // j records per ring stage
  int32_t stages;          // at least 3
  float eps2;
  uint64_t wait_ns;

  // first unit of CTA g's part (grid <= units: every part has one), and the CTA of a unit
  __host__ __device__ int64_t part(int64_t g) const { return (g * units + grid - 1) / grid; }
  __host__ __device__ int64_t owner(int64_t u) const { return (u * grid) / units; }
};

enum RowForm : int {
  kRowForce = 0,
  kRowForcePot = 1,
  kRowEpsI = 2,     // softening per i-particle
  kRowEpsIPot = 3,
};

size_t rows_smem_bytes(RowForm form, int k, int chunk, int stages);
cudaError_t occupancy_rows(RowForm form, int k, size_t smem, int* ctas);
cudaError_t launch_rows(RowForm form, int k, const RowArgs& a, size_t smem, cudaStream_t s);

}  // namespace cn
