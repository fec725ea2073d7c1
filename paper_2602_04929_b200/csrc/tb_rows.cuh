// Row bookkeeping and kernel arguments of a quantization step, shared by the kernels of the group loop.
#pragma once

#include "tb_common.cuh"

namespace tb {

// Active row m of a step maps to head m / g, row i0 + m % g of that head.  "Units" are sets of rows
// that share one H_in / U_in: the whole step when H_in is shared, one head otherwise.
struct RowMap {
  int g, d_head, i0;
  __host__ __device__ long long row(int m) const {
    return (long long)(m / g) * d_head + i0 + (m % g);
  }
};

// Grid search (Algorithm 1, grid step) of one step's rows.
struct GridP {
  const double* Wt;   // [d_out][d]
  const float* Hin;   // [n_hin][d][d]
  double* sD;         // [d_out][ng]
  float* s_out;       // [d_out][ng]
  int* z_out;         // [d_out][ng]
  unsigned char* cand_out;  // or nullptr
  RowMap rm;
  int M, d, seg, ng, maxq, n_cand, ncp, rt;
  int units, rows_per_unit, tiles_per_unit;
  const double* Wloc;  // or nullptr: the step's rows as a contiguous [M][d] working copy, read instead of Wt
  int grp0;            // column group of blockIdx.x = 0
};

// The search for column groups wider than 128 columns (tb_grid_wide.cu).  scratch: grid_wide_doubles() doubles
// for a chunk of rows; with less, the rows go through in several chunks.
size_t grid_wide_row_doubles(int d, int ng, int ncp);  // doubles of scratch per row
tb_status grid_wide(const GridP& p, double* scratch, size_t scratch_doubles, cudaStream_t st);

}  // namespace tb
