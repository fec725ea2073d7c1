// Row bookkeeping and kernel arguments of a quantization step, shared by the kernels of the group loop.
#pragma once

#include "tb_common.cuh"
#include "tb_i8.cuh"

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

// Column sweep (Algorithm 2; Eq. 2) of one step's rows over the blocks of 128 columns [blk0, blk1) (tb_sweep.cu).
struct SweepArgs {
  const double* src;     // values before the sweep, row m of the step at src + src_row(m) d
  bool src_mapped;       // src_row(m) = rm.row(m) (the weights), else m (a working copy of the step's rows)
  const float* U;        // [n_hin][d][d]
  const float* P;        // [n_hin][d][d] or nullptr
  double* Err;           // [M][err_ld] out: normalised errors, column c at c - err_col0
  double* Arr;           // the same for arrival values (with P)
  int err_ld, err_col0;
  unsigned char* codes;  // [d_out][d]
  const double* sD;      // [d_out][ng]
  const int* z;          // [d_out][ng]
  tb_stats* stats;       // or nullptr
  RowMap rm;
  int M, d, seg, ng, maxq;
  int units;             // 1, or the number of heads when every head has its own U
  int blk0, blk1;
};
tb_status sweep_columns(const SweepArgs& a, cudaStream_t st);

// The sweep over all columns of a step.  Up to SWEEP_OUTER columns go through in one launch; more are taken that many at
// a time, each followed by one update of everything further right in a working copy of the step's rows.
enum { SWEEP_OUTER = 512, SWEEP_I8_WORK = 1200000 };
struct SweepScratch {
  double *work;          // [M][d]
  double *err, *arr;     // [M][SWEEP_OUTER], arr with P only
  bool use_i8;           // the updates on the integer tensor cores (one shared U, sweep_wants_i8); then:
  I8Mat Udig, Pdig;      // digits of U and P by columns (prepared by sweep_prepare, one set for all steps)
  I8Mat Edig, Adig;      // digits of a block's errors and arrival values
  unsigned long long *u_max, *p_max, *e_max, *a_max;
  int* u_exp;            // exponents of U's diagonal
};
bool sweep_wants_i8(int d, int units, int rows_per_unit);
void sweep_scratch(Bump& b, int M, int d, bool with_p, bool use_i8, SweepScratch* s);  // err .. u_exp
tb_status sweep_prepare(const float* U, const float* P, int d, const SweepScratch& s, cudaStream_t st);
// a.src: the weights (mapped); a.Err, a.Arr, blk0, blk1 and the like are set here
tb_status sweep_step(SweepArgs a, const SweepScratch& s, cudaStream_t st);

// Dynamic-grid variant of the sweep (the grid of a column group is searched when the sweep arrives at the group, from the
// group's current values).  Right-looking, one column group of up to 128 columns at a time on a contiguous working copy of
// the step's rows: the search, then group_panel: Algorithm 2's column loop restricted to the group, and the rank-seg
// update of every column right of it.
struct GroupPanelP {
  double* Wk;            // [M][d] working copy of the step's rows
  const float* U;        // [n_hin][d][d]
  const float* P;        // or nullptr
  double* Err;           // [M][seg] normalised errors of this group
  double* Arr;           // [M][seg] arrival values of this group (with P)
  unsigned char* codes;  // [d_out][d]
  const double* sD;      // [d_out][ng]
  const int* z;          // [d_out][ng]
  tb_stats* stats;
  RowMap rm;
  int M, d, seg, ng, maxq, grp;
  int units, rows_per_unit;
};
tb_status group_panel(const GroupPanelP& p, cudaStream_t st);

// Scale refinement of heads with few coordinates (d_head x groups) as a triangular solve (tb_cd_gram.cu).
enum { CD_GRAM_MAX = 2048 };
struct CdGram {
  const void* Yw;      // [heads dh][ng][d], float or double
  bool yw_float;
  const float* Wb;     // [heads dh][d]
  const float* Hout;   // [heads][dh][dh]
  double* scratch;     // cd_gram_doubles
  int heads, d, seg, ng, dh;
};
bool cd_gram_pays(int heads, int dh, int ng);  // heads of a batch
size_t cd_gram_doubles(int heads, int dh, int ng);
tb_status cd_gram_form(const CdGram& p, cudaStream_t st);
tb_status cd_gram_pass(const CdGram& p, const double* G, double* Dm, double* sD, cudaStream_t st);

// The search for column groups wider than 128 columns (tb_grid_wide.cu).  scratch: grid_wide_doubles() doubles
// for a chunk of rows; with less, the rows go through in several chunks.
size_t grid_wide_row_doubles(int d, int ng, int ncp);  // doubles of scratch per row
tb_status grid_wide(const GridP& p, double* scratch, size_t scratch_doubles, cudaStream_t st);

// The search with many rows, any group width, on the integer tensor cores (tb_grid_digits.cu).
struct GridDigits {
  int rows;              // rows per chunk
  unsigned char *A, *B;  // integers of the candidates, digits of H_in (one set for all steps)
  double *h, *r, *range, *lin, *part;
  unsigned int* hmax;
  int* list;
};
bool grid_wants_digits(int M, int units, int d, int seg, int ncp);
void grid_digits_scratch(Bump& b, int M, int units, int d, int seg, int ncp, int bits, GridDigits* s);
tb_status grid_digits_prepare(const float* H, int units, int d, int seg, const GridDigits& s, cudaStream_t st);
tb_status grid_digits(const GridP& p, const GridDigits& s, cudaStream_t st);

}  // namespace tb
