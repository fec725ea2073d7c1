// tb_quantize_layer: the out-channel-group loop of Algorithm 1 and its closing steps.
//
// Per step i (a group of g = out_block rows of every head, M = n_heads * g
// rows in all, heads being independent):
//   grid     k_grid_tri       Algorithm 1, grid     candidate search per (row, column group); tb_grid_wide.cu,
//                                                   tb_grid_digits.cu
//   sweep    k_sweep_rows     Algorithm 2 / Eq. 2   one launch, 8 to 32 rows per CTA for the whole sweep (tb_sweep.cu)
//   update   k_compensate     W~[rem] -= T_i E      (Algorithm 1, update), E = W0 - Q_B (Proposition 3.1);
//            with R first k_residual and a product: E -= W0 C (Proposition 3.2)
// then, once: coordinate descent on the scales (Algorithm 3), Q = s (W_int - z),
// and the loss of the proofs of Propositions 3.1 / 3.2.
//
// All of this runs in IEEE double, on the FP64 pipe or as exact digit products on the integer tensor cores
// (tb_i8.cuh, tb_grid_digits.cu).  The codes are integer
// decisions inside an error-feedback chain d_in steps long; in float the
// accumulated rounding error of the chain (a few 1e-6 code units) exceeds the
// 1e-6 band inside which a rounding decision may legitimately differ, and one
// different decision changes every later code of its row.
#include <cooperative_groups.h>

#include "tb_common.cuh"
#include "tb_gemm.cuh"
#include "tb_i8.cuh"
#include "tb_profile.cuh"
#include "tb_rows.cuh"
#include "tb_tma.cuh"

namespace cg = cooperative_groups;

namespace tb {
// tensor-core blockwise product of the scale refinement (tb_gemm_tc.cu)
tb_status yw_tensor(float* Yw, const unsigned char* codes, const int* zeros, const float* H_in, __nv_bfloat16* WbT,
                    __nv_bfloat16* Hp, bool split_h, long long rows, int d, int seg, int ng, int hunits,
                    cudaStream_t st);
// C = alpha A B (+ add) in double from operands split into three bf16 pieces each (tb_gemm_tc.cu)
tb_status gemm_split_presplit(double* C, long long ldc, const __nv_bfloat16* AT, const __nv_bfloat16* Bp, long long M,
                              int N, int K, const double* add, cudaStream_t st, int hunits = 1, double alpha = 1.0);
tb_status split3_transpose(const double* A, __nv_bfloat16* AT, long long M, int K, cudaStream_t st);
tb_status split3_transpose(const float* A, __nv_bfloat16* AT, long long M, int K, cudaStream_t st);
tb_status split3(const float* B, __nv_bfloat16* Bp, long long n, cudaStream_t st);
}

namespace tb {

__global__ void k_widen(const float* __restrict__ W, double* __restrict__ Wt, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    Wt[i] = (double)W[i];
}

// Wk[m][:] = W~[row(m)][:]  (and a second untouched copy W0c when the
// propagated-error term needs the snapshot as a contiguous GEMM operand)
__global__ void k_gather(const double* __restrict__ Wt, double* __restrict__ Wk,
                         double* __restrict__ W0c, RowMap rm, int M, int d) {
  const long long n = (long long)M * d;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(i / d), k = (int)(i % d);
    const double v = Wt[rm.row(m) * d + k];
    Wk[i] = v;
    if (W0c) W0c[i] = v;
  }
}

// ---------------------------------------------------------------------------
// Compensation matrices of Propositions 3.1 / 3.2 for every head and step:
//   T = [U_out^T]_{rem,B} ([U_out^T]_{B,B})^{-1},  B = {i0..i0+g-1}, rem = rows after B.
// With A = U_out^T lower triangular, T A_BB = A_remB is solved row by row,
// last column first.  T is stored [head][step][d_head][g] (first rem rows used).
// ---------------------------------------------------------------------------
// The g factor rows of the step are staged in shared memory ([c][column from i0 on], when they fit); four threads
// share a row, every fourth term of a dot product each.  Bound by the chain of g divisions and dot products: two steps of
// 64 rows in 8 heads of 128 take 54 us (76 with a thread per row).
__global__ void k_comp_matrices(const float* __restrict__ Uout, double* __restrict__ T, int dh,
                                int g, int n_steps, int staged) {
  extern __shared__ __align__(16) float cm_u[];
  const int step = blockIdx.x, head = blockIdx.y;
  const int i0 = step * g, r0 = i0 + g, nrem = dh - r0;
  if (nrem <= 0) return;
  const float* Uo = Uout + (long long)head * dh * dh;
  double* Th = T + ((long long)head * n_steps + step) * dh * g;
  const int w = dh - i0;
  if (staged) {
    for (int i = threadIdx.x; i < g * w; i += blockDim.x) cm_u[i] = Uo[(long long)(i0 + i / w) * dh + i0 + i % w];
    __syncthreads();
  }
  const int part = threadIdx.x & 3, slot = threadIdx.x >> 2;
  for (int rb = 0; rb < nrem; rb += 128) {
    const int r = rb + slot;
    const bool on = r < nrem;
    double* Tr = Th + (long long)(on ? r : 0) * g;
    // the row under construction: in shared memory where the factor rows are, [c][row]
    double* ct = staged ? reinterpret_cast<double*>(cm_u + (((size_t)g * dh + 3) & ~(size_t)3)) + slot : Tr;
    const int cs = staged ? 128 : 1;
    for (int c = g - 1; c >= 0; --c) {
      const float* urow = staged ? cm_u + c * w - i0 : Uo + (long long)(i0 + c) * dh;
      double v0 = 0.0, v1 = 0.0;
      if (on) {
        if (part == 0) v0 = (double)urow[r0 + r];
        int c2 = c + 1 + part;
        for (; c2 + 4 < g; c2 += 8) {
          v0 = fma(-ct[c2 * cs], (double)urow[i0 + c2], v0);
          v1 = fma(-ct[(c2 + 4) * cs], (double)urow[i0 + c2 + 4], v1);
        }
        if (c2 < g) v0 = fma(-ct[c2 * cs], (double)urow[i0 + c2], v0);
      }
      v0 += v1;
      v0 += __shfl_xor_sync(0xffffffffu, v0, 1);
      v0 += __shfl_xor_sync(0xffffffffu, v0, 2);
      if (on && part == 0) ct[c * cs] = v0 / (double)urow[i0 + c];
      __syncwarp();
    }
    if (staged && on)
      for (int c = part; c < g; c += 4) Tr[c] = ct[c * cs];
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Grid search (Algorithm 1, grid step).  For every (row, column group): n_cand
// clipped min-max grids, p_k = 1 - k/32; score e H_in[G,G] e^T with e the
// round-to-nearest error on that grid; the lowest score wins, lowest k on ties.
// Groups wider than 128 columns: tb_grid_wide.cu; many rows: tb_grid_digits.cu.  Here the search
// for groups of at most 128 columns, where the whole problem of a CTA (128
// candidate rows x one group) fits shared memory.  One CTA takes RT = 128 / NCP
// rows (NCP = n_cand rounded up to a power of two) of one column group:
// RT * NCP = 128 "candidate rows".  H_in[G,G] is symmetric,
// so e H e^T = 2 e T e^T with T the upper triangle of H (diagonal halved): only the
// part k <= n of the product is formed, about half of the tensor-pipe work.  The
// scores are compared, never output, so the factor 2 is dropped.  The candidate
// errors are staged once (and read again for the row dots), T as float; after one
// barrier the product runs without further synchronisation.  Column fragments
// (8 columns) are dealt to the warps so that every warp has the same share of the
// triangle: warp column c owns fragments c, 7-c, 8+c, 15-c.  Reads the upper
// triangle of H_in only.
// ---------------------------------------------------------------------------
enum { GT_LDE = 132, GT_LDB = 136 };
static constexpr size_t GRID_TRI_SMEM = (size_t)128 * GT_LDE * sizeof(double) + (size_t)128 * GT_LDB * sizeof(float);

__global__ void __launch_bounds__(GEMM_THREADS, 1) k_grid_tri(GridP p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* Es = reinterpret_cast<double*>(smem_raw);                                    // [k][candidate row]
  float* Bs = reinterpret_cast<float*>(smem_raw + (size_t)128 * GT_LDE * sizeof(double));  // [k][n]
  __shared__ double c_s[128], c_rs[128], c_z[128], c_J[128];
  __shared__ long long c_row[128];  // global row of a candidate row, or -1
  __shared__ long long c_src[128];  // element offset of that row's first column in the source matrix

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = p.grp0 + blockIdx.x;
  const int unit = blockIdx.y / p.tiles_per_unit;
  const double* Wsrc = p.Wloc ? p.Wloc : p.Wt;
  const int tile = blockIdx.y % p.tiles_per_unit;
  const int seg0 = grp * p.seg;
  const int d = p.d, seg = p.seg;
  const double maxq = (double)p.maxq;
  const float* H = p.Hin + (long long)unit * p.d * p.d * (p.units > 1 ? 1 : 0);

  // T = upper triangle of H_in[G,G], diagonal halved; issued first, it lands while phase 1 runs
  {
    const int n = tid & 127;
    float hv[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      const int k = (tid >> 7) + 2 * i;
      hv[i] = (k <= n && n < seg) ? H[(long long)(seg0 + k) * d + seg0 + n] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) {
      const int k = (tid >> 7) + 2 * i;
      Bs[k * GT_LDB + n] = (k == n) ? 0.5f * hv[i] : hv[i];
    }
  }

  // Phase 1: min / max of every row segment, then the candidates' (s, z).
  for (int r = warp; r < p.rt; r += GEMM_THREADS / 32) {
    const int rloc = tile * p.rt + r;
    const bool valid = rloc < p.rows_per_unit;
    long long grow = -1, src = 0;
    double mn = 0.0, mx = 0.0;
    if (valid) {
      grow = p.rm.row(unit * p.rows_per_unit + rloc);
      src = (p.Wloc ? (long long)(unit * p.rows_per_unit + rloc) : grow) * p.d;
      const double* w = Wsrc + src + seg0;
      for (int a = lane; a < p.seg; a += 32) {
        const double v = w[a];
        mn = fmin(mn, v);
        mx = fmax(mx, v);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
    }
    if (lane < p.ncp) {
      const int k = lane, cr = r * p.ncp + k;
      double s = 1.0, z = 0.0;
      if (valid && k < p.n_cand) {
        const double pk = 1.0 - (double)k / 32.0;
        const double lo = pk * mn, hi = pk * mx;
        if (hi != lo) {
          s = (hi - lo) / maxq;
          z = fmin(fmax(rne(-lo / s), 0.0), maxq);
        }
      }
      c_s[cr] = s;
      c_rs[cr] = 1.0 / s;
      c_z[cr] = z;
      c_row[cr] = (valid && k < p.n_cand) ? grow : -1;
      c_src[cr] = src;
    }
  }
  __syncthreads();

  // Phase 2: the candidates' round-to-nearest errors, Es[k][cr] (0 outside the problem)
  {
    const int cr = tid & 127;
    const long long grow = c_row[cr];
    const double s = c_s[cr], rs = c_rs[cr], z = c_z[cr];
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    const double zm = z + magic;
    const double* w = Wsrc + (grow < 0 ? 0 : c_src[cr]) + seg0;
#pragma unroll 8
    for (int i = 0; i < 64; ++i) {
      const int k = (tid >> 7) + 2 * i;
      double e = 0.0;
      if (grow >= 0 && k < seg) {
        // the fused multiply-add into z + 1.5 * 2^52 rounds to nearest-even and leaves the integer in the
        // low word (|v / s + z| < 2^31), where the clamp is two integer instructions
        const double v = w[k];
        int n = __double2loint(fma(v, rs, zm));
        n = min(max(n, 0), p.maxq);
        const double q = __hiloint2double(0x43380000, n) - magic;
        e = v - s * (q - z);
      }
      Es[k * GT_LDE + cr] = e;
    }
  }
  __syncthreads();

  // Phase 3: acc = E T on the FP64 tensor pipe, fragments with k <= n only
  const int wc = warp & 3, kq = lane & 3, rq = lane >> 2;
  int fr[4];
  fr[0] = wc;
  fr[1] = 7 - wc;
  fr[2] = 8 + wc;
  fr[3] = 15 - wc;
  double acc[8][4][2];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
  const double* ap = Es + kq * GT_LDE + (warp >> 2) * 64 + rq;
  const float* bp = Bs + kq * GT_LDB + rq;
  const int k4_end = (seg + 3) / 4;
#pragma unroll 1
  for (int k4 = 0; k4 < k4_end; ++k4) {
    double a[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = ap[k4 * 4 * GT_LDE + i * 8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (8 * fr[j] + 7 < 4 * k4 || 8 * fr[j] >= seg) continue;  // wholly below the diagonal, or outside the group
      const double b = (double)bp[k4 * 4 * GT_LDB + 8 * fr[j]];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        dmma(acc[i][j], a[i], b);
    }
  }

  // Phase 4: row dots of (E T) with E.  A candidate row's score is spread over the 4 lanes of a
  // quad and the 4 warps that share its rows; quads reduce by shuffle, warps through shared
  // memory in a fixed order.
  double jpart[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int cr = (warp >> 2) * 64 + i * 8 + rq;
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = 8 * fr[j] + 2 * kq;
      v = fma(acc[i][j][0], Es[n * GT_LDE + cr], v);
      v = fma(acc[i][j][1], Es[(n + 1) * GT_LDE + cr], v);
    }
    jpart[i] = v;
  }
  __syncthreads();  // every warp is done with Bs: its storage takes the partial scores
  double* c_Jw = reinterpret_cast<double*>(Bs);  // [4][128]
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    double v = jpart[i];
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (kq == 0) c_Jw[wc * 128 + (warp >> 2) * 64 + i * 8 + rq] = v;
  }
  __syncthreads();
  if (tid < 128) c_J[tid] = ((c_Jw[tid] + c_Jw[128 + tid]) + c_Jw[256 + tid]) + c_Jw[384 + tid];
  __syncthreads();

  // Phase 5: argmin per row, strict '<' so that the lowest k wins ties.
  if (tid < p.rt) {
    const int r = tid;
    const long long grow = c_row[r * p.ncp];
    if (grow >= 0) {
      int best = 0;
      double bj = c_J[r * p.ncp];
      for (int k = 1; k < p.n_cand; ++k) {
        const double j = c_J[r * p.ncp + k];
        if (j < bj) {
          bj = j;
          best = k;
        }
      }
      const int cr = r * p.ncp + best;
      const long long o = grow * p.ng + grp;
      p.sD[o] = c_s[cr];
      p.s_out[o] = (float)c_s[cr];
      p.z_out[o] = (int)c_z[cr];
      if (p.cand_out) p.cand_out[o] = (unsigned char)best;
    }
  }
}

// E[m][k] = W~[row(m)][k] - s (code - z): the quantization error of the group on
// the weights it saw (Proposition 3.1's W_B - Q_B).
__global__ void k_residual(const double* __restrict__ Wt, const unsigned char* __restrict__ codes,
                           const double* __restrict__ sD, const int* __restrict__ z,
                           double* __restrict__ E, RowMap rm, int M, int d, int seg, int ng) {
  const long long n = (long long)M * d;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(i / d), k = (int)(i % d);
    const long long r = rm.row(m);
    const long long so = r * ng + k / seg;
    const double q = (double)codes[r * d + k] - (double)z[so];
    E[i] = Wt[r * d + k] - sD[so] * q;
  }
}

// W~[rem] -= T E for the rows of every head not yet quantized (Propositions 3.1 / 3.2; Algorithm 1, update step).  CTA: 32
// rows x 128 columns of one head; thread: 8 rows x 2 columns, the group's rows 32 at a time from shared memory.  E is the
// group's residual W~ - s (code - z), formed where it is needed, or (HAVE_E, propagated error) a matrix.
// Bound: reading and writing W~ once.  As a residual launch and a product of the 128 x 128 engine it took, per step of
// one row in 8 heads x 4096 columns, 24 us, of 32 rows in 32 heads 115 us; now 13 us and 82 us.
// AHEAD: in short launches it is the loads that follow one another, so the matrices come ahead of the wait for the sweep and
// the rows to be updated beside the residual (256 rows of 256 columns in 32 steps, whole chain 1.70 -> 1.66 ms).  Held through
// the product, those rows take 128 registers instead of 74 (64 with HAVE_E), two CTAs an SM instead of three (four): where
// several waves of CTAs hide one another's loads anyway it loses (comp_ahead()).
template <bool HAVE_E, bool AHEAD>
__global__ void __launch_bounds__(256) k_compensate(double* Wt, const unsigned char* codes, const double* sD, const int* z,
                                                    const double* E, const double* T, int i0, int g, int dh,
                                                    long long t_head, int d, int seg, int ng) {
  __shared__ double Es[32][128], Ts[32][33];
  const int head = blockIdx.y, c0 = blockIdx.x * 128, q0 = blockIdx.z * 32;  // first of 32 remaining rows
  const int nrem = dh - i0 - g;
  const int tid = threadIdx.x, ct = (tid & 63) * 2, rt = tid >> 6;  // rows rt + 4 k
  const double* Th = T + head * t_head;
  auto matrices = [&](int e0, int ge) {
    for (int i = tid; i < 32 * ge; i += 256) {
      const int r = i / ge, c = i % ge;
      Ts[c][r] = (q0 + r < nrem) ? Th[(long long)(q0 + r) * g + e0 + c] : 0.0;
    }
  };
  if (AHEAD) matrices(0, min(32, g));  // from the call's beginning: ahead of the wait
  pdl_wait();
  auto to_update = [&](int r) { return reinterpret_cast<double2*>(Wt + ((long long)head * dh + i0 + g + r) * d + c0 + ct); };
  double2 old[8];  // the rows to be updated, on their way while the product is formed
  if (AHEAD) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int r = q0 + rt + 4 * k;
      old[k] = (r < nrem) ? *to_update(r) : make_double2(0.0, 0.0);
    }
  }
  double acc[8][2];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k][0] = acc[k][1] = 0.0;
  for (int e0 = 0; e0 < g; e0 += 32) {
    const int ge = min(32, g - e0);
    for (int i = tid; i < ge * 64; i += 256) {
      const int r = i >> 6, c = (i & 63) * 2;
      double2 v;
      if (HAVE_E) {
        v = *reinterpret_cast<const double2*>(E + ((long long)head * g + e0 + r) * d + c0 + c);
      } else {
        const long long row = (long long)head * dh + i0 + e0 + r, so = row * ng + (c0 + c) / seg;  // groups: multiples of 32
        v = *reinterpret_cast<const double2*>(Wt + row * d + c0 + c);
        const unsigned char* q = codes + row * d + c0 + c;  // the caller's pointer: of any alignment
        const double s = sD[so], zz = (double)z[so];
        v.x -= s * ((double)q[0] - zz);
        v.y -= s * ((double)q[1] - zz);
      }
      *reinterpret_cast<double2*>(&Es[r][c]) = v;
    }
    if (!AHEAD || e0 > 0) matrices(e0, ge);
    __syncthreads();
    for (int i = 0; i < ge; ++i) {
      const double2 e = *reinterpret_cast<const double2*>(&Es[i][ct]);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const double t = Ts[i][rt + 4 * k];
        acc[k][0] = fma(t, e.x, acc[k][0]);
        acc[k][1] = fma(t, e.y, acc[k][1]);
      }
    }
    __syncthreads();
  }
  pdl_trigger();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int r = q0 + rt + 4 * k;
    if (r >= nrem) continue;
    const double2 v = AHEAD ? old[k] : *to_update(r);
    *to_update(r) = make_double2(v.x - acc[k][0], v.y - acc[k][1]);
  }
}

// Which form of k_compensate: ahead without R for steps of up to 8 rows (4096 columns, 64 heads: 94 -> 88 us) and as long as CTAs
// times rows stay below 48 K (4096 columns, 16 heads: 16 rows 35.6 -> 33.1 us, 32 rows 47.8 -> 44.2, 64 rows 73.5 against 75.0 with
// it; 8192 columns, 64 heads, 64 rows 490 against 536); with R for what the SMs hold at once in that form (4096 columns, 4 heads, 64
// rows 18.7 -> 17.0; 16 heads 46.4 against 61.9, 8192 columns and 64 heads 317 against 494).
static bool comp_ahead(long long ctas, int g, bool with_r) { return with_r ? ctas <= 2 * 148 : g <= 8 || ctas * g <= 48 * 1024; }

// ---------------------------------------------------------------------------
// Coordinate descent on the scales (Proposition 3.3 / Algorithm 3), with the
// codes frozen.  Wbar = W_int - z.  State kept current through the pass:
//   Dm = (Q - W) H_in + W R      [rows][d]
// and, so that a scale step costs no product with H_in,
//   Yw[r][g2][:] = Wbar[r, G_g2] H_in[G_g2, :]      (one row of products per scale)
// A step on scale (j, g2) by delta adds delta * Yw[j][g2][:] to row j of Dm.
// Rows of a head are visited in order (Gauss-Seidel); per row:
//   k_cd_row_stats : n0[g]  = <Wbar[j,G_g], (H_out Dm)[j,G_g]>
//                    A[g2][g] = <Yw[j][g2][G_g], Wbar[j,G_g]>   (A[g][g] is the denominator's
//                                                                Wbar H_in[G,G] Wbar^T)
//   k_cd_row_update: the scalar chain over the row's groups,
//                    delta_g2 = -num_g2 / (A[g2][g2] H_out[j][j]),  num_g += H_out[j][j] delta_g2 A[g2][g],
//                    then Dm[j,:] += sum_g2 delta_g2 Yw[j][g2][:] and s += delta.
// ---------------------------------------------------------------------------
__global__ void k_cd_prep(const float* __restrict__ W, const unsigned char* __restrict__ codes,
                          const double* __restrict__ sD, const int* __restrict__ z,
                          double* __restrict__ Dq, float* __restrict__ Wb, long long rows, int d,
                          int seg, int ng) {
  const long long n = rows * d;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / d;
    const int k = (int)(i % d);
    const long long so = r * ng + k / seg;
    const double wb = (double)codes[i] - (double)z[so];
    if (Wb) Wb[i] = (float)wb;
    Dq[i] = sD[so] * wb - (double)W[i];
  }
}

struct CdP {
  double* Dm;           // [rows][d]            (rows of this batch)
  const void* Yw;       // [rows][ng][d], element type TY of the kernel
  const float* Wb;      // [rows][d]
  const float* Hout;    // [heads][dh][dh] of this batch, or nullptr
  double* sD;           // [rows][ng]
  double* n0;           // [lines][ng]
  double* Amat;         // [lines][ng][ng]
  int d, seg, ng, dh, j0, lines_per_head;  // lines_per_head = 1 (row j0 of each head) or dh
  int groups_per_cta;
  int a_in_smem;
};

// line = head * lines_per_head + l; its row inside the head is j0 + l.
// Partial sums are kept per 32-column chunk and added in chunk order, so the
// result does not depend on warp scheduling.
template <typename TY>
__global__ void __launch_bounds__(256) k_cd_row_stats(CdP p) {
  extern __shared__ double cd_sm[];  // part[chunks][ng + 1], then hrow[dh]
  const int tid = threadIdx.x, lane = tid & 31;
  const int line = blockIdx.y, head = line / p.lines_per_head, j = p.j0 + line % p.lines_per_head;
  const int d = p.d, seg = p.seg, ng = p.ng, dh = p.dh;
  const int g_first = blockIdx.x * p.groups_per_cta;
  const int g_count = min(p.groups_per_cta, ng - g_first);
  const int c_first = g_first * seg, c_count = g_count * seg;
  const int chunks_per_group = seg / 32;
  const int max_chunks = p.groups_per_cta * chunks_per_group;
  const long long row = (long long)head * dh + j;
  double* part = cd_sm;                           // [max_chunks][ng + 1]
  double* hrow = cd_sm + (size_t)max_chunks * (ng + 1);  // [dh]
  if (p.Hout)
    for (int i = tid; i < dh; i += blockDim.x) hrow[i] = (double)p.Hout[((long long)head * dh + j) * dh + i];
  __syncthreads();
  const double* Dh = p.Dm + (long long)head * dh * d;
  const TY* Yr = static_cast<const TY*>(p.Yw) + row * ng * d;
  const float* wbr = p.Wb + row * d;
  // every warp walks 32 consecutive columns at a time; they lie in one group
  for (int cb = (tid >> 5) * 32; cb < c_count; cb += (blockDim.x >> 5) * 32) {
    const int col = c_first + cb + lane;
    const int chunk = cb / 32;
    const int g = g_first + cb / seg;
    const double wb = (double)wbr[col];
    double gj;
    if (p.Hout) {
      gj = 0.0;
      for (int i = 0; i < dh; ++i) gj = fma(hrow[i], Dh[(long long)i * d + col], gj);
    } else {
      gj = Dh[(long long)j * d + col];
    }
    const double v = warp_sum(wb * gj);
    if (lane == 0) part[chunk * (ng + 1) + ng] = v;
    for (int g2 = 0; g2 <= g; ++g2) {
      const double a = warp_sum((double)Yr[(long long)g2 * d + col] * wb);
      if (lane == 0) part[chunk * (ng + 1) + g2] = a;
    }
  }
  __syncthreads();
  for (int i = tid; i < g_count * (ng + 1); i += blockDim.x) {
    const int gl = i / (ng + 1), g2 = i % (ng + 1), g = g_first + gl;
    if (g2 != ng && g2 > g) continue;
    double t = 0.0;
    for (int c = 0; c < chunks_per_group; ++c) t += part[(gl * chunks_per_group + c) * (ng + 1) + g2];
    if (g2 == ng)
      p.n0[(long long)line * ng + g] = t;
    else
      p.Amat[((long long)line * ng + g2) * ng + g] = t;
  }
}

template <typename TY>
__global__ void __launch_bounds__(256) k_cd_row_update(CdP p) {
  extern __shared__ double cd_sm[];  // num[ng], delta[ng], then A[ng][ng] if it fits
  const int tid = threadIdx.x, lane = tid & 31;
  const int line = blockIdx.y, head = line / p.lines_per_head, j = p.j0 + line % p.lines_per_head;
  const int d = p.d, seg = p.seg, ng = p.ng, dh = p.dh;
  const long long row = (long long)head * dh + j;
  double* num = cd_sm;
  double* delta = cd_sm + ng;
  const double hjj = p.Hout ? (double)p.Hout[((long long)head * dh + j) * dh + j] : 1.0;
  const double* A = p.Amat + (long long)line * ng * ng;
  for (int g = tid; g < ng; g += blockDim.x) num[g] = p.n0[(long long)line * ng + g];
  if (p.a_in_smem) {
    double* As = cd_sm + 2 * ng;
    for (int i = tid; i < ng * ng; i += blockDim.x) {
      const int g2 = i / ng, g = i % ng;
      As[i] = (g >= g2) ? A[i] : 0.0;
    }
    A = As;
  }
  __syncthreads();
  if (tid < 32) {
    for (int g2 = 0; g2 < ng; ++g2) {
      const double den = A[(long long)g2 * ng + g2] * hjj;
      const double dl = (den == 0.0) ? 0.0 : -num[g2] / den;
      if (lane == 0) delta[g2] = dl;
      for (int g = g2 + 1 + lane; g < ng; g += 32) num[g] = fma(hjj * dl, A[(long long)g2 * ng + g], num[g]);
      __syncwarp();
    }
  }
  __syncthreads();
  const int g_first = blockIdx.x * p.groups_per_cta;
  const int g_count = min(p.groups_per_cta, ng - g_first);
  const int c_first = g_first * seg, c_count = g_count * seg;
  const TY* Yr = static_cast<const TY*>(p.Yw) + row * ng * d;
  double* dm = p.Dm + row * d;
  for (int c = tid; c < c_count; c += blockDim.x) {
    const int col = c_first + c;
    double acc = dm[col];
    for (int g2 = 0; g2 < ng; ++g2) acc = fma(delta[g2], (double)Yr[(long long)g2 * d + col], acc);
    dm[col] = acc;
  }
  if (blockIdx.x == 0)
    for (int g = tid; g < ng; g += blockDim.x) p.sD[row * ng + g] += delta[g];
}

// ---------------------------------------------------------------------------
// One Gauss-Seidel pass of Algorithm 3 over ALL rows of one head in a single
// launch.  A thread-block cluster of C CTAs owns a head; CTA r owns the column
// groups r ng/C .. (r+1) ng/C - 1 (whole groups, so every sum over a group is
// local to one CTA).  The cluster walks the head's rows in order and works on
//   G = H_out Dm    (rows of the head, formed once by a batched GEMM),
// whose row j is what the numerator of Proposition 3.3 needs.  A step on the
// scales of row i adds u_i = sum_g2 delta_g2 Yw[i][g2][:] to row i of Dm, hence
// H_out[j][i] u_i to every row j of G.  Those rank-1 terms are applied lazily:
// rows of the current block of 16 read the u_i of their block on the fly, and
// when a block is finished its 16 vectors are folded into the rows of G that
// are still to come.  Per row, each CTA forms n0[g] and A[.][g] for its groups,
// stores them into the shared memory of every CTA of the cluster (distributed
// shared memory, two buffers by row parity), and after one cluster barrier every
// CTA runs the short scalar chain itself.  The u_i are kept (Uacc) so that Dm
// can be refreshed after the pass.  All sums have a fixed order.
// ---------------------------------------------------------------------------
enum { CDH_THREADS = 512, CDH_BLOCK = 16 };
struct CdHeadP {
  double* G;           // [heads*dh][d]   H_out Dm, updated in place
  double* Uacc;        // [heads*dh][d]   out: the rank-1 vectors u_i
  const void* Yw;      // [heads*dh][ng][d], element type TY of the kernel
  const float* Wb;     // [heads*dh][d]
  const float* Hout;   // [heads][dh][dh]
  double* sD;          // [heads*dh][ng]
  int d, seg, ng, dh;
  int csize;           // CTAs per cluster (divides ng)
  int uw;              // columns per work unit (a divisor of seg, multiple of 32, at most 128)
};

template <typename TY>
__global__ void __launch_bounds__(CDH_THREADS, 1) k_cd_head(CdHeadP p) {
  extern __shared__ double cdh_sm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster.block_rank();
  const int head = blockIdx.x / p.csize;
  const int d = p.d, seg = p.seg, ng = p.ng, dh = p.dh, uw = p.uw;
  const int gpc = ng / p.csize;                 // groups of this CTA
  const int g_lo = rank * gpc;
  const int upg = seg / uw;                     // units per group
  const int n_units = gpc * upg;                // units of this CTA
  const int c_lo = g_lo * seg, c_cnt = gpc * seg;  // its columns
  double* part = cdh_sm;                                   // [n_units][ng + 1]
  double* Am = part + (size_t)n_units * (ng + 1);          // [2][ng][ng]  (entries g2 <= g)
  double* num = Am + (size_t)2 * ng * ng;                  // [2][ng]
  double* delta = num + 2 * ng;                            // [ng]
  const long long row0 = (long long)head * dh;
  const float* Ho = p.Hout + (long long)head * dh * dh;

  for (int j = 0; j < dh; ++j) {
    const long long row = row0 + j;
    const int buf = j & 1;
    const int blk0 = (j / CDH_BLOCK) * CDH_BLOCK;
    const double hjj = (double)Ho[(long long)j * dh + j];
    const TY* Yr = static_cast<const TY*>(p.Yw) + row * ng * d;
    const float* wbr = p.Wb + row * d;
    const double* Gr = p.G + row * d;
    const float* hrow = Ho + (long long)j * dh;
    // ---- statistics of the row for this CTA's groups: n0[g] and A[g2][g], g2 <= g ----
    for (int u = warp; u < n_units; u += CDH_THREADS / 32) {
      const int g = g_lo + u / upg;
      const int cbase = g * seg + (u % upg) * uw;
      double wb[4], gv[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int col = cbase + lane + 32 * c;
        const bool on = lane + 32 * c < uw;
        wb[c] = on ? (double)wbr[col] : 0.0;
        gv[c] = on ? Gr[col] : 0.0;
      }
      for (int i = blk0; i < j; ++i) {
        const double h = (double)hrow[i];
        const double* ui = p.Uacc + (row0 + i) * d + cbase + lane;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (lane + 32 * c < uw) gv[c] = fma(h, ui[32 * c], gv[c]);
      }
      double v = 0.0;
#pragma unroll
      for (int c = 0; c < 4; ++c) v = fma(wb[c], gv[c], v);
      v = warp_sum(v);
      if (lane == 0) part[(size_t)u * (ng + 1) + ng] = v;
      const TY* yb = Yr + cbase + lane;
      int g2 = 0;
      for (; g2 + 4 <= g + 1; g2 += 4) {
        double a4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (lane + 32 * c < uw) a4[t] = fma((double)yb[(long long)(g2 + t) * d + 32 * c], wb[c], a4[t]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int t = 0; t < 4; ++t) a4[t] += __shfl_xor_sync(0xffffffffu, a4[t], o);
        if (lane < 4) part[(size_t)u * (ng + 1) + g2 + lane] = (lane == 0) ? a4[0] : (lane == 1) ? a4[1] : (lane == 2) ? a4[2] : a4[3];
      }
      for (; g2 <= g; ++g2) {
        double a = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (lane + 32 * c < uw) a = fma((double)yb[(long long)g2 * d + 32 * c], wb[c], a);
        a = warp_sum(a);
        if (lane == 0) part[(size_t)u * (ng + 1) + g2] = a;
      }
    }
    __syncthreads();
    // ---- reduce the units of each group in order and publish to every CTA of the cluster ----
    for (int idx = tid; idx < gpc * (ng + 1); idx += CDH_THREADS) {
      const int gl = idx / (ng + 1), g2 = idx % (ng + 1), g = g_lo + gl;
      if (g2 != ng && g2 > g) continue;
      double t = 0.0;
      for (int c = 0; c < upg; ++c) t += part[(size_t)(gl * upg + c) * (ng + 1) + g2];
      for (int r = 0; r < p.csize; ++r) {
        if (g2 == ng)
          cluster.map_shared_rank(num, r)[buf * ng + g] = t;
        else
          cluster.map_shared_rank(Am, r)[((size_t)buf * ng + g2) * ng + g] = t;
      }
    }
    cluster.sync();
    // ---- the scalar chain over the row's groups (every CTA runs it) ----
    if (warp == 0) {
      double* nm = num + buf * ng;
      const double* A = Am + (size_t)buf * ng * ng;
      for (int g2 = 0; g2 < ng; ++g2) {
        const double den = A[(size_t)g2 * ng + g2] * hjj;
        const double dl = (den == 0.0) ? 0.0 : -nm[g2] / den;
        if (lane == 0) delta[g2] = dl;
        for (int g = g2 + 1 + lane; g < ng; g += 32) nm[g] = fma(hjj * dl, A[(size_t)g2 * ng + g], nm[g]);
        __syncwarp();
      }
    }
    __syncthreads();
    // ---- u_j on this CTA's columns, and the scales ----
    double* ur = p.Uacc + row * d;
    for (int c0 = tid; c0 < c_cnt; c0 += 4 * CDH_THREADS) {
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      for (int g2 = 0; g2 < ng; ++g2) {
        const double dl = delta[g2];
        const TY* y = Yr + (long long)g2 * d + c_lo + c0;
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (c0 + t * CDH_THREADS < c_cnt) acc[t] = fma(dl, (double)y[t * CDH_THREADS], acc[t]);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (c0 + t * CDH_THREADS < c_cnt) ur[c_lo + c0 + t * CDH_THREADS] = acc[t];
    }
    if (rank == 0)
      for (int g = tid; g < ng; g += CDH_THREADS) p.sD[row * ng + g] += delta[g];
    __syncthreads();
    // ---- end of a block: fold its vectors into the rows of G still to come ----
    if ((j + 1) % CDH_BLOCK == 0 && j + 1 < dh) {
      for (int c = tid; c < c_cnt; c += CDH_THREADS) {
        const int col = c_lo + c;
        double u16[CDH_BLOCK];
#pragma unroll
        for (int i = 0; i < CDH_BLOCK; ++i) u16[i] = p.Uacc[(row0 + blk0 + i) * d + col];
        for (int jj = j + 1; jj < dh; ++jj) {
          const float* hr = Ho + (long long)jj * dh + blk0;
          double gvv = p.G[(row0 + jj) * d + col];
#pragma unroll
          for (int i = 0; i < CDH_BLOCK; ++i) gvv = fma((double)hr[i], u16[i], gvv);
          p.G[(row0 + jj) * d + col] = gvv;
        }
      }
      __syncthreads();
    }
  }
  cluster.sync();  // no CTA may exit while another can still store into its shared memory
}

// ---------------------------------------------------------------------------
// Column-parallel form of the same pass, for up to 32 groups and at most 1024
// columns per CTA.  The quadratic forms A[g2][g] = Wbar_g2^T H_in[g2, g] Wbar_g
// of a row depend on the integers only, so k_cd_amat forms them for every row
// up front, in parallel, and with them the row's whole chain over its groups as one
// triangular matrix: delta = -M num / hjj.  In the walk, thread t owns columns 2t, 2t+1 of its
// CTA for the whole pass: the u_i of the current block of 16 rows stay in its
// registers, the lazily corrected row of G is formed there, and one row costs
// four block barriers, one cluster barrier and a product with M by warp 0 of every CTA.
// What the next row needs (its row of G, Wbar, M and H_out) is fetched while the current row is
// processed; its slice of Yw (float: up to 128 KB) is copied into shared memory meanwhile.
// A row of 32 heads with 32 groups of 128 takes 8 us (18 k clocks: numerators and their exchange 5 k, the product with
// M 1.5, u 2.7, its float -> double conversions most of it, the fold at a block's end 4.2), of which 2.5 are the HBM time
// of Yw.  It took 11 when the chain ran group by group (2.7 k clocks), Yw came from L2 (6.7 k) and the fold read
// H_out entry by entry (5.4 k).  4096 rows: 1.40 -> 1.02 ms, k_cd_chain 0.03.
// ---------------------------------------------------------------------------
enum { CDC_THREADS = 512, CDC_MAXG = 32, CDC_FOLD = 64 };

template <typename TY>
__global__ void __launch_bounds__(256) k_cd_amat(const void* __restrict__ Yw_, const float* __restrict__ Wb,
                                                 double* __restrict__ Amat, int d, int seg, int ng) {
  extern __shared__ float amat_wb[];
  const long long row = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int c = tid; c < d; c += 256) amat_wb[c] = Wb[row * d + c];
  __syncthreads();
  const TY* Yr = static_cast<const TY*>(Yw_) + row * ng * d;
  double* A = Amat + row * ng * ng;
  for (int g2 = 0; g2 < ng; ++g2)
    for (int g = g2 + warp; g < ng; g += 8) {
      const TY* y = Yr + (long long)g2 * d + g * seg;
      const float* w = amat_wb + g * seg;
      double v = 0.0;
      for (int c = lane; c < seg; c += 32) v = fma((double)y[c], (double)w[c], v);
      v = warp_sum(v);
      if (lane == 0) A[g2 * ng + g] = v;
    }
}

// In place, A[g2][g] -> M[g2][g], g2 <= g: with r_g = 1 / A[g][g] (0 for a skipped coordinate), the group-by-group rule
// n_g -= sum_(g2 < g) A[g2][g] r_g2 n_g2 as a product, n = L num, and M[g2][g] = r_g L[g][g2].  A warp per row, a lane
// per column of L in registers.  (At the end of k_cd_amat it would cost that kernel its occupancy: 844 us instead of 308.)
__global__ void __launch_bounds__(128) k_cd_chain(double* __restrict__ Amat, long long rows, int ng) {
  __shared__ double sA[4][CDC_MAXG][CDC_MAXG];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long row = (long long)blockIdx.x * 4 + warp;
  if (row >= rows) return;
  double* A = Amat + row * ng * ng;
  double(*As)[CDC_MAXG] = sA[warp];
  for (int g2 = 0; g2 < CDC_MAXG; ++g2) As[g2][lane] = (g2 < ng && lane < ng && g2 <= lane) ? A[g2 * ng + lane] : 0.0;
  __syncwarp();
  const double r_mine = (As[lane][lane] == 0.0) ? 0.0 : 1.0 / As[lane][lane];
  double L[CDC_MAXG];
#pragma unroll
  for (int g = 0; g < CDC_MAXG; ++g) {
    double v[4] = {(g == lane) ? 1.0 : 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int g2 = 0; g2 < g; ++g2) v[g2 & 3] = fma(-As[g2][g], L[g2], v[g2 & 3]);
    L[g] = __shfl_sync(0xffffffffu, r_mine, g) * ((v[0] + v[1]) + (v[2] + v[3]));
    if (lane < ng && g < ng) A[lane * ng + g] = L[g];
  }
}

__device__ __forceinline__ double2 load_pair(const float* q) {
  const float2 v = *reinterpret_cast<const float2*>(q);
  return make_double2((double)v.x, (double)v.y);
}
__device__ __forceinline__ double2 load_pair(const double* q) { return *reinterpret_cast<const double2*>(q); }
struct CdColP {
  double* G;           // [heads*dh][d]   H_out Dm, rows still to come updated in place at block ends
  double* Uacc;        // [heads*dh][d]   out: the rank-1 vectors u_i
  const void* Yw;      // [heads*dh][ng][d], element type TY of the kernel
  const float* Wb;     // [heads*dh][d]
  const float* Hout;   // [heads][dh][dh]
  const double* Mmat;  // [heads*dh][ng][ng], of k_cd_chain
  double* sD;          // [heads*dh][ng]
  int d, seg, ng, dh;
  int csize;           // CTAs per cluster (divides ng)
};

__device__ int g_cd_error = 0;
int cd_error_read_clear() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_cd_error, sizeof(int)) != cudaSuccess) return -1;
  if (v) {
    int z = 0;
    cudaMemcpyToSymbol(g_cd_error, &z, sizeof(int));
  }
  return v;
}

template <typename TY>
__global__ void __launch_bounds__(CDC_THREADS, 1) k_cd_head_cols(CdColP p) {
  __shared__ double part[CDC_THREADS];
  __shared__ double Am[2][CDC_MAXG * CDC_MAXG];
  __shared__ double num[2][CDC_MAXG];
  __shared__ double delta[CDC_MAXG];
  __shared__ double hs[CDH_BLOCK][2 * CDH_BLOCK];  // the block's rows of H_out: columns of the block behind as many zeros
  __shared__ __align__(16) double hf[CDC_FOLD][CDH_BLOCK];  // columns of H_out for the fold
  __shared__ unsigned long long slab_bar;
  __shared__ int abort_flag;
  extern __shared__ __align__(128) unsigned char cdc_slab[];  // float: this CTA's columns of the row's Yw, [ng][c_cnt]
  constexpr bool STAGED = sizeof(TY) == 4;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster.block_rank();
  const int head = blockIdx.x / p.csize;
  const int d = p.d, seg = p.seg, ng = p.ng, dh = p.dh;
  const int gpc = ng / p.csize, g_lo = rank * gpc;
  const int c_lo = g_lo * seg, c_cnt = gpc * seg;
  const int c0 = 2 * tid;
  const bool on = c0 < c_cnt;
  const int col = c_lo + c0;
  const long long row0 = (long long)head * dh;
  const float* Ho = p.Hout + (long long)head * dh * dh;
  const TY* Yw = static_cast<const TY*>(p.Yw);
  const int a_cnt = ng * ng;
  const int half = seg / 2;  // partial sums per group
  const int slab_lines = (c_cnt * (int)sizeof(TY) + 127) / 128;
  const uint32_t sbar = smem_u32(&slab_bar);
  if (tid == 0) {
    mbar_init(sbar, 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  auto fetch_slab = [&](long long row) {  // one warp, a group per lane
    if (lane == 0) mbar_expect_tx(sbar, (uint32_t)(ng * c_cnt) * 4u);
    __syncwarp();
    if (lane < ng)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       smem_u32(cdc_slab) + (uint32_t)(lane * c_cnt) * 4u),
                   "l"(Yw + (row * ng + lane) * d + c_lo), "r"((uint32_t)c_cnt * 4u), "r"(sbar)
                   : "memory");
  };

  // what row 0 needs
  double2 gn = make_double2(0.0, 0.0);
  float2 wn = make_float2(0.0f, 0.0f);
  double an0 = 0.0, an1 = 0.0;
  if (on) {
    gn = *reinterpret_cast<const double2*>(p.G + row0 * d + col);
    wn = *reinterpret_cast<const float2*>(p.Wb + row0 * d + col);
  }
  if (tid < a_cnt) an0 = p.Mmat[row0 * a_cnt + tid];
  if (tid + CDC_THREADS < a_cnt) an1 = p.Mmat[row0 * a_cnt + tid + CDC_THREADS];
  double sdn = (rank == 0 && tid < ng) ? p.sD[row0 * ng + tid] : 0.0;  // the row's scales, fetched one row ahead
  // the vectors move down one slot per row, so slot k of row j holds u of row j - 16 + k (zero while that row lies
  // before the block) and meets hs[j % 16][j % 16 + k]
  auto fetch_h = [&](int blk) {
    const int r = tid >> 5, c = (tid & 31) - CDH_BLOCK;
    if (r < CDH_BLOCK) hs[r][tid & 31] = (c >= 0 && blk + r < dh && blk + c < dh) ? (double)Ho[(long long)(blk + r) * dh + blk + c] : 0.0;
  };
  fetch_h(0);
  __syncthreads();
  if (STAGED && warp == CDC_THREADS / 32 - 1) fetch_slab(row0);

  double2 ureg[CDH_BLOCK];
#pragma unroll
  for (int i = 0; i < CDH_BLOCK; ++i) ureg[i] = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int j = 0; j < dh; ++j) {
    const long long row = row0 + j;
    const int buf = j & 1, jl = j % CDH_BLOCK;
    double2 gv = gn;
    const float2 w = wn;
    const double sd_cur = sdn;
    if (tid < a_cnt) Am[buf][tid] = an0;
    if (tid + CDC_THREADS < a_cnt) Am[buf][tid + CDC_THREADS] = an1;
    // ---- fetch for row j + 1 ----
    if (j + 1 < dh) {
      const long long rn = row + 1;
      if (on) {
        gn = *reinterpret_cast<const double2*>(p.G + rn * d + col);
        wn = *reinterpret_cast<const float2*>(p.Wb + rn * d + col);
      }
      if (tid < a_cnt) an0 = p.Mmat[rn * a_cnt + tid];
      if (tid + CDC_THREADS < a_cnt) an1 = p.Mmat[rn * a_cnt + tid + CDC_THREADS];
      if (rank == 0 && tid < ng) sdn = p.sD[rn * ng + tid];
      if (!STAGED)
        for (int idx = tid; idx < slab_lines * ng; idx += CDC_THREADS) {
          const int g2 = idx / slab_lines, l = idx % slab_lines;
          const char* ptr = reinterpret_cast<const char*>(Yw + (rn * ng + (long long)g2) * d + c_lo) + l * 128;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr));
        }
    }
    // ---- numerators of this CTA's groups: Wbar . (G + pending rank-1 terms of the block) ----
#pragma unroll
    for (int i = 0; i < CDH_BLOCK; ++i) {
      const double h = hs[jl][jl + i];
      gv.x = fma(h, ureg[i].x, gv.x);
      gv.y = fma(h, ureg[i].y, gv.y);
    }
    part[tid] = on ? fma((double)w.y, gv.y, (double)w.x * gv.x) : 0.0;
    const double hjj = hs[jl][jl + CDH_BLOCK];
    __syncthreads();
    for (int gl = warp; gl < gpc; gl += CDC_THREADS / 32) {
      double v = 0.0;
      for (int k = lane; k < half; k += 32) v += part[gl * half + k];
      v = warp_sum(v);
      if (lane == 0)
        for (int r = 0; r < p.csize; ++r) cluster.map_shared_rank(&num[0][0], r)[buf * CDC_MAXG + g_lo + gl] = v;
    }
    cluster.sync();
    // ---- the row's groups: delta = -M num / hjj, lane g (every CTA) ----
    if (warp == 0) {
      const bool in = lane < ng;
      double a4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int g2 = 0; g2 < CDC_MAXG; ++g2) {  // selects, not branches: those keep the loads of one step behind another's
        const double t = fma(Am[buf][g2 * ng + lane], num[buf][g2], a4[g2 & 3]);
        a4[g2 & 3] = (g2 <= lane) ? t : a4[g2 & 3];
      }
      const double mine = (hjj == 0.0) ? 0.0 : -((a4[0] + a4[1]) + (a4[2] + a4[3])) / hjj;
      if (in) {
        delta[lane] = mine;
        if (rank == 0) p.sD[row * ng + lane] = sd_cur + mine;
      }
    }
    __syncthreads();
    if (STAGED) mbar_wait(sbar, (uint32_t)buf, &abort_flag, &g_cd_error);
    // ---- u_j on this thread's columns ----
    double2 u = make_double2(0.0, 0.0);
    if (on) {
      const TY* y = STAGED ? reinterpret_cast<const TY*>(cdc_slab) + c0 : Yw + row * ng * d + col;
      const long long ld = STAGED ? c_cnt : d;
#pragma unroll 8
      for (int g2 = 0; g2 < ng; ++g2) {
        const double dl = delta[g2];
        const double2 yv = load_pair(y + g2 * ld);
        u.x = fma(dl, yv.x, u.x);
        u.y = fma(dl, yv.y, u.y);
      }
      *reinterpret_cast<double2*>(p.Uacc + row * d + col) = u;
    }
    if (STAGED && j + 1 < dh) {
      __syncthreads();  // the slice is read: the next row's takes its place
      if (warp == CDC_THREADS / 32 - 1) fetch_slab(row + 1);
    }
#pragma unroll
    for (int i = 0; i + 1 < CDH_BLOCK; ++i) ureg[i] = ureg[i + 1];
    ureg[CDH_BLOCK - 1] = u;
    // ---- end of a block: fold its vectors into the rows of G still to come ----
    if ((j + 1) % CDH_BLOCK == 0 && j + 1 < dh) {
      const int blk0 = j + 1 - CDH_BLOCK;
      for (int jb = j + 1; jb < dh; jb += CDC_FOLD) {
        const int n = min((int)CDC_FOLD, dh - jb);
        __syncthreads();
        for (int i = tid; i < n * CDH_BLOCK; i += CDC_THREADS)
          hf[i / CDH_BLOCK][i % CDH_BLOCK] = (double)Ho[(long long)(jb + i / CDH_BLOCK) * dh + blk0 + i % CDH_BLOCK];
        __syncthreads();
        if (on) {
          for (int jj = 0; jj < n; jj += 4) {  // four rows of G on their way at a time
            double2* gp = reinterpret_cast<double2*>(p.G + (row0 + jb + jj) * d + col);
            double2 g[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (jj + q < n) g[q] = gp[(long long)q * d / 2];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (jj + q < n) {
#pragma unroll
                for (int i = 0; i < CDH_BLOCK; i += 2) {
                  const double2 h = *reinterpret_cast<const double2*>(&hf[jj + q][i]);
                  g[q].x = fma(h.x, ureg[i].x, g[q].x);
                  g[q].y = fma(h.x, ureg[i].y, g[q].y);
                  g[q].x = fma(h.y, ureg[i + 1].x, g[q].x);
                  g[q].y = fma(h.y, ureg[i + 1].y, g[q].y);
                }
                gp[(long long)q * d / 2] = g[q];
                if (jb + jj + q == j + 1) gn = g[q];
              }
          }
        }
      }
      fetch_h(j + 1);  // (the first barrier of the fold came after the block's last use)
      __syncthreads();
#pragma unroll
      for (int i = 0; i < CDH_BLOCK; ++i) ureg[i] = make_double2(0.0, 0.0);
    }
  }
  cluster.sync();  // no CTA may exit while another can still store into its shared memory
}

// Dm += Uacc (the effect of one pass on (Q - W) H_in + W R)
__global__ void k_axpy(double* __restrict__ y, const double* __restrict__ x, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] += x[i];
}

// Q = s (W_int - z) in float, and the scales in float (Algorithm 1, final step).
__global__ void k_dequant(const unsigned char* __restrict__ codes, const double* __restrict__ sD,
                          const int* __restrict__ z, float* __restrict__ What,
                          float* __restrict__ s_out, long long rows, int d, int seg, int ng) {
  const long long n = rows * d;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const long long r = i / d;
    const int k = (int)(i % d);
    const long long so = r * ng + k / seg;
    if (What) What[i] = (float)(sD[so] * ((double)codes[i] - (double)z[so]));
    if (k % seg == 0) s_out[so] = (float)sD[so];
  }
}

// loss[h] = sum over the head's rows of <Z[r,:], dW[r,:]> (Z already multiplied by H_out when there
// is one: tr(H_out Z dW^T) = sum of (H_out Z) .* dW), in two steps with a fixed order: one partial
// sum per block of 32 rows, then the partial sums of a head.
__global__ void __launch_bounds__(256) k_loss_identity_partial(const double* __restrict__ Z,
                                                               const double* __restrict__ Dq,
                                                               double* __restrict__ partial,
                                                               long long rows_per_head, int d, int chunks) {
  __shared__ double part[8];
  const int h = blockIdx.y, c = blockIdx.x;
  const long long r0 = (long long)c * 32, r1 = (r0 + 32 < rows_per_head) ? r0 + 32 : rows_per_head;
  const long long base = ((long long)h * rows_per_head + r0) * d, n = (r1 - r0) * d;
  double acc = 0.0;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) acc = fma(Z[base + i], Dq[base + i], acc);
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += part[i];
    partial[(long long)h * chunks + c] = t;
  }
}
__global__ void k_loss_identity_final(const double* __restrict__ partial, double* __restrict__ loss, int chunks) {
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int c = 0; c < chunks; ++c) t += partial[(long long)blockIdx.x * chunks + c];
    loss[blockIdx.x] = t;
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct Plan {
  int d_out, d, H, dh, n_hin, bits, seg, ng, g, S, maxq, n_cand, ncp, rt, cd_iters;
  bool adaptive, dynamic, cd, with_r, with_loss, has_hout;
  double *dynErr, *dynArr;  // [Mmax][seg] errors / arrival values of the current column group (dynamic grid)
  int Mmax;
  size_t e_doubles;   // of E
  long long cd_rows;  // rows per coordinate-descent batch
  // workspace
  double *Wt, *Wk, *W0c, *E, *sD, *T, *Dq, *Dm, *Yw, *n0, *Amat, *G2;
  double* gram;  // scale refinement as a triangular solve: the heads' matrices
  SweepScratch sweep;
  bool grid_digits;  // the search on the integer tensor cores, with
  GridDigits gd;
  I8Mat Cdig, Wdig;                // digits of C (all steps) and of the step's W0 (propagated error, one shared H_in)
  unsigned long long *c_max, *w_max;
  float* Wb;
  __nv_bfloat16 *WbT, *Hp;  // tensor-core path of the blockwise product
  bool yw_tensor;    // and with it (Q - W) H_in through the split-bf16 product
  double* WR;        // W R, kept from the refinement for the loss (one shared H_in, split products)
  bool loss_tensor;  // the loss's own dW H_in (no scale refinement) through it too
  int loss_heads;    // with one H_in per head: heads per launch of that product (their pieces of H_in fit 2 GiB)
  size_t ws_total;
};

static int pow2_ceil(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

static tb_status make_plan(const tb_layer_desc* D, bool has_hout, bool with_r, bool with_loss,
                           void* ws, Plan* pl) {
  if (!D) return TB_ERR_INVALID_ARG;
  if (D->d_out <= 0 || D->d_in <= 0 || D->n_heads <= 0 || D->d_head <= 0) return TB_ERR_INVALID_ARG;
  if ((long long)D->n_heads * D->d_head != D->d_out) return TB_ERR_INVALID_ARG;
  if (D->d_in % 128) return TB_ERR_UNSUPPORTED;
  if (D->n_hin != 1 && D->n_hin != D->n_heads) return TB_ERR_INVALID_ARG;
  if (D->bits < 2 || D->bits > 8) return TB_ERR_INVALID_ARG;
  if (D->quant_group < 0) return TB_ERR_INVALID_ARG;
  if (D->quant_group > 0 && (D->d_in % D->quant_group)) return TB_ERR_INVALID_ARG;
  if (D->quant_group > 0 && (D->quant_group % 32)) return TB_ERR_UNSUPPORTED;
  if (D->out_block < 1 || D->out_block > D->d_head || (D->d_head % D->out_block)) return TB_ERR_INVALID_ARG;
  if (D->n_cand < 1 || D->n_cand > 32) return TB_ERR_INVALID_ARG;
  if (D->cd_iters < 0) return TB_ERR_INVALID_ARG;
  Plan& p = *pl;
  p.d_out = D->d_out;
  p.d = D->d_in;
  p.H = D->n_heads;
  p.dh = D->d_head;
  p.n_hin = D->n_hin;
  p.bits = D->bits;
  p.seg = D->quant_group > 0 ? D->quant_group : D->d_in;
  p.ng = p.d / p.seg;
  p.has_hout = has_hout;
  p.g = has_hout ? D->out_block : D->d_head;  // H_out = I: all rows of a head at once
  p.S = p.dh / p.g;
  p.maxq = (1 << D->bits) - 1;
  p.n_cand = D->n_cand;
  p.ncp = pow2_ceil(D->n_cand);
  p.rt = 128 / p.ncp;
  p.cd_iters = D->cd_iters;
  // dynamic grid: with one group per row it IS the adaptive grid (the group arrives unchanged)
  p.dynamic = (D->flags & TB_F_DYNAMIC_GRID) != 0 && p.ng > 1;
  p.adaptive = (D->flags & TB_F_ADAPTIVE_GRID) != 0 || ((D->flags & TB_F_DYNAMIC_GRID) != 0 && !p.dynamic);
  if (p.dynamic && p.seg > 128) return TB_ERR_UNSUPPORTED;
  p.cd = (D->flags & TB_F_CD_REFINE) != 0 && D->cd_iters > 0;
  p.with_r = with_r;
  p.with_loss = with_loss;
  p.Mmax = p.H * p.g;
  if (p.ng > 1024) return TB_ERR_UNSUPPORTED;

  Bump b(ws);
  const size_t dd = (size_t)p.d;
  p.Wt = b.take<double>((size_t)p.d_out * dd);
  p.Wk = b.take<double>((size_t)p.Mmax * dd);
  // E is also the scratch of the search of wide groups, which needs a little more than d_in doubles a row with 17 and
  // more candidates: a step's rows go through in one chunk
  p.e_doubles = (size_t)p.Mmax * dd;
  if (p.seg > 128) {
    const size_t search = (size_t)p.Mmax * grid_wide_row_doubles(p.d, p.ng, p.ncp);
    if (search > p.e_doubles) p.e_doubles = search;
  }
  p.E = b.take<double>(p.e_doubles);
  p.W0c = with_r ? b.take<double>((size_t)p.Mmax * dd) : nullptr;
  p.sweep = SweepScratch{};
  if (!p.dynamic) {
    const int units = (p.n_hin == 1) ? 1 : p.H;
    sweep_scratch(b, p.Mmax, p.d, with_r, sweep_wants_i8(p.d, units, p.Mmax / units), &p.sweep);
    p.sweep.work = p.Wk;
  }
  p.Cdig = p.Wdig = I8Mat{nullptr, 0, 0};
  p.c_max = p.w_max = nullptr;
  if (with_r && has_hout && p.S > 1 && p.n_hin == 1 && p.d <= 16384) {
    p.Cdig.row_blocks = p.d / I8_RB;  // d is a multiple of 128
    p.Wdig.row_blocks = (p.Mmax + I8_RB - 1) / I8_RB;
    p.Cdig.k_blocks = p.Wdig.k_blocks = p.d / I8_KB;
    p.Cdig.data = b.take<unsigned char>(i8_bytes(p.Cdig.row_blocks, p.Cdig.k_blocks));
    p.Wdig.data = b.take<unsigned char>(i8_bytes(p.Wdig.row_blocks, p.Wdig.k_blocks));
    p.c_max = b.take<unsigned long long>(dd);
    p.w_max = b.take<unsigned long long>((size_t)p.Mmax);
  }
  {  // the search of a fixed grid takes all rows at once, the adaptive one a step's
    const int units = (p.n_hin == 1) ? 1 : p.H, rows = p.adaptive ? p.Mmax : p.d_out;
    p.grid_digits = !p.dynamic && grid_wants_digits(rows, units, p.d, p.seg, p.ncp);
    if (p.grid_digits) grid_digits_scratch(b, rows, units, p.d, p.seg, p.ncp, p.bits, &p.gd);
  }
  p.sD = b.take<double>((size_t)p.d_out * p.ng);
  p.T = (has_hout && p.S > 1) ? b.take<double>((size_t)p.H * p.S * p.dh * p.g) : nullptr;
  p.dynErr = p.dynamic ? b.take<double>((size_t)p.Mmax * p.seg) : nullptr;
  p.dynArr = (p.dynamic && with_r) ? b.take<double>((size_t)p.Mmax * p.seg) : nullptr;
  p.WR = p.Dq = p.Dm = p.Yw = p.n0 = p.Amat = p.G2 = p.gram = nullptr;
  p.Wb = nullptr;
  p.WbT = p.Hp = nullptr;
  p.yw_tensor = false;
  p.cd_rows = 0;
  if (p.cd || with_loss) {
    p.Dq = b.take<double>((size_t)p.d_out * dd);
    p.Dm = b.take<double>((size_t)p.d_out * dd);
  }
  if (p.cd) {
    p.Wb = b.take<float>((size_t)p.d_out * dd);
    // batch of rows whose Yw fits 4 GiB: whole heads when rows of a head are coupled
    const size_t per_row = (size_t)p.ng * dd * sizeof(double);
    const size_t budget = (size_t)4 << 30;
    long long unit_rows = (has_hout || p.n_hin > 1) ? p.dh : 1;
    long long units = (long long)(budget / (per_row * unit_rows));
    if (units < 1) units = 1;
    long long rows = units * unit_rows;
    if (rows > p.d_out) rows = p.d_out;
    if (!(has_hout || p.n_hin > 1) && rows > 128) rows = (rows / 128) * 128;
    p.cd_rows = rows;
    p.Yw = b.take<double>((size_t)rows * p.ng * dd);
    // Products on the tensor cores, the blockwise one with a float result: one shared H_in, groups that are whole TMA boxes.
    // With one H_in per head the heads of a batch go through the same launches, each against its own pieces of H_in
    // (with these groups the batch of Yw holds at most 3 GiB of them): heads of whole 128-row tiles and groups of at most
    // 128 columns.  Everything else is formed in double, its scales correctly rounded and its loss good to 1e-15; the split
    // products leave 1e-6 of the loss and twice the scales' rounding error.
    const bool per_head_ok = (p.n_hin > 1) && (p.dh % 128 == 0) && (p.seg <= 128) && (rows % p.dh == 0);
    p.yw_tensor = (p.n_hin == 1 || per_head_ok) && (p.seg % 64 == 0) && (rows % 8 == 0) && (p.d_out % 8 == 0) &&
                  (p.dh % 8 == 0 || rows == p.d_out);
    if (p.yw_tensor) {
      p.WbT = b.take<__nv_bfloat16>((size_t)rows * dd);
      p.Hp = b.take<__nv_bfloat16>((size_t)3 * dd * dd * (p.n_hin > 1 ? (size_t)(rows / p.dh) : 1));
    }
    if (p.yw_tensor && with_r && with_loss && p.n_hin == 1) p.WR = b.take<double>((size_t)p.d_out * dd);
    const long long lines = rows;  // one set of statistics per row (the column-parallel pass keeps them all)
    if (has_hout && cd_gram_pays((int)(rows / p.dh), p.dh, p.ng)) p.gram = b.take<double>(cd_gram_doubles((int)(rows / p.dh), p.dh, p.ng));
    p.n0 = b.take<double>((size_t)lines * p.ng);
    p.Amat = b.take<double>((size_t)lines * p.ng * p.ng);
  }
  // without the scale refinement the loss forms dW H_in itself: the same split-bf16 product
  // (with one H_in per head the heads of a batch share the launch, each against its own pieces: that
  // needs heads of whole 128-row tiles)
  p.loss_tensor = with_loss && !p.cd && (p.n_hin == 1 || p.dh % 128 == 0) && (p.d % 32 == 0) && (p.d_out % 8 == 0);
  p.loss_heads = 1;
  if (p.loss_tensor && p.n_hin > 1) {
    const size_t per_head = (size_t)3 * dd * dd * sizeof(__nv_bfloat16);
    size_t fit = ((size_t)2 << 30) / per_head;
    if (fit < 1) fit = 1;
    p.loss_heads = (fit < (size_t)p.H) ? (int)fit : p.H;
  }
  if (p.loss_tensor) p.Hp = b.take<__nv_bfloat16>((size_t)3 * dd * dd * (size_t)p.loss_heads);
  if (with_loss) p.G2 = b.take<double>((size_t)p.H * p.dh * (has_hout ? p.dh : 1));  // Z dW^T, or partial sums
  p.ws_total = b.total();
  return TB_OK;
}

static int ew_blocks(long long n) {
  long long b = (n + 255) / 256;
  if (b > 148 * 16) b = 148 * 16;
  if (b < 1) b = 1;
  return (int)b;
}

static tb_status run_grid(const Plan& p, const float* H_in, float* scales, int* zeros,
                          unsigned char* cand, RowMap rm, int M, cudaStream_t st) {
  GridP gp;
  gp.Wt = p.Wt;
  gp.Hin = H_in;
  gp.sD = p.sD;
  gp.s_out = scales;
  gp.z_out = zeros;
  gp.cand_out = cand;
  gp.rm = rm;
  gp.M = M;
  gp.d = p.d;
  gp.seg = p.seg;
  gp.ng = p.ng;
  gp.maxq = p.maxq;
  gp.n_cand = p.n_cand;
  gp.ncp = p.ncp;
  gp.rt = p.rt;
  gp.units = (p.n_hin == 1) ? 1 : p.H;
  gp.rows_per_unit = M / gp.units;
  gp.tiles_per_unit = (gp.rows_per_unit + p.rt - 1) / p.rt;
  gp.Wloc = nullptr;
  gp.grp0 = 0;
  if (p.grid_digits) return grid_digits(gp, p.gd, st);
  if (p.seg > 128)  // E is free until the sweep of a step
    return grid_wide(gp, p.E, p.e_doubles, st);
  static bool configured_tri[64] = {false};
  TB_TRY(allow_smem(k_grid_tri, GRID_TRI_SMEM, configured_tri));
  const long long ytiles = (long long)gp.units * gp.tiles_per_unit;
  if (ytiles > 65535) return TB_ERR_UNSUPPORTED;
  dim3 grid(p.ng, (unsigned)ytiles);
  k_grid_tri<<<grid, GEMM_THREADS, GRID_TRI_SMEM, st>>>(gp);
  TB_LAUNCH_CHECK();
  return TB_OK;
}

static tb_status run_sweep_rows(const Plan& p, const float* U_in, const float* P, unsigned char* codes,
                                const int* zeros, tb_stats* stats, RowMap rm, int M, cudaStream_t st) {
  SweepArgs a;
  a.src = p.Wt;
  a.src_mapped = true;
  a.U = U_in;
  a.P = P;
  a.Err = p.Wk;  // error history of the step's rows (up to SWEEP_OUTER columns)
  a.Arr = p.E;   // arrival values; E itself is formed after the sweep
  a.err_ld = a.err_col0 = 0;
  a.codes = codes;
  a.sD = p.sD;
  a.z = zeros;
  a.stats = stats;
  a.rm = rm;
  a.M = M;
  a.d = p.d;
  a.seg = p.seg;
  a.ng = p.ng;
  a.maxq = p.maxq;
  a.units = (p.n_hin == 1) ? 1 : p.H;
  a.blk0 = a.blk1 = 0;
  return sweep_step(a, p.sweep, st);
}

// Dynamic-grid variant: group by group on the working copy Wk of the step's rows.
static tb_status run_sweep_dynamic(const Plan& p, const float* H_in, const float* U_in, const float* P,
                                   unsigned char* codes, float* scales, int* zeros, unsigned char* cand,
                                   tb_stats* stats, RowMap rm, int M, cudaStream_t st) {
  const int d = p.d, seg = p.seg;
  const int units = (p.n_hin == 1) ? 1 : p.H;
  k_gather<<<ew_blocks((long long)M * d), 256, 0, st>>>(p.Wt, p.Wk, nullptr, rm, M, d);
  TB_LAUNCH_CHECK();
  GridP gp;
  gp.Wt = p.Wt;
  gp.Hin = H_in;
  gp.sD = p.sD;
  gp.s_out = scales;
  gp.z_out = zeros;
  gp.cand_out = cand;
  gp.rm = rm;
  gp.M = M;
  gp.d = d;
  gp.seg = seg;
  gp.ng = p.ng;
  gp.maxq = p.maxq;
  gp.n_cand = p.n_cand;
  gp.ncp = p.ncp;
  gp.rt = p.rt;
  gp.units = units;
  gp.rows_per_unit = M / units;
  gp.tiles_per_unit = (gp.rows_per_unit + p.rt - 1) / p.rt;
  gp.Wloc = p.Wk;
  const long long ytiles = (long long)gp.units * gp.tiles_per_unit;
  if (ytiles > 65535) return TB_ERR_UNSUPPORTED;
  static bool configured_tri[64] = {false};
  TB_TRY(allow_smem(k_grid_tri, GRID_TRI_SMEM, configured_tri));
  GroupPanelP pp;
  pp.Wk = p.Wk;
  pp.U = U_in;
  pp.P = P;
  pp.Err = p.dynErr;
  pp.Arr = p.dynArr;
  pp.codes = codes;
  pp.sD = p.sD;
  pp.z = zeros;
  pp.stats = stats;
  pp.rm = rm;
  pp.M = M;
  pp.d = d;
  pp.seg = seg;
  pp.ng = p.ng;
  pp.maxq = p.maxq;
  pp.units = units;
  pp.rows_per_unit = M / units;
  for (int grp = 0; grp < p.ng; ++grp) {
    gp.grp0 = grp;
    k_grid_tri<<<dim3(1, (unsigned)ytiles), GEMM_THREADS, GRID_TRI_SMEM, st>>>(gp);
    TB_LAUNCH_CHECK();
    pp.grp = grp;
    TB_TRY(group_panel(pp, st));
  }
  return TB_OK;
}

}  // namespace tb

using namespace tb;

namespace tb {
bool g_profile_on = false;
PhaseSpan g_spans[TB_MAX_SPANS];
int g_n_spans = 0;
}  // namespace tb

extern "C" void tb_profile_enable(int on) {
  for (int i = 0; i < g_n_spans; ++i) {
    cudaEventDestroy(g_spans[i].a);
    cudaEventDestroy(g_spans[i].b);
  }
  g_n_spans = 0;
  g_profile_on = (on != 0);
}

extern "C" int tb_profile_read(double* ms_by_phase, int n) {
  for (int i = 0; i < n; ++i) ms_by_phase[i] = 0.0;
  for (int i = 0; i < g_n_spans; ++i) {
    float ms = 0.0f;
    if (cudaEventSynchronize(g_spans[i].b) == cudaSuccess &&
        cudaEventElapsedTime(&ms, g_spans[i].a, g_spans[i].b) == cudaSuccess && g_spans[i].phase < n)
      ms_by_phase[g_spans[i].phase] += (double)ms;
    cudaEventDestroy(g_spans[i].a);
    cudaEventDestroy(g_spans[i].b);
  }
  g_n_spans = 0;
  return PH_COUNT;
}

extern "C" size_t tb_quantize_layer_workspace(const tb_layer_desc* desc, int with_r, int with_loss) {
  Plan p;
  // the larger of the two H_out cases, so that one query serves both
  size_t a = 0, b = 0;
  if (make_plan(desc, true, with_r != 0, with_loss != 0, nullptr, &p) == TB_OK) a = p.ws_total;
  if (make_plan(desc, false, with_r != 0, with_loss != 0, nullptr, &p) == TB_OK) b = p.ws_total;
  return a > b ? a : b;
}

extern "C" tb_status tb_quantize_layer(const tb_layer_desc* desc, const float* W, const float* H_in,
                                       const float* U_in, const float* H_out, const float* U_out,
                                       const float* R, const float* P, const float* C,
                                       unsigned char* codes, float* scales, int* zeros,
                                       unsigned char* cand, float* W_hat, double* W_comp, double* loss,
                                       tb_stats* stats, void* ws, size_t ws_bytes, void* stream) {
  if (!desc || !W || !H_in || !U_in || !codes || !scales || !zeros) return TB_ERR_INVALID_ARG;
  if ((H_out == nullptr) != (U_out == nullptr)) return TB_ERR_INVALID_ARG;
  const bool with_r = (R != nullptr);
  if (with_r != (P != nullptr) || with_r != (C != nullptr)) return TB_ERR_INVALID_ARG;
  if (!aligned(W, 16) || !aligned(H_in, 16) || !aligned(U_in, 16) || (P && !aligned(P, 16)))
    return TB_ERR_INVALID_ARG;
  Plan p;
  TB_TRY(make_plan(desc, H_out != nullptr, with_r, loss != nullptr, nullptr, &p));
  if (!ws || !aligned(ws, 256) || ws_bytes < p.ws_total) return TB_ERR_WORKSPACE;
  TB_TRY(make_plan(desc, H_out != nullptr, with_r, loss != nullptr, ws, &p));
  cudaStream_t st = as_stream(stream);
  const int d = p.d;
  const long long n_all = (long long)p.d_out * d;
  const long long dd = (long long)d * d;

  {
    PhaseScope ph(PH_SETUP, st);
    if (stats) TB_CUDA_CHECK(cudaMemsetAsync(stats, 0, sizeof(tb_stats), st));
    k_widen<<<ew_blocks(n_all), 256, 0, st>>>(W, p.Wt, n_all);
    TB_LAUNCH_CHECK();
    if (p.T) {
      const size_t cm_smem = (size_t)p.g * p.dh * sizeof(float) + 16 + (size_t)p.g * 128 * sizeof(double);
      const bool staged = cm_smem <= 200 * 1024;
      static bool conf_cm[64] = {false};
      TB_TRY(allow_smem(k_comp_matrices, 200 * 1024, conf_cm));
      k_comp_matrices<<<dim3(p.S, p.H), 512, staged ? cm_smem : 0, st>>>(U_out, p.T, p.dh, p.g, p.S, staged ? 1 : 0);
      TB_LAUNCH_CHECK();
    }
    if (p.c_max) {  // C by columns, once for all steps
      const I8Src c{C, d, 0, d, d, 1, true, false, 0, nullptr, 0};
      TB_TRY(i8_row_max(c, p.c_max, d, st));
      TB_TRY(i8_slice(c, p.c_max, d, 0, p.Cdig, 0, 0, 0, st));
    }
  }
  if (!p.dynamic) {
    PhaseScope ph(PH_SWEEP, st);
    TB_TRY(sweep_prepare(U_in, P, d, p.sweep, st));
  }
  if (p.grid_digits) {
    PhaseScope ph(PH_GRID, st);
    TB_TRY(grid_digits_prepare(H_in, (p.n_hin == 1) ? 1 : p.H, d, p.seg, p.gd, st));
  }
  if (!p.adaptive && !p.dynamic) {
    // fixed grid: every row, once, from the original weights
    PhaseScope ph(PH_GRID, st);
    RowMap all{p.dh, p.dh, 0};
    TB_TRY(run_grid(p, H_in, scales, zeros, cand, all, p.d_out, st));
  }

  for (int step = 0; step < p.S; ++step) {
    const int i0 = step * p.g, M = p.H * p.g;
    RowMap rm{p.g, p.dh, i0};
    if (p.adaptive) {
      PhaseScope ph(PH_GRID, st);
      TB_TRY(run_grid(p, H_in, scales, zeros, cand, rm, M, st));
    }
    {
      PhaseScope ph(PH_SWEEP, st);
      if (with_r) {  // the snapshot W0 as a contiguous GEMM operand of the propagated-error term
        k_gather<<<ew_blocks((long long)M * d), 256, 0, st>>>(p.Wt, p.W0c, nullptr, rm, M, d);
        TB_LAUNCH_CHECK();
      }
      if (p.dynamic)
        TB_TRY(run_sweep_dynamic(p, H_in, U_in, P, codes, scales, zeros, cand, stats, rm, M, st));
      else
        TB_TRY(run_sweep_rows(p, U_in, P, codes, zeros, stats, rm, M, st));
    }
    const int nrem = p.dh - i0 - p.g;
    if (!p.has_hout || nrem <= 0) continue;
    PhaseScope ph_comp(PH_COMP, st);
    if (with_r) {
      k_residual<<<ew_blocks((long long)M * d), 256, 0, st>>>(p.Wt, codes, p.sD, zeros, p.E, rm, M, d,
                                                              p.seg, p.ng);
      TB_LAUNCH_CHECK();
    }
    if (p.c_max) {
      // E <- E - W0 (R H_in^{-1})   (Proposition 3.2), a double-precision product on the integer tensor cores.  It
      // feeds the codes.  Two projections, three steps each of 1024 rows x 4096 columns,
      // 12.8 ms on the FP64 pipe, 3.7 ms here.
      const I8Src w{p.W0c, d, 0, M, d, 1, false, true, 0, nullptr, 0};
      TB_TRY(i8_row_max(w, p.w_max, M, st));
      TB_TRY(i8_slice(w, p.w_max, M, 0, p.Wdig, 0, 0, 0, st));
      I8Gemm g = i8_gemm_params();
      g.A = p.Wdig;
      g.B = p.Cdig;
      g.k_blocks = d / I8_KB;
      g.a_max = p.w_max;
      g.b_max = p.c_max;
      g.C = p.E;
      g.ldc = d;
      g.M = M;
      g.N = d;
      g.alpha = -1.0;
      g.beta = 1.0;
      TB_TRY(i8_gemm(g, st));
    } else if (with_r) {
      // the same with one H_in per head
      GemmP g = gemm_params();
      const int units = (p.n_hin == 1) ? 1 : p.H;
      g.A = p.W0c;
      g.a_m = d;
      g.a_k = 1;
      g.B = C;
      g.b_k = d;
      g.b_n = 1;
      g.C = p.E;
      g.ldc = d;
      g.M = M / units;
      g.N = d;
      g.K = d;
      g.n_batch = units;
      g.a_batch = (long long)g.M * d;
      g.c_batch = (long long)g.M * d;
      g.b_batch = (units > 1) ? dd : 0;
      g.alpha = -1.0;
      g.beta = 1.0;
      TB_TRY((gemm_launch<double, float, double, double, false, true>(g, st)));
    }
    if (p.H > 65535) return TB_ERR_UNSUPPORTED;
    const dim3 cgrid(d / 128, p.H, (nrem + 31) / 32);
    const double* Ti = p.T + (long long)step * p.dh * p.g;
    const long long t_head = (long long)p.S * p.dh * p.g;
    const bool ahead = comp_ahead((long long)cgrid.x * cgrid.y * cgrid.z, p.g, with_r);
    auto* kern = with_r ? (ahead ? k_compensate<true, true> : k_compensate<true, false>)
                        : (ahead ? k_compensate<false, true> : k_compensate<false, false>);
    TB_CUDA_CHECK(launch_pdl(kern, cgrid, dim3(256), 0, st, p.Wt, codes, p.sD, zeros, p.E, Ti, i0, p.g, p.dh, t_head, d, p.seg, p.ng));
    TB_LAUNCH_CHECK();
  }

  // A group's rows are never written after they have been taken, and the rows of later groups only by
  // the compensation of the groups before them: after the loop row r of W~ is what the sweep saw.
  if (W_comp)
    TB_CUDA_CHECK(cudaMemcpyAsync(W_comp, p.Wt, (size_t)n_all * sizeof(double), cudaMemcpyDeviceToDevice, st));

  // ---- coordinate descent on the scales (Algorithm 3) ----
  if (p.cd) {
    PhaseScope ph(PH_CD, st);
    const int units = (p.n_hin == 1) ? 1 : p.H;
    k_cd_prep<<<ew_blocks(n_all), 256, 0, st>>>(W, codes, p.sD, zeros, p.Dq, p.Wb, p.d_out, d, p.seg,
                                               p.ng);
    TB_LAUNCH_CHECK();
    for (long long r0 = 0; r0 < p.d_out; r0 += p.cd_rows) {
      const long long rows = (p.d_out - r0 < p.cd_rows) ? (p.d_out - r0) : p.cd_rows;
      // Dm = (Q - W) H_in (+ W R); Yw = blockwise Wbar H_in.  With one H_in per head the batch is whole heads, which share
      // the launches.
      const int hunits = (units > 1) ? (int)(rows / p.dh) : 1;
      const long long head0 = (units > 1) ? (r0 / p.dh) * dd : 0;
      const float* Hb = H_in + head0;
      if (p.yw_tensor) {
        // the pieces of W and of (Q - W), transposed, live in this batch's rows of the W~ buffer (free by now,
        // and overwritten by G = H_out Dm only after the products)
        __nv_bfloat16* DqT = reinterpret_cast<__nv_bfloat16*>(p.Wt + r0 * d);
        double* wr = p.WR ? p.WR + r0 * d : p.Dm + r0 * d;
        if (with_r) {  // W R, to which (Q - W) H_in is added below; the pieces of H_in take the place of R's
          TB_TRY(split3_transpose(W + r0 * d, DqT, rows, d, st));
          TB_TRY(split3(R + head0, p.Hp, dd * hunits, st));
          TB_TRY(gemm_split_presplit(wr, d, DqT, p.Hp, rows, d, d, nullptr, st, hunits));
        }
        // also splits H_in into its bf16 pieces
        TB_TRY(yw_tensor(reinterpret_cast<float*>(p.Yw), codes + r0 * d, zeros + r0 * p.ng, Hb, p.WbT, p.Hp,
                         r0 == 0 || with_r || units > 1, rows, d, p.seg, p.ng, hunits, st));
        TB_TRY(split3_transpose(p.Dq + r0 * d, DqT, rows, d, st));
        TB_TRY(gemm_split_presplit(p.Dm + r0 * d, d, DqT, p.Hp, rows, d, d, with_r ? wr : nullptr, st, hunits));
      } else {
        const long long per = rows / hunits;  // rows against one H_in
        GemmP g = gemm_params();
        g.A = p.Dq + r0 * d;
        g.a_m = d;
        g.a_k = 1;
        g.a_batch = per * d;
        g.B = Hb;
        g.b_k = d;
        g.b_n = 1;
        g.b_batch = dd;
        g.C = p.Dm + r0 * d;
        g.ldc = d;
        g.c_batch = per * d;
        g.M = (int)per;
        g.N = d;
        g.K = d;
        g.n_batch = hunits;
        TB_TRY((gemm_launch<double, float, double, double, false, true>(g, st)));
        if (with_r) {
          GemmP h = g;
          h.A = W + r0 * d;
          h.B = R + head0;
          h.beta = 1.0;
          TB_TRY((gemm_launch<float, float, double, double, false, true>(h, st)));
        }
        // Yw: a launch for each group with all heads, or for each head with all groups, whichever are fewer.  Refinement of 8
        // heads of 128 rows x 2048 columns, groups of 256: 4.00 ms head by head, 1.34 together; 32 heads x 4096, one group:
        // 46.9 and 10.4.
        const bool by_group = p.ng < hunits;
        const long long head_y = per * p.ng * d;
        for (int i = 0; i < (by_group ? p.ng : hunits); ++i) {
          GemmP y = gemm_params();
          y.A = p.Wb + r0 * d + (by_group ? (long long)i * p.seg : i * per * d);
          y.a_m = d;
          y.a_k = 1;
          y.a_batch = by_group ? per * d : p.seg;
          y.B = Hb + (by_group ? (long long)i * p.seg * d : i * dd);
          y.b_k = d;
          y.b_n = 1;
          y.b_batch = by_group ? dd : (long long)p.seg * d;
          y.C = p.Yw + (by_group ? (long long)i * d : i * head_y);
          y.ldc = (long long)p.ng * d;
          y.c_batch = by_group ? head_y : d;
          y.M = (int)per;
          y.N = d;
          y.K = p.seg;
          y.n_batch = by_group ? hunits : p.ng;
          TB_TRY((gemm_launch<float, float, double, double, false, true>(y, st)));
        }
      }
      if (p.has_hout) {
        // rows of a head are coupled through H_out: one CTA per head walks them in order
        const int heads_b = (int)(rows / p.dh);
        const long long nb_el = rows * d;
        CdGram cg_p;
        if (p.gram) {
          cg_p.Yw = p.Yw;
          cg_p.yw_float = p.yw_tensor;
          cg_p.Wb = p.Wb + r0 * d;
          cg_p.Hout = H_out + (r0 / p.dh) * (long long)p.dh * p.dh;
          cg_p.scratch = p.gram;
          cg_p.heads = heads_b;
          cg_p.d = d;
          cg_p.seg = p.seg;
          cg_p.ng = p.ng;
          cg_p.dh = p.dh;
          TB_TRY(cd_gram_form(cg_p, st));
        }
        CdHeadP hp;
        hp.G = p.Wt + r0 * d;      // W~ is no longer needed: its buffer holds G = H_out Dm
        hp.Uacc = p.Dq + r0 * d;   // (Q - W) has been consumed by the product above
        hp.Yw = p.Yw;
        hp.Wb = p.Wb + r0 * d;
        hp.Hout = H_out + (r0 / p.dh) * (long long)p.dh * p.dh;
        hp.sD = p.sD + r0 * p.ng;
        hp.d = d;
        hp.seg = p.seg;
        hp.ng = p.ng;
        hp.dh = p.dh;
        hp.uw = (p.seg % 128 == 0) ? 128 : (p.seg <= 128 ? p.seg : 32);
        // CTAs per head: whole groups per CTA, and no more CTAs than the GPU holds at once
        int csize = 8;
        while (csize > 1 && ((p.ng % csize) || (long long)heads_b * csize > 148)) csize >>= 1;
        hp.csize = csize;
        const int n_units = (p.ng / csize) * (p.seg / hp.uw);
        const size_t sm_head =
            ((size_t)n_units * (p.ng + 1) + 2 * (size_t)p.ng * p.ng + 3 * (size_t)p.ng) * sizeof(double);
        if (!p.gram && sm_head > 200 * 1024) return TB_ERR_UNSUPPORTED;
        static bool conf_head[64] = {false}, conf_head2[64] = {false};
        auto cd_head_kern = p.yw_tensor ? k_cd_head<float> : k_cd_head<double>;
        if (p.yw_tensor)
          TB_TRY(allow_smem(k_cd_head<float>, 200 * 1024, conf_head));
        else
          TB_TRY(allow_smem(k_cd_head<double>, 200 * 1024, conf_head2));
        // column-parallel pass where a CTA's columns fit two per thread and the chain fits a warp
        const int c_cnt = (p.ng / csize) * p.seg;
        const bool by_cols = (p.ng <= CDC_MAXG) && (c_cnt <= 2 * CDC_THREADS) && (p.seg % 2 == 0) && (d % 2 == 0) &&
                             ((size_t)d * sizeof(float) <= 48 * 1024);
        CdColP cp2;
        cp2.G = hp.G;
        cp2.Uacc = hp.Uacc;
        cp2.Yw = hp.Yw;
        cp2.Wb = hp.Wb;
        cp2.Hout = hp.Hout;
        cp2.Mmat = p.Amat;
        cp2.sD = hp.sD;
        cp2.d = d;
        cp2.seg = p.seg;
        cp2.ng = p.ng;
        cp2.dh = p.dh;
        cp2.csize = csize;
        if (by_cols && !p.gram) {
          if (p.yw_tensor)
            k_cd_amat<float><<<(unsigned)rows, 256, (size_t)d * sizeof(float), st>>>(p.Yw, hp.Wb, p.Amat, d, p.seg, p.ng);
          else
            k_cd_amat<double><<<(unsigned)rows, 256, (size_t)d * sizeof(float), st>>>(p.Yw, hp.Wb, p.Amat, d, p.seg, p.ng);
          TB_LAUNCH_CHECK();
          k_cd_chain<<<(unsigned)((rows + 3) / 4), 128, 0, st>>>(p.Amat, rows, p.ng);
          TB_LAUNCH_CHECK();
        }
        for (int it = 0; it < p.cd_iters; ++it) {
          GemmP g = gemm_params();  // G = H_out Dm, head by head
          g.A = hp.Hout;
          g.a_m = p.dh;
          g.a_k = 1;
          g.a_batch = (long long)p.dh * p.dh;
          g.B = p.Dm + r0 * d;
          g.b_k = d;
          g.b_n = 1;
          g.b_batch = (long long)p.dh * d;
          g.C = hp.G;
          g.ldc = d;
          g.c_batch = (long long)p.dh * d;
          g.M = p.dh;
          g.N = d;
          g.K = p.dh;
          g.n_batch = heads_b;
          TB_TRY((gemm_launch<float, double, double, double, false, true>(g, st)));
          if (p.gram) {
            TB_TRY(cd_gram_pass(cg_p, hp.G, p.Dm + r0 * d, hp.sD, st));
            continue;
          }
          cudaLaunchConfig_t cfg = {};
          cfg.gridDim = dim3((unsigned)(heads_b * csize));
          cfg.blockDim = dim3(by_cols ? CDC_THREADS : CDH_THREADS);
          const size_t slab = p.yw_tensor ? (size_t)p.ng * c_cnt * sizeof(float) : 0;
          static bool conf_cols[64] = {false};
          if (by_cols && slab) TB_TRY(allow_smem(k_cd_head_cols<float>, (size_t)CDC_MAXG * 2 * CDC_THREADS * sizeof(float), conf_cols));
          cfg.dynamicSmemBytes = by_cols ? slab : sm_head;
          cfg.stream = st;
          cudaLaunchAttribute attr[1];
          attr[0].id = cudaLaunchAttributeClusterDimension;
          attr[0].val.clusterDim.x = (unsigned)csize;
          attr[0].val.clusterDim.y = 1;
          attr[0].val.clusterDim.z = 1;
          cfg.attrs = attr;
          cfg.numAttrs = 1;
          if (by_cols) {
            if (p.yw_tensor)
              TB_CUDA_CHECK(cudaLaunchKernelEx(&cfg, k_cd_head_cols<float>, cp2));
            else
              TB_CUDA_CHECK(cudaLaunchKernelEx(&cfg, k_cd_head_cols<double>, cp2));
          } else {
            TB_CUDA_CHECK(cudaLaunchKernelEx(&cfg, cd_head_kern, hp));
          }
          TB_LAUNCH_CHECK();
          k_axpy<<<ew_blocks(nb_el), 256, 0, st>>>(p.Dm + r0 * d, hp.Uacc, nb_el);
          TB_LAUNCH_CHECK();
        }
        continue;
      }
      // H_out = I: rows are independent, every row is its own line of one row
      CdP cp;
      cp.Dm = p.Dm + r0 * d;
      cp.Yw = p.Yw;
      cp.Wb = p.Wb + r0 * d;
      cp.sD = p.sD + r0 * p.ng;
      cp.n0 = p.n0;
      cp.Amat = p.Amat;
      cp.d = d;
      cp.seg = p.seg;
      cp.ng = p.ng;
      cp.Hout = nullptr;
      cp.dh = 1;
      cp.lines_per_head = 1;
      cp.j0 = 0;
      const int lines = (int)rows;
      // columns per CTA: whole groups, about 512 columns
      int gpc = 512 / p.seg;
      if (gpc < 1) gpc = 1;
      if (gpc > p.ng) gpc = p.ng;
      cp.groups_per_cta = gpc;
      const int xctas = (p.ng + gpc - 1) / gpc;
      const size_t sm_stats = ((size_t)gpc * (p.seg / 32) * (p.ng + 1) + cp.dh) * sizeof(double);
      size_t sm_upd = ((size_t)2 * p.ng + (size_t)p.ng * p.ng) * sizeof(double);
      cp.a_in_smem = 1;
      if (sm_upd > 200 * 1024) {
        sm_upd = (size_t)2 * p.ng * sizeof(double);
        cp.a_in_smem = 0;
      }
      static bool conf_stats[64] = {false}, conf_upd[64] = {false};
      static bool conf_stats_f[64] = {false}, conf_upd_f[64] = {false};
      TB_TRY(allow_smem(k_cd_row_stats<double>, 200 * 1024, conf_stats));
      TB_TRY(allow_smem(k_cd_row_update<double>, 200 * 1024, conf_upd));
      TB_TRY(allow_smem(k_cd_row_stats<float>, 200 * 1024, conf_stats_f));
      TB_TRY(allow_smem(k_cd_row_update<float>, 200 * 1024, conf_upd_f));
      const size_t ysz = p.yw_tensor ? sizeof(float) : sizeof(double);
      if (sm_stats > 200 * 1024) return TB_ERR_UNSUPPORTED;
      for (int it = 0; it < p.cd_iters; ++it) {
        for (int l0 = 0; l0 < lines; l0 += 65535) {
          const int nl = (lines - l0 < 65535) ? (lines - l0) : 65535;
          CdP cq = cp;  // advance every per-line pointer by l0 rows
          cq.Dm = cp.Dm + (long long)l0 * d;
          cq.Yw = static_cast<const char*>(cp.Yw) + (size_t)l0 * p.ng * d * ysz;
          cq.Wb = cp.Wb + (long long)l0 * d;
          cq.sD = cp.sD + (long long)l0 * p.ng;
          cq.n0 = cp.n0 + (long long)l0 * p.ng;
          cq.Amat = cp.Amat + (long long)l0 * p.ng * p.ng;
          if (p.yw_tensor) {
            k_cd_row_stats<float><<<dim3(xctas, nl), 256, sm_stats, st>>>(cq);
            TB_LAUNCH_CHECK();
            k_cd_row_update<float><<<dim3(xctas, nl), 256, sm_upd, st>>>(cq);
          } else {
            k_cd_row_stats<double><<<dim3(xctas, nl), 256, sm_stats, st>>>(cq);
            TB_LAUNCH_CHECK();
            k_cd_row_update<double><<<dim3(xctas, nl), 256, sm_upd, st>>>(cq);
          }
          TB_LAUNCH_CHECK();
        }
      }
    }
  }

  {
    PhaseScope ph(PH_OUTPUT, st);
    k_dequant<<<ew_blocks(n_all), 256, 0, st>>>(codes, p.sD, zeros, W_hat, scales, p.d_out, d, p.seg,
                                               p.ng);
    TB_LAUNCH_CHECK();
  }

  // ---- loss of the proofs of Propositions 3.1 / 3.2 ----
  if (loss) {
    PhaseScope ph(PH_LOSS, st);
    const int units = (p.n_hin == 1) ? 1 : p.H;
    k_cd_prep<<<ew_blocks(n_all), 256, 0, st>>>(W, codes, p.sD, zeros, p.Dq, nullptr, p.d_out, d,
                                               p.seg, p.ng);
    TB_LAUNCH_CHECK();
    GemmP g = gemm_params();
    g.A = p.Dq;
    g.a_m = d;
    g.a_k = 1;
    g.B = H_in;
    g.b_k = d;
    g.b_n = 1;
    g.C = p.Dm;
    g.ldc = d;
    g.M = p.d_out / units;
    g.N = d;
    g.K = d;
    g.n_batch = units;
    g.a_batch = g.c_batch = (long long)g.M * d;
    g.b_batch = (units > 1) ? dd : 0;
    // Z = dW H_in (+ 2 W R).  After the scale refinement without R the buffer Dm already holds
    // dW H_in for the final scales (it was kept current through the pass), so the product is skipped.
    // With R the pass keeps Dm = dW H_in + W R, so only one more W R is missing.
    // A product of its own takes all of H_in, not the triangle that it folds into (the loss is symmetric in the two dW): half
    // the contraction (4096 rows and columns 0.69 -> 0.42 ms), but what cancels inside dW H_in then cancels after the tensor
    // core's truncating float sums.  Relative error of the loss, 1024 to 2048 columns with a common factor of ten times the usual
    // strength: 0.5e-6 to 1.5e-6 with all of H_in, 2.4e-6 to 3.6e-6 with the triangle; 8 bits, damping 1e-4: up to 4.4e-6, 17e-6.
    const bool dm_is_current = p.cd;
    if (!dm_is_current && p.loss_tensor && units == 1) {
      __nv_bfloat16* DqT = reinterpret_cast<__nv_bfloat16*>(p.Wt);  // W~ is no longer needed
      TB_TRY(split3_transpose(p.Dq, DqT, p.d_out, d, st));
      TB_TRY(split3(H_in, p.Hp, dd, st));
      TB_TRY(gemm_split_presplit(p.Dm, d, DqT, p.Hp, p.d_out, d, d, nullptr, st));
    } else if (!dm_is_current && p.loss_tensor) {
      // one H_in per head: a batch of heads per launch, every head against its own pieces
      for (int h0 = 0; h0 < p.H; h0 += p.loss_heads) {
        const int nb = (p.H - h0 < p.loss_heads) ? (p.H - h0) : p.loss_heads;
        const long long rr = (long long)h0 * p.dh, rows = (long long)nb * p.dh;
        __nv_bfloat16* DqT = reinterpret_cast<__nv_bfloat16*>(p.Wt + rr * d);  // W~ is no longer needed
        TB_TRY(split3_transpose(p.Dq + rr * d, DqT, rows, d, st));
        TB_TRY(split3(H_in + (long long)h0 * dd, p.Hp, dd * nb, st));
        TB_TRY(gemm_split_presplit(p.Dm + rr * d, d, DqT, p.Hp, rows, d, d, nullptr, st, nb));
      }
    } else if (!dm_is_current) {
      TB_TRY((gemm_launch<double, float, double, double, false, true>(g, st)));
    }
    if (p.WR) {
      k_axpy<<<ew_blocks(n_all), 256, 0, st>>>(p.Dm, p.WR, n_all);
      TB_LAUNCH_CHECK();
    } else if (with_r && p.loss_tensor && units == 1) {
      __nv_bfloat16* WT = reinterpret_cast<__nv_bfloat16*>(p.Wt);  // W~ is no longer needed
      TB_TRY(split3_transpose(W, WT, p.d_out, d, st));
      TB_TRY(split3(R, p.Hp, dd, st));
      // doubled in the double result: 2 W would not hold entries above half the float range
      TB_TRY(gemm_split_presplit(p.Dm, d, WT, p.Hp, p.d_out, d, d, p.Dm, st, 1, 2.0));
    } else if (with_r) {
      GemmP h = g;
      h.A = W;
      h.B = R;
      h.alpha = dm_is_current ? 1.0 : 2.0;
      h.beta = 1.0;
      TB_TRY((gemm_launch<float, float, double, double, false, true>(h, st)));
    }
    // loss_h = tr(H_out,h Z_h dW_h^T) = sum over the head's entries of (H_out,h Z_h) .* dW_h: a product
    // with d_in columns (many tiles) and an elementwise reduction, instead of a d_head x d_head product
    // whose contraction runs over d_in on a handful of tiles.
    const double* lhs = p.Dm;
    if (p.has_hout) {
      GemmP q = gemm_params();
      q.A = H_out;
      q.a_m = p.dh;
      q.a_k = 1;
      q.a_batch = (long long)p.dh * p.dh;
      q.B = p.Dm;  // Z
      q.b_k = d;
      q.b_n = 1;
      q.b_batch = (long long)p.dh * d;
      q.C = p.Wt;  // W~ is no longer needed
      q.ldc = d;
      q.c_batch = (long long)p.dh * d;
      q.M = p.dh;
      q.N = d;
      q.K = p.dh;
      q.n_batch = p.H;
      TB_TRY((gemm_launch<float, double, double, double, false, true>(q, st)));
      lhs = p.Wt;
    }
    const int chunks = (p.dh + 31) / 32;
    k_loss_identity_partial<<<dim3(chunks, p.H), 256, 0, st>>>(lhs, p.Dq, p.G2, p.dh, d, chunks);
    TB_LAUNCH_CHECK();
    k_loss_identity_final<<<p.H, 32, 0, st>>>(p.G2, loss, chunks);
    TB_LAUNCH_CHECK();
  }
  return TB_OK;
}
