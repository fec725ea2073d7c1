// tb_factor: U upper triangular with H^{-1} = U^T U (Eq. 2), batched, and
// tb_prepare_correction: P and C of Algorithm 2 (masked operand) / Proposition 3.2.
//
// Route taken for U (the positive-diagonal factor is unique, so any route to it
// is the factor of Eq. 2): with J the index reversal, J H J = L L^T is an
// ordinary lower Cholesky factorisation; then H = (J L J)(J L J)^T with
// M = J L J upper triangular, H^{-1} = M^{-T} M^{-1}, hence U = M^{-1} = J L^{-1} J.
// No inverse of H is formed.  Everything runs in double: with cond(H_in) ~ 1e5
// a float factorisation would lose most of U's digits.
//
// H is first scaled by powers of two to diagonal entries in [1/2, 2), H = D A D: exact, undone exactly in U (whose
// columns it scales), and every entry of L is then below 1.42.  The matrix is padded to dp, the next
// multiple of 64 (identity in the padding).
//   1. A = J D^-1 H D^-1 J                              (k_scale_exp, k_reverse_in)
//   2. right-looking blocked Cholesky, 64-column panels, two launches per panel:
//        k_chol_panel  every CTA factors the 64 x 64 diagonal block and inverts its factor,
//                      then multiplies its rows of the panel by the inverse
//                      (after applying the previous panel's update to its own columns)
//        GEMM          trailing matrix -= panel panel^T from the panel after the next on
//                      (tiles on/below the diagonal)
//   3. the inverses of the 64 x 64 diagonal blocks, a by-product of the panels, to their places (k_inv_diag64)
//   4. L^{-1} by recursive doubling: for block size s = 64, 128, ... every pair of
//      neighbouring inverted blocks A, B with coupling C = L[B rows, A cols] gets
//      its off-diagonal block -B^{-1} C A^{-1} from two batched GEMMs.  Steps 3 and 4
//      follow the factorisation block by block of 512 columns, so that with the
//      look-ahead they run beside the later panels.  L^{-1} takes the place of L: a block of L
//      is dead once its pair has been formed.
//   5. U = J L^{-1} J D^-1, written as float with an explicit zero lower triangle.
// From 1024 columns on the rank-256 updates and the doubling steps of 512 to 16384 columns run on the
// integer tensor cores (tb_i8.cuh); a step of 32768 contracts more than their sums hold and stays on the FP64 pipe.  The digits of L (one exponent for all, see the scaling) serve the
// updates and the first product of a pair; the digits of a pair's inverse halves and of its first product
// take the places of the digits of L that the pair has used up.
#include "tb_common.cuh"
#include "tb_gemm.cuh"
#include "tb_gemm64.cuh"
#include "tb_i8.cuh"
#include "tb_rcp.cuh"

namespace tb {

enum { FNB = 64 };

// exps[i] = e with H_ii 2^(-2e) in [1/2, 2) (0 where the diagonal is not positive and finite); also clears the
// error words of the matrix.  Rows in elimination order: row r of A is row d - 1 - r of H.
__global__ void k_scale_exp(const float* __restrict__ H, int* __restrict__ exps, int* __restrict__ bad, int* info, int d,
                            int dp) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
  if (r == 0) info[b] = 0;
  if (r >= dp) return;
  int e = 0;
  if (r < d) {
    const int i = d - 1 - r;
    const float h = H[((long long)b * d + i) * d + i];
    if (h > 0.0f && h < INFINITY) {
      int x;
      frexp((double)h, &x);  // h = f 2^x, f in [1/2, 1)
      e = x >> 1;            // floor(x / 2): f or 2 f remains
    }
  }
  exps[(long long)b * dp + r] = e;
  bad[(long long)b * dp + r] = 0;
}

// A (dp x dp) <- J D^-1 H D^-1 J in the leading d x d block, identity elsewhere (lower triangle and the
// diagonal blocks only: nothing else is read).  A CTA: 8 rows x 256 columns.
__global__ void __launch_bounds__(256) k_reverse_in(const float* __restrict__ H, const int* __restrict__ exps,
                                                    double* __restrict__ A, int d, int dp) {
  const int j = blockIdx.x * 256 + threadIdx.x, i0 = blockIdx.y * 8;
  if (j >= dp || blockIdx.x * 256 > i0 + 7 + FNB) return;
  const float* Hb = H + (long long)blockIdx.z * d * d;
  const int* eb = exps + (long long)blockIdx.z * dp;
  double* Ab = A + (long long)blockIdx.z * dp * dp;
  const int ej = eb[j];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = i0 + k;
    double v = (i == j) ? 1.0 : 0.0;
    if (i < d && j < d) v = (double)Hb[(long long)(d - 1 - i) * d + (d - 1 - j)] * pow2d(-(eb[i] + ej));
    Ab[(long long)i * dp + j] = v;
  }
}

// U = J L^-1 J D^-1; clean: L^-1 D^-1 (columns scaled, zeros above the diagonal) also replaces L^-1
__global__ void __launch_bounds__(256) k_reverse_out(double* __restrict__ Li, const int* __restrict__ exps,
                                                     float* __restrict__ U, int d, int dp, int clean) {
  const int j = blockIdx.x * 256 + threadIdx.x;
  if (j >= d) return;
  double* Lb = Li + (long long)blockIdx.z * dp * dp;
  float* Ub = U + (long long)blockIdx.z * d * d;
  const int c = d - 1 - j;
  const double sc = pow2d(-exps[(long long)blockIdx.z * dp + c]);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int i = blockIdx.y * 8 + k;
    if (i >= d) break;
    double* l = Lb + (long long)(d - 1 - i) * dp + c;
    const double v = (j >= i) ? *l * sc : 0.0;
    Ub[(long long)i * d + j] = (float)v;
    if (clean) *l = v;
  }
}

// One panel step of the Cholesky factorisation, columns k0 .. k0+63 of the dp x dp matrix.
// Every CTA factors the diagonal block itself (same arithmetic everywhere, so the same result) and inverts its factor;
// CTA x then forms rows k0+64+64y, y = x, x + gridDim.x, .. of the panel, X = A_panel L_kk^{-T}.  L_kk^{-1} is stored in
// Linv[k0 / 64] (64 x 64, row-major, zero upper triangle); nothing reads L_kk itself.  A non-positive pivot is recorded
// in info (first one wins) and replaced by 1.
//
// The chain of 64 dependent pivots bounds a panel.  It runs in one warp, 16 columns at a time: lane (row, half) holds
// 8 entries of its row of [remaining block | inverse so far] (what is eliminated on the left becomes the inverse of
// the unit factor in the same registers), a step is a broadcast of the pivot row, a reciprocal (tb_rcp.cuh) and one multiply-add per entry, about 100 clocks of dependent work.  Nothing
// else runs on that warp's scheduler meanwhile (beside FP64 tensor steps a dependent multiply-add waits 137 clocks
// instead of 9); the warps of the other three apply the previous panel's update to the panel rows.  Everything
// between the blocks of 16 - solving the rows below, updating them - is FP64 tensor steps from shared memory, and so
// is the joining of the 16 x 16 inverses, most of it beside the chain too.  A panel of 2048 columns: 31.6 us with 64
// barrier-separated steps of all threads, 16.4 us now.
//
// update_first: the previous panel's rank-64 update of these 64 columns has not been applied yet (the
// trailing update after a panel leaves out the next panel's columns); the kernel applies it to the
// diagonal block and to its own rows.  That keeps a GEMM launch per panel off the chain of dependent launches.
enum { PLD = 68, PANEL_THREADS = 256 };  // PLD: row pitch of the 64 x 64 tiles (doubles); fragment loads without conflicts
static constexpr size_t PANEL_SMEM = (size_t)(5 * 64 + 32) * PLD * sizeof(double);

__device__ __forceinline__ void cp_async_16(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem_dst)), "l"(gsrc)
               : "memory");
}

// 16 x 16 block at (o, o) of D (lower triangle) -> inverse of its lower Cholesky factor at (o, o) of I, by one warp
__device__ __forceinline__ void panel_factor16(const double* D, double* I, int o, const int* sbad, int* info, int first,
                                               bool report) {
  const int lane = threadIdx.x & 31, row = lane & 15, half = lane >> 4;
  double v[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int col = 8 * half + c, hi = max(row, col), lo = min(row, col);
    v[c] = D[(o + hi) * PLD + o + lo];
  }
  constexpr unsigned all = 0xffffffffu;
  const unsigned badmask = __ballot_sync(all, sbad[o + row] != 0);  // lanes 0-15: the block's rows
  unsigned fail = 0;
  double piv = 1.0;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int hj = j >> 3, cj = j & 7;
    double pj = __shfl_sync(all, v[cj], hj * 16 + j);
    const double fi = __shfl_sync(all, v[cj], hj * 16 + row);
    double t[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) t[c] = fi * __shfl_sync(all, v[c], half * 16 + j);
    const bool ok = (pj > 0.0) && !((badmask >> j) & 1u);
    fail |= ok ? 0u : 1u << j;
    pj = ok ? pj : 1.0;
    const double r = panel_rcp(pj);
    if (row == j) piv = pj;
    if (row > j) {
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = fma(-t[c], r, v[c]);
      if (half == hj) v[cj] = -fi * r;
    }
  }
  if (fail && report && lane == 0) atomicCAS(info, 0, first + o + __ffs(fail));
  const double rs = rsqrt(piv);
#pragma unroll
  for (int c = 0; c < 8; c += 2) {
    const int col = 8 * half + c;
    const double x = (col < row) ? v[c] * rs : (col == row) ? rs : 0.0;
    const double y = (col + 1 < row) ? v[c + 1] * rs : (col + 1 == row) ? rs : 0.0;
    *reinterpret_cast<double2*>(I + (o + row) * PLD + o + col) = make_double2(x, y);
  }
}

__global__ void __launch_bounds__(PANEL_THREADS) k_chol_panel(double* __restrict__ A, double* __restrict__ Linv,
                                                              long long linv_batch, int* __restrict__ info, int dp,
                                                              int k0, int row_blocks, int update_first,
                                                              const int* __restrict__ bad) {
  extern __shared__ __align__(16) unsigned char panel_raw[];
  double* sD = reinterpret_cast<double*>(panel_raw);  // the diagonal block, its factor's off-diagonal 16 x 16 blocks
  double* sI = sD + 64 * PLD;                         // inverse of the factor
  double* sR = sI + 64 * PLD;                         // panel rows
  double* sPd = sR + 64 * PLD;                        // previous panel, rows of the diagonal block
  double* sPr = sPd + 64 * PLD;                       // previous panel, the panel rows
  double* sT = sPr + 64 * PLD;                        // scratch of the joins, 32 rows
  __shared__ int sbad[FNB];  // rows whose entries left of this panel were not finite
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b = blockIdx.y;
  const int fr = lane >> 2, fk = lane & 3;
  double* Ab = A + (long long)b * dp * dp;
  double* diag = Ab + (long long)k0 * dp + k0;
  if (tid < FNB) sbad[tid] = bad[(long long)b * dp + k0 + tid];
  auto load_tile = [&](double* dst, const double* src) {
    const int ch = tid & 31, r0 = tid >> 5;  // 16-byte piece ch of rows r0, r0 + 8, ...
#pragma unroll
    for (int i = 0; i < 8; ++i) cp_async_16(dst + (8 * i + r0) * PLD + 2 * ch, src + (long long)(8 * i + r0) * dp + 2 * ch);
  };
  auto panel_row = [&](int y) { return diag + (long long)(y + 1) * FNB * dp; };
  int y = blockIdx.x;
  load_tile(sD, diag);
  if (update_first) load_tile(sPd, diag - FNB);
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (y < row_blocks) {
    load_tile(sR, panel_row(y));
    if (update_first) load_tile(sPr, panel_row(y) - FNB);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int i = tid; i < 64 * 32; i += PANEL_THREADS)
    *reinterpret_cast<double2*>(sI + (i >> 5) * PLD + (i & 31) * 2) = make_double2(0.0, 0.0);
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();
  if (update_first) {  // D -= Pd Pd^T, the 36 fragments on and below the diagonal dealt to the warps in turn
    int fm[5], fn[5];
    double acc[5][2];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      int m = 0, n = warp + 8 * i;
      while (n > m) n -= ++m;
      fm[i] = m;
      fn[i] = n;
      acc[i][0] = acc[i][1] = 0.0;
    }
    const int nt = (warp < 4) ? 5 : 4;
#pragma unroll 4
    for (int q = 0; q < 16; ++q)
#pragma unroll
      for (int i = 0; i < 5; ++i)
        if (i < nt) dmma(acc[i], sPd[(8 * fm[i] + fr) * PLD + 4 * q + fk], sPd[(8 * fn[i] + fr) * PLD + 4 * q + fk]);
#pragma unroll
    for (int i = 0; i < 5; ++i)
      if (i < nt) {
        double2* d = reinterpret_cast<double2*>(sD + (8 * fm[i] + fr) * PLD + 8 * fn[i] + 2 * fk);
        const double2 v = *d;
        *d = make_double2(v.x - acc[i][0], v.y - acc[i][1]);
      }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // fragment (m, n) of R -= Pr Pd^T
  auto update_rows = [&](int m, int n) {
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 4
    for (int q = 0; q < 16; ++q)
      dmma(acc[q & 1], sPr[(8 * m + fr) * PLD + 4 * q + fk], sPd[(8 * n + fr) * PLD + 4 * q + fk]);
    double2* d = reinterpret_cast<double2*>(sR + (8 * m + fr) * PLD + 8 * n + 2 * fk);
    const double2 v = *d;
    *d = make_double2(v.x - (acc[0][0] + acc[1][0]), v.y - (acc[0][1] + acc[1][1]));
  };
  // Joining two neighbouring inverses of s columns, [A 0; C B]^{-1} = [A^{-1} 0; -B^{-1} (C A^{-1}) B^{-1}], A at
  // column o: the first product goes to scratch (sT, column tc), fragments dealt to nw warps
  auto first_product = [&](int o, int s, int tc, int w, int nw) {
    const int nfs = s / 8;
    for (int i = w; i < nfs * nfs; i += nw) {
      const int m = i / nfs, n = i % nfs;
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
      for (int q = 2 * n; q < s / 4; q += 2) {  // A^{-1}(k, n) = 0 for k < n
        dmma(acc[0], sD[(o + s + 8 * m + fr) * PLD + o + 4 * q + fk], sI[(o + 4 * q + fk) * PLD + o + 8 * n + fr]);
        dmma(acc[1], sD[(o + s + 8 * m + fr) * PLD + o + 4 * q + 4 + fk], sI[(o + 4 * q + 4 + fk) * PLD + o + 8 * n + fr]);
      }
      *reinterpret_cast<double2*>(sT + (8 * m + fr) * PLD + tc + 8 * n + 2 * fk) =
          make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
    }
  };
  auto second_product = [&](int o, int s, int tc, int w, int nw) {
    const int nfs = s / 8;
    for (int i = w; i < nfs * nfs; i += nw) {
      const int m = nfs - 1 - i / nfs, n = i % nfs;
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
      for (int q = 0; q < 2 * (m + 1); q += 2) {  // B^{-1}(m, k) = 0 for k > m
        dmma(acc[0], sI[(o + s + 8 * m + fr) * PLD + o + s + 4 * q + fk], sT[(4 * q + fk) * PLD + tc + 8 * n + fr]);
        dmma(acc[1], sI[(o + s + 8 * m + fr) * PLD + o + s + 4 * q + 4 + fk], sT[(4 * q + 4 + fk) * PLD + tc + 8 * n + fr]);
      }
      *reinterpret_cast<double2*>(sI + (o + s + 8 * m + fr) * PLD + o + 8 * n + 2 * fk) =
          make_double2(-(acc[0][0] + acc[1][0]), -(acc[0][1] + acc[1][1]));
    }
  };
#pragma unroll 1
  for (int jb = 0; jb < 4; ++jb) {
    const int o = 16 * jb;
    if (warp == 0) {
      panel_factor16(sD, sI, o, sbad, info + b, k0, blockIdx.x == 0);
    } else if (warp != 4) {  // warp 4 shares warp 0's scheduler
      const int w = warp < 4 ? warp - 1 : warp - 2;
      // what the inverse needs of finished blocks: the join of the first two, then the first products of the rest
      if (jb == 2 && w == 0) {
        first_product(0, 16, 0, 0, 1);
        __syncwarp();
        second_product(0, 16, 0, 0, 1);
      }
      if (jb == 3) {
        first_product(0, 32, 0, w, 6);
        if (w == 5) first_product(32, 16, 32, 0, 1);
      }
      if (update_first && y < row_blocks)
        for (int i = w; i < 16; i += 6) update_rows(2 * jb + (i >> 3), i & 7);
    }
    __syncthreads();
    if (jb == 3) break;
    const int nf = 2 * (3 - jb);
    if (warp < nf) {  // rows below: L = D I^T, 8 rows a warp
      const int r = o + 16 + 8 * warp;
      double a[4], acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] = sD[(r + fr) * PLD + o + 4 * q + fk];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int n = 0; n < 2; ++n) dmma(acc[n], a[q], sI[(o + 8 * n + fr) * PLD + o + 4 * q + fk]);
      __syncwarp();
#pragma unroll
      for (int n = 0; n < 2; ++n)
        *reinterpret_cast<double2*>(sD + (r + fr) * PLD + o + 8 * n + 2 * fk) = make_double2(acc[n][0], acc[n][1]);
    }
    __syncthreads();
    for (int i = warp; i < nf * (nf + 1) / 2; i += 8) {  // D -= L L^T, fragments on and below the diagonal
      int m = 0, n = i;
      while (n > m) n -= ++m;
      const int r = o + 16 + 8 * m, c = o + 16 + 8 * n;
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        dmma(acc[q & 1], sD[(r + fr) * PLD + o + 4 * q + fk], sD[(c + fr) * PLD + o + 4 * q + fk]);
      double2* d = reinterpret_cast<double2*>(sD + (r + fr) * PLD + c + 2 * fk);
      const double2 v = *d;
      *d = make_double2(v.x - (acc[0][0] + acc[1][0]), v.y - (acc[0][1] + acc[1][1]));
    }
    __syncthreads();
  }
  second_product(32, 16, 32, warp, 8);
  __syncthreads();
  second_product(0, 32, 0, warp, 8);
  __syncthreads();
  if (blockIdx.x == 0) {
    // never over the input: the CTAs of this launch need not run at the same time, and one that starts late must
    // still find the unfactored block
    double* dst = Linv + (long long)b * linv_batch + (long long)(k0 / FNB) * FNB * FNB;
    for (int i = tid; i < 64 * 32; i += PANEL_THREADS)
      *reinterpret_cast<double2*>(dst + 2 * i) = *reinterpret_cast<const double2*>(sI + (i >> 5) * PLD + (i & 31) * 2);
  }
  for (; y < row_blocks; y += gridDim.x) {
    if (y != (int)blockIdx.x) {  // further rows of this CTA
      __syncthreads();
      load_tile(sR, panel_row(y));
      if (update_first) load_tile(sPr, panel_row(y) - FNB);
      asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (update_first)
        for (int n = 0; n < 8; ++n) update_rows(warp, n);
      __syncwarp();  // a warp's rows are its own from here on
    }
    // X = R I^T, 8 rows a warp; I(n, k) = 0 for k > n
    double a[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = sR[(8 * warp + fr) * PLD + 4 * q + fk];
    double* out = panel_row(y) + (long long)(8 * warp + fr) * dp + 2 * fk;
#pragma unroll
    for (int n = 0; n < 8; ++n) {
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
      for (int q = 0; q < 2 * (n + 1); ++q) dmma(acc[q & 1], a[q], sI[(8 * n + fr) * PLD + 4 * q + fk]);
      *reinterpret_cast<double2*>(out + 8 * n) = make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
    }
  }
}

// The inverses of the 64 x 64 diagonal blocks of L to their places in L^{-1}.  The part of the block's rows right of
// it, up to the end of its block of 512 columns, becomes zero: the doubling products inside that block read it.
__global__ void __launch_bounds__(256) k_inv_diag64(const double* __restrict__ Linv, long long linv_batch,
                                                    double* __restrict__ Li, int dp, int blk0, int col_end) {
  const int blk = blk0 + blockIdx.x, b = blockIdx.y;
  double* dst = Li + (long long)b * dp * dp + (long long)blk * FNB * (dp + 1);
  const double2* src = reinterpret_cast<const double2*>(Linv + (long long)b * linv_batch + (long long)blk * FNB * FNB);
  const int width = (col_end - blk * FNB) / 2;
  for (int i = threadIdx.x; i < FNB * width; i += 256) {
    const int r = i / width, c = i % width;
    reinterpret_cast<double2*>(dst + (long long)r * dp)[c] = (c < FNB / 2) ? src[r * (FNB / 2) + c] : make_double2(0.0, 0.0);
  }
}

// strictly-upper mask of a square matrix (Algorithm 2: (R U^T) .* M_U)
__global__ void k_mask_strict_upper(const double* __restrict__ src, double* __restrict__ dst, int d) {
  const long long n = (long long)d * d;
  for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
       idx += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(idx / d), j = (int)(idx % d);
    dst[idx] = (j > i) ? src[idx] : 0.0;
  }
}

enum { INV_BLOCK = 512 };  // the inverse is completed block by block of this many columns (see factor_run)

struct FactorWs {
  double *A, *tmp;  // A: the scaled matrix, then L, then L^-1
  int *exps, *bad;
  unsigned long long* mx;  // largest magnitudes of the rows and columns of the doubling products' operands
  I8Mat digits;            // of L, then of the operands of the doubling products
  bool use_i8;
  int dp;
  size_t tmp_per;   // doubles of tmp per matrix
  size_t low_off;   // products of the doubling levels inside one block of INV_BLOCK columns (two regions in turn)
  size_t high_off;  // products of the levels above, one region per level (level s at high_off + sum of the lower s^2)
  size_t total;
};

// The digits pay where the contraction and the matrix are large: one factor of 2048 columns takes the same time
// either way (1.36 ms on the FP64 pipe, 1.37), of 4096 3.44 and 2.86, 8 x 8192 114 and 62; below 1024 there
// is no block update wide enough.
enum { FACTOR_I8_MIN = 1024 };

static FactorWs factor_ws(int n_batch, int d, void* ws) {
  FactorWs f;
  Bump b(ws);
  f.dp = ((d + FNB - 1) / FNB) * FNB;
  const size_t dp = (size_t)f.dp, n = dp * dp;
  f.use_i8 = f.dp >= FACTOR_I8_MIN;
  f.A = b.take<double>((size_t)n_batch * n);
  f.exps = b.take<int>((size_t)n_batch * dp);
  f.bad = b.take<int>((size_t)n_batch * dp);
  // tmp per matrix: the inverses of the factored diagonal blocks (dp x 64), then the intermediate products of the
  // doubling steps.  The inverse proceeds while later panels are still being factored, and a product
  // of a high level stays alive while lower levels run, so each gets a region of its own.
  const size_t gdim = (dp < INV_BLOCK) ? dp : (size_t)INV_BLOCK;
  f.low_off = dp * FNB;
  f.high_off = f.low_off + 2 * (gdim * gdim / 4);  // two regions: neighbouring blocks are inverted side by side
  f.tmp_per = f.high_off;
  for (size_t sb = INV_BLOCK; sb < dp; sb <<= 1) f.tmp_per += sb * sb;
  f.tmp = b.take<double>((size_t)n_batch * f.tmp_per + 64);
  f.mx = nullptr;
  f.digits = I8Mat{nullptr, 0, 0};
  if (f.use_i8) {
    f.digits.row_blocks = (long long)n_batch * (f.dp / I8_RB);
    f.digits.k_blocks = f.dp / I8_KB;
    f.digits.data = b.take<unsigned char>(i8_bytes(f.digits.row_blocks, f.digits.k_blocks));
    // columns of the first product's right operand, rows and columns of the second's
    f.mx = b.take<unsigned long long>((size_t)n_batch * 3 * dp);
  }
  f.total = b.total();
  return f;
}

// Helper stream of the look-ahead (one per device, created on first use, kept until exit).
// The panels with the update of their own 64 columns are the critical path: they get a stream of the
// highest priority, so that their few CTAs are placed before the many tiles of a trailing update that
// is still being dispatched.  The first products of the upper doubling levels are large, and nothing
// needs them before the pair's second half has been factored and inverted: they get a stream of the
// lowest priority of their own (one per level: a small product must not queue behind a large one of the
// level above), so that the block-by-block part of the inverse does not wait for them needlessly.
struct FactorSide {
  cudaStream_t crit;    // panels (each applies the previous panel's update to its own columns first)
  cudaStream_t stream;  // trailing updates
  cudaStream_t inv;     // the inverse above the blocks: second products of the upper levels
  cudaStream_t low[2];  // the inverse inside a block of 512 columns, blocks in turn
  cudaStream_t inv2[8];  // first products of the doubling levels above one block, a stream per level
  cudaStream_t rest;    // the wide rank-256 updates beyond the next outer block's columns
  cudaEvent_t fork, panel, trail[2], block_done, inv_done, crit_done, half_done, first_done[8], low_done[2];
  cudaEvent_t outer_panels, strip_done, rest_done;
  bool ready;
};

static FactorSide* factor_side() {
  static FactorSide per_device[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  FactorSide* s = &per_device[dev];
  if (!s->ready) {
    int least = 0, greatest = 0;
    if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) return nullptr;
    const int middle = (greatest < least) ? greatest + 1 : least;  // numerically lower = more urgent
    if (cudaStreamCreateWithPriority(&s->crit, cudaStreamNonBlocking, greatest) != cudaSuccess) return nullptr;
    if (cudaStreamCreateWithPriority(&s->stream, cudaStreamNonBlocking, middle) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->crit_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->fork, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->panel, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->trail[0], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->trail[1], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaStreamCreateWithPriority(&s->inv, cudaStreamNonBlocking, middle) != cudaSuccess) return nullptr;
    for (int i = 0; i < 8; ++i)
      if (cudaStreamCreateWithPriority(&s->inv2[i], cudaStreamNonBlocking, least) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->half_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    for (int i = 0; i < 2; ++i) {
      if (cudaStreamCreateWithPriority(&s->low[i], cudaStreamNonBlocking, middle) != cudaSuccess) return nullptr;
      if (cudaEventCreateWithFlags(&s->low_done[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    }
    for (int i = 0; i < 8; ++i)
      if (cudaEventCreateWithFlags(&s->first_done[i], cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->block_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->inv_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaStreamCreateWithPriority(&s->rest, cudaStreamNonBlocking, least) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->outer_panels, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->strip_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    if (cudaEventCreateWithFlags(&s->rest_done, cudaEventDisableTiming) != cudaSuccess) return nullptr;
    s->ready = true;
  }
  return s;
}

tb_status factor_run(const float* H, int n_batch, int d, float* U, float* Hinv, int* info, void* ws, size_t ws_bytes,
                     void* stream, bool lookahead);

}  // namespace tb

using namespace tb;

extern "C" size_t tb_factor_workspace(int n_batch, int d) {
  if (n_batch <= 0 || d <= 0) return 0;
  // never less than two matrices in double, the bound that callers' arenas go by (one place fewer is in use since
  // L^-1 takes the place of L)
  const size_t two = ((size_t)2 * n_batch * d * d * sizeof(double) / 256 + 1) * 256;
  const size_t total = factor_ws(n_batch, d, nullptr).total;
  return total > two ? total : two;
}

extern "C" tb_status tb_factor(const float* H, int n_batch, int d, float* U, float* Hinv, int* info,
                               void* ws, size_t ws_bytes, void* stream) {
  return factor_run(H, n_batch, d, U, Hinv, info, ws, ws_bytes, stream, true);
}

// lookahead: the panels run on a stream of high priority, the trailing updates (which leave out the
// next panel's columns: that panel applies its share itself) on a second stream beside the next panel,
// the inverse of the blocks already factored on a third.  Every entry still receives its updates in
// the same order and every product is the same launch, so the result is the same bit for bit.  Without
// it (callers that must not create a stream) everything runs on the caller's stream.
tb_status tb::factor_run(const float* H, int n_batch, int d, float* U, float* Hinv, int* info, void* ws,
                         size_t ws_bytes, void* stream, bool lookahead) {
  if (!H || !U || !info || n_batch <= 0 || n_batch > 65535 || d <= 0) return TB_ERR_INVALID_ARG;
  if (!ws || !aligned(ws, 256) || ws_bytes < tb_factor_workspace(n_batch, d)) return TB_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  FactorWs f = factor_ws(n_batch, d, ws);
  const int dp = f.dp;
  const long long pp = (long long)dp * dp;
  if (dp > 65536) return TB_ERR_UNSUPPORTED;
  k_scale_exp<<<dim3((dp + 255) / 256, n_batch), 256, 0, st>>>(H, f.exps, f.bad, info, d, dp);
  TB_LAUNCH_CHECK();
  k_reverse_in<<<dim3((dp + 255) / 256, dp / 8, n_batch), 256, 0, st>>>(H, f.exps, f.A, d, dp);
  TB_LAUNCH_CHECK();

  static bool panel_configured[64] = {false};
  TB_TRY(allow_smem(k_chol_panel, PANEL_SMEM, panel_configured));
  const int d_fact = dp;
  FactorSide* side = nullptr;
  if (lookahead && d_fact >= 16 * FNB) {
    side = factor_side();
    if (!side) return TB_ERR_CUDA;
    TB_CUDA_CHECK(cudaEventRecord(side->fork, st));
    TB_CUDA_CHECK(cudaStreamWaitEvent(side->stream, side->fork, 0));
    TB_CUDA_CHECK(cudaStreamWaitEvent(side->crit, side->fork, 0));
    TB_CUDA_CHECK(cudaStreamWaitEvent(side->rest, side->fork, 0));
  }
  // L^{-1} block by block of G columns.  Block j can be inverted as soon as its last panel is factored:
  // its 64 x 64 diagonal inverses, the doubling levels inside the block, then every level above whose
  // pair this block completes (second product), and the first product of the one pair whose first half
  // it completes (that product needs only columns already final).  With the look-ahead all of this runs
  // on a stream of its own beside the later panels, and little of the inverse is left after the last
  // panel; without it the same launches follow the panels on the caller's stream.  Every product is
  // the same launch either way, so the result is the same bit for bit.
  const int G = INV_BLOCK;
  const int n_inv_blocks = (dp + G - 1) / G, n_panels = dp / FNB;
  const long long rb = dp / I8_RB;  // row blocks of digits per matrix
  cudaStream_t inv_st = side ? side->inv : st;
  cudaStream_t cs = side ? side->crit : st;  // stream of the panels
  // A pair at level s: columns off .. off + s - 1 (inverse A^{-1} in place) and the m2 <= s rows below them.
  // first product: T = C A^{-1}, C = L[off+s.., off..], m2 x s
  auto pair_first = [&](int sblk, int m2, long long off, long long pair_stride, int batch, double* tmp, long long tmp_stride,
                        cudaStream_t stream_first) -> tb_status {
    GemmP g = gemm_params();
    g.A = f.A + off + (long long)sblk * dp;
    g.a_m = dp;
    g.a_k = 1;
    g.a_batch = pair_stride;
    g.B = f.A + off;
    g.b_k = dp;
    g.b_n = 1;
    g.b_batch = pair_stride;
    g.C = tmp;
    g.ldc = sblk;
    g.c_batch = tmp_stride;
    g.M = m2;
    g.N = sblk;
    g.K = sblk;
    g.n_batch = batch;
    g.btrim = 2;
    g.flags = GEMM_HEAVY_N_FIRST;
    return gemm64_launch<true>(g, stream_first);
  };
  // second product: L^{-1}[off+s.., off..] = -B^{-1} T, B^{-1} = L^{-1}[off+s.., off+s..] (lower triangular)
  auto pair_second = [&](int sblk, int m2, long long off, long long pair_stride, int batch, double* tmp, long long tmp_stride,
                         cudaStream_t stream_second) -> tb_status {
    GemmP h = gemm_params();
    h.A = f.A + off + (long long)sblk * (dp + 1);
    h.a_m = dp;
    h.a_k = 1;
    h.a_batch = pair_stride;
    h.B = tmp;
    h.b_k = sblk;
    h.b_n = 1;
    h.b_batch = tmp_stride;
    h.C = f.A + off + (long long)sblk * dp;
    h.ldc = dp;
    h.c_batch = pair_stride;
    h.M = m2;
    h.N = sblk;
    h.K = m2;
    h.n_batch = batch;
    h.alpha = -1.0;
    h.atrim = 1;
    h.flags = GEMM_HEAVY_M_LAST;
    return gemm64_launch<true>(h, stream_second);
  };
  // The same two products on the integer tensor cores, all matrices of the batch (o: first column of the pair).  The
  // digits of A^{-1} (by columns) take the place of those of the square of L it is the inverse of, and so do the
  // digits of B^{-1}; the digits of T (by columns) that of C's.  Every update that reads one of these parts of L
  // belongs to columns that have been factored by then.
  // beside the panels: CTAs that end soon, unless the products of many matrices bound the time anyway
  const int tile_life = side ? (n_batch >= 4 ? 8 : 2) : 0;
  // row / column maxima, indexed by the pair's columns: pairs whose products run side by side have no column in common
  auto level_max = [&](int which) { return f.mx + (size_t)n_batch * dp * which; };
  auto pair_first_i8 = [&](int sblk, int m2, int o, double* tmp, cudaStream_t s1) -> tb_status {
    unsigned long long* mx = level_max(0) + o;
    I8Src b{f.A + (long long)o * (dp + 1), dp, pp, sblk, sblk, n_batch, false, false, 2, nullptr, 0};
    TB_TRY(i8_row_max(b, mx, dp, s1));
    TB_TRY(i8_slice(b, mx, dp, 0, f.digits, o / I8_RB, rb, o / I8_KB, s1));
    I8Gemm g = i8_gemm_params();
    g.A = g.B = f.digits;
    g.a_rb = (o + sblk) / I8_RB;
    g.b_rb = o / I8_RB;
    g.a_rb_batch = g.b_rb_batch = rb;
    g.a_kb = g.b_kb = o / I8_KB;
    g.k_blocks = sblk / I8_KB;
    g.a_exp = 1;
    g.b_max = mx;
    g.b_max_batch = dp;
    g.C = tmp;
    g.ldc = sblk;
    g.c_batch = (long long)f.tmp_per;
    g.M = m2;
    g.N = sblk;
    g.n_batch = n_batch;
    g.zeros = 2;
    g.order = 1;
    g.tiles_per_cta = tile_life;
    return i8_gemm(g, s1);
  };
  auto pair_second_i8 = [&](int sblk, int m2, int o, double* tmp, cudaStream_t s2) -> tb_status {
    unsigned long long *ma = level_max(1) + o, *mt = level_max(2) + o;
    const int o2 = o + sblk;
    I8Src a{f.A + (long long)o2 * (dp + 1), dp, pp, m2, m2, n_batch, false, true, 1, nullptr, 0};
    TB_TRY(i8_row_max(a, ma, dp, s2));
    TB_TRY(i8_slice(a, ma, dp, 0, f.digits, o2 / I8_RB, rb, o2 / I8_KB, s2));
    // T: sblk columns (rows of digits), m2 contraction steps
    I8Src t{tmp, sblk, (long long)f.tmp_per, sblk, m2, n_batch, false, false, 0, nullptr, 0};
    TB_TRY(i8_row_max(t, mt, dp, s2));
    TB_TRY(i8_slice(t, mt, dp, 0, f.digits, o / I8_RB, rb, o2 / I8_KB, s2));
    I8Gemm g = i8_gemm_params();
    g.A = g.B = f.digits;
    g.a_rb = o2 / I8_RB;
    g.b_rb = o / I8_RB;
    g.a_rb_batch = g.b_rb_batch = rb;
    g.a_kb = g.b_kb = o2 / I8_KB;
    g.k_blocks = m2 / I8_KB;
    g.a_max = ma;
    g.a_max_batch = dp;
    g.b_max = mt;
    g.b_max_batch = dp;
    g.C = f.A + (long long)o2 * dp + o;
    g.ldc = dp;
    g.c_batch = pp;
    g.M = m2;
    g.N = sblk;
    g.n_batch = n_batch;
    g.alpha = -1.0;
    g.zeros = 1;
    g.order = 2;
    g.tiles_per_cta = tile_life;
    return i8_gemm(g, s2);
  };
  auto high_tmp = [&](int sblk) {  // region of the level-sblk product (first matrix of the batch)
    size_t o = f.high_off;
    for (size_t sb = (size_t)G; sb < (size_t)sblk; sb <<= 1) o += sb * sb;
    return f.tmp + o;
  };
  auto invert_block = [&](int j) -> tb_status {
    const int o0 = j * G, width = (dp - o0 < G) ? dp - o0 : G;  // the last block may be narrower
    const long long boff = (long long)o0 * (dp + 1);
    // inside the block: a stream per block parity, so that a block does not wait for its neighbour's
    // upper levels; the caller has just recorded block_done
    cudaStream_t low_st = side ? side->low[j & 1] : inv_st;
    const size_t low_region = f.low_off + (size_t)(j & 1) * ((f.high_off - f.low_off) / 2);
    if (side) TB_CUDA_CHECK(cudaStreamWaitEvent(low_st, side->block_done, 0));
    k_inv_diag64<<<dim3(width / FNB, n_batch), 256, 0, low_st>>>(f.tmp, (long long)f.tmp_per, f.A, dp, j * (G / FNB),
                                                                 o0 + width);
    TB_LAUNCH_CHECK();
    for (int sblk = FNB; sblk < width; sblk <<= 1) {
      const int full = width / (2 * sblk);                  // pairs with both halves complete
      const int rest = width - full * 2 * sblk - sblk;      // rows of a shorter second half, if positive
      // one batched launch covers all pairs of one matrix's block, or (a single pair) all matrices
      const int outer = (full <= 1) ? 1 : n_batch;
      for (int mb = 0; full > 0 && mb < outer; ++mb) {
        const long long off = (long long)mb * pp + boff;
        const long long pair_stride = (full == 1) ? pp : (long long)2 * sblk * (dp + 1);
        const int batch = (full == 1) ? n_batch : full;
        double* tmp = f.tmp + (size_t)mb * f.tmp_per + low_region;
        const long long tmp_stride = (full == 1) ? (long long)f.tmp_per : (long long)sblk * sblk;
        TB_TRY(pair_first(sblk, sblk, off, pair_stride, batch, tmp, tmp_stride, low_st));
        TB_TRY(pair_second(sblk, sblk, off, pair_stride, batch, tmp, tmp_stride, low_st));
      }
      if (rest > 0) {
        const long long off = boff + (long long)full * 2 * sblk * (dp + 1);
        double* tmp = f.tmp + low_region;
        TB_TRY(pair_first(sblk, rest, off, pp, n_batch, tmp, (long long)f.tmp_per, low_st));
        TB_TRY(pair_second(sblk, rest, off, pp, n_batch, tmp, (long long)f.tmp_per, low_st));
      }
    }
    if (side) {
      TB_CUDA_CHECK(cudaEventRecord(side->low_done[j & 1], low_st));
      TB_CUDA_CHECK(cudaStreamWaitEvent(side->inv, side->low_done[j & 1], 0));
    }
    const bool last = j == n_inv_blocks - 1;
    int level = 0;
    for (int sblk = G; sblk < dp; sblk <<= 1, ++level) {
      const int mblk = sblk / G;  // blocks per half of a pair at this level
      if (!last && (j + 1) % mblk) break;
      const bool level_i8 = f.use_i8 && sblk <= I8_MAX_K_BLOCKS * I8_KB;
      const int half = j / mblk;  // which half of that size this block completes (the last one may be short)
      if (!(half & 1)) {
        if (last) continue;  // a first half without a second one: its inverse is complete
        if (side) {
          TB_CUDA_CHECK(cudaEventRecord(side->half_done, side->inv));
          TB_CUDA_CHECK(cudaStreamWaitEvent(side->inv2[level & 7], side->half_done, 0));
        }
        const int o = half * sblk, m2 = (dp - o - sblk < sblk) ? dp - o - sblk : sblk;
        cudaStream_t s1 = side ? side->inv2[level & 7] : inv_st;
        if (level_i8)
          TB_TRY(pair_first_i8(sblk, m2, o, high_tmp(sblk), s1));
        else
          TB_TRY(pair_first(sblk, m2, (long long)o * (dp + 1), pp, n_batch, high_tmp(sblk), (long long)f.tmp_per, s1));
        if (side) TB_CUDA_CHECK(cudaEventRecord(side->first_done[level & 7], side->inv2[level & 7]));
        break;
      }
      if (side) TB_CUDA_CHECK(cudaStreamWaitEvent(side->inv, side->first_done[level & 7], 0));
      const int o = (half - 1) * sblk, m2 = (dp - o - sblk < sblk) ? dp - o - sblk : sblk;
      if (level_i8)
        TB_TRY(pair_second_i8(sblk, m2, o, high_tmp(sblk), inv_st));
      else
        TB_TRY(pair_second(sblk, m2, (long long)o * (dp + 1), pp, n_batch, high_tmp(sblk), (long long)f.tmp_per, inv_st));
    }
    return TB_OK;
  };
  int next_inv_block = 0;

  // Two levels of blocking.  Outer blocks of OB = 256 columns (four panels).  Panel k applies the
  // update of panel k-1 to its own 64 columns itself; the rank-64 update after panel k covers the
  // columns from panel k+2 on up to ZL = 128 columns past the end of its outer block (a strip at most
  // 256 columns wide), so that the first two panels of the next block never wait for anything wide.
  // After a block's last panel its 256 columns update the columns up to ZL past the next block's end ("near": the
  // next block's third panel is the first to need it), and all columns finished so far update the OB columns
  // behind those ("far"), which the next block's near update will meet.  So every column is read and written
  // by one far update with a long contraction, not by one per block: rank-256 updates of the whole
  // trailing matrix moved it through memory once per block and spent half their time on that.
  // With the look-ahead: panels on the high-priority stream, the rank-64 strips and the near updates
  // in order on the trailing stream, the far updates on a low-priority stream beside the next block's
  // panels.  The far update of block J and the near update of block J+1 overlap in their columns, so
  // the latter waits for the former: every entry receives its updates in the same order as in the
  // single-stream schedule, and the results agree bit for bit.
  enum { OB = 4 * FNB, ZL = 2 * FNB };
  bool trail_set[2] = {false, false};
  bool strip_set = false, rest_set = false;
  auto rank_update = [&](int k_lo, int k_cnt, int c_lo, int c_hi, cudaStream_t stream_u) -> tb_status {
    // A[r][c] -= sum_k L[r][k_lo + k] L[c][k_lo + k] for c in [c_lo, c_hi), r >= c (tiles on or below the diagonal)
    if (c_hi <= c_lo) return TB_OK;
    if (f.use_i8 && k_cnt > FNB) {
      I8Gemm g = i8_gemm_params();
      g.A = g.B = f.digits;
      g.a_rb = g.b_rb = c_lo / I8_RB;
      g.a_rb_batch = g.b_rb_batch = rb;
      g.a_kb = g.b_kb = k_lo / I8_KB;
      g.k_blocks = k_cnt / I8_KB;
      g.a_exp = g.b_exp = 1;
      g.C = f.A + (long long)c_lo * (dp + 1);
      g.ldc = dp;
      g.c_batch = pp;
      g.M = d_fact - c_lo;
      g.N = c_hi - c_lo;
      g.n_batch = n_batch;
      g.alpha = -1.0;
      g.beta = 1.0;
      g.zeros = 4;
      g.tiles_per_cta = tile_life;
      return i8_gemm(g, stream_u);
    }
    GemmP t = gemm_params();
    t.A = f.A + (long long)c_lo * dp + k_lo;
    t.a_m = dp;
    t.a_k = 1;
    t.a_batch = pp;
    t.B = t.A;  // B(k, n) = L[c_lo + n][k_lo + k]
    t.b_k = 1;
    t.b_n = dp;
    t.b_batch = pp;
    t.C = f.A + (long long)c_lo * dp + c_lo;
    t.ldc = dp;
    t.c_batch = pp;
    t.M = d_fact - c_lo;
    t.N = c_hi - c_lo;
    t.K = k_cnt;
    t.n_batch = n_batch;
    t.alpha = -1.0;
    t.beta = 1.0;
    t.flags = GEMM_LOWER_TILES;
    return gemm64_launch<false>(t, stream_u);
  };
  // all finished columns [0, done) into the columns [c_lo, c_lo + OB), a piece of the contraction at a time: a piece's
  // tiles end soon enough for the panels of one matrix, of many matrices the products bound the time anyway
  auto far_update = [&](int done, int c_lo, cudaStream_t stream_u) -> tb_status {
    const int c_hi = (c_lo + OB < d_fact) ? c_lo + OB : d_fact;
    const int piece = (n_batch >= 4) ? 4096 : 1024;
    for (int k = 0; k < done; k += piece)
      TB_TRY(rank_update(k, (done - k < piece) ? done - k : piece, c_lo, c_hi, stream_u));
    return TB_OK;
  };
  for (int k0 = 0; k0 < d_fact; k0 += FNB) {
    const int r0 = k0 + FNB, m = d_fact - r0;
    const int xt = (m > 0) ? m / FNB : 1;
    const int pi = k0 / FNB;
    const int j0 = (k0 / OB) * OB;                               // first column of this outer block
    const int j1 = (j0 + OB < d_fact) ? j0 + OB : d_fact;        // one past its last column
    const bool last_in_block = (r0 >= j1);
    auto clip = [&](int c) { return c < d_fact ? c : d_fact; };
    if (side && trail_set[pi & 1]) TB_CUDA_CHECK(cudaStreamWaitEvent(cs, side->trail[pi & 1], 0));
    // a CTA per 64 rows while the SMs hold them, else several row blocks per CTA: the diagonal block is every CTA's work
    const int px = (xt * n_batch <= 148) ? xt : (148 / n_batch > 0 ? 148 / n_batch : 1);
    k_chol_panel<<<dim3(px < xt ? px : xt, n_batch), PANEL_THREADS, PANEL_SMEM, cs>>>(
        f.A, f.tmp, (long long)f.tmp_per, info, dp, k0, m / FNB, k0 > 0 ? 1 : 0, f.bad);
    TB_LAUNCH_CHECK();
    if (f.use_i8 && last_in_block) {  // digits of the outer block's columns, for the updates and the inverse
      I8Src l{f.A + (long long)j0 * (dp + 1), dp, pp, d_fact - j0, j1 - j0, n_batch, false, true, 0, nullptr, 0};
      TB_TRY(i8_slice(l, nullptr, dp, 1, f.digits, j0 / I8_RB, rb, j0 / I8_KB, cs, f.bad + j0));
    }
    if (side) {
      // blocks whose last factored panel this was (the identity padding needs no panel)
      bool waited = false;
      while (next_inv_block < n_inv_blocks) {
        int last = (next_inv_block + 1) * (G / FNB) - 1;
        if (last > n_panels - 1) last = n_panels - 1;
        if (last != pi) break;
        if (!waited) {
          TB_CUDA_CHECK(cudaEventRecord(side->block_done, cs));
          TB_CUDA_CHECK(cudaStreamWaitEvent(side->inv, side->block_done, 0));
          waited = true;
        }
        TB_TRY(invert_block(next_inv_block));
        ++next_inv_block;
      }
    }
    if (m <= 0) break;
    trail_set[pi & 1] = false;
    // rank-64 strip: the columns from panel k+2 on, up to ZL past the end of the outer block
    const int t_lo = clip(r0 + FNB), t_hi = clip(j1 + ZL);
    if (side && (t_hi > t_lo || last_in_block)) {
      TB_CUDA_CHECK(cudaEventRecord(side->panel, cs));
      TB_CUDA_CHECK(cudaStreamWaitEvent(side->stream, side->panel, 0));
    }
    if (t_hi > t_lo) {
      TB_TRY(rank_update(k0, FNB, t_lo, t_hi, side ? side->stream : st));
      if (side) {
        TB_CUDA_CHECK(cudaEventRecord(side->trail[pi & 1], side->stream));
        trail_set[pi & 1] = true;
      }
    }
    if (!last_in_block) continue;
    // the block is factored: rank-(j1 - j0) update of everything further right
    const int n_lo = clip(j1 + ZL), n_hi = clip(j1 + OB + ZL);
    if (!side) {
      TB_TRY(rank_update(j0, j1 - j0, n_lo, n_hi, st));
      TB_TRY(far_update(j1, n_hi, st));
      continue;
    }
    if (n_hi > n_lo) {
      // near: overlaps the previous block's far update in these columns, so after it
      if (rest_set) TB_CUDA_CHECK(cudaStreamWaitEvent(side->stream, side->rest_done, 0));
      TB_TRY(rank_update(j0, j1 - j0, n_lo, n_hi, side->stream));
      // later strips of this stream follow it in order; the panels that need it wait for those strips
      TB_CUDA_CHECK(cudaEventRecord(side->strip_done, side->stream));
      strip_set = true;
    }
    if (n_hi < d_fact) {
      TB_CUDA_CHECK(cudaStreamWaitEvent(side->rest, side->panel, 0));
      TB_TRY(far_update(j1, n_hi, side->rest));
      TB_CUDA_CHECK(cudaEventRecord(side->rest_done, side->rest));
      rest_set = true;
    }
  }
  if (side) {
    for (int i = 0; i < 2; ++i)
      if (trail_set[i]) TB_CUDA_CHECK(cudaStreamWaitEvent(st, side->trail[i], 0));
    if (strip_set) TB_CUDA_CHECK(cudaStreamWaitEvent(st, side->strip_done, 0));
    if (rest_set) TB_CUDA_CHECK(cudaStreamWaitEvent(st, side->rest_done, 0));
    TB_CUDA_CHECK(cudaEventRecord(side->crit_done, side->crit));
    TB_CUDA_CHECK(cudaStreamWaitEvent(st, side->crit_done, 0));
  }

  // what is left of the inverse (all of it without the look-ahead)
  while (next_inv_block < n_inv_blocks) {
    TB_TRY(invert_block(next_inv_block));
    ++next_inv_block;
  }
  if (side) {
    TB_CUDA_CHECK(cudaEventRecord(side->inv_done, side->inv));
    TB_CUDA_CHECK(cudaStreamWaitEvent(st, side->inv_done, 0));
  }
  k_reverse_out<<<dim3((d + 255) / 256, (d + 7) / 8, n_batch), 256, 0, st>>>(f.A, f.exps, U, d, dp, Hinv ? 1 : 0);
  TB_LAUNCH_CHECK();

  if (Hinv) {
    // Hinv = U^T U with U(k, m) = Li[d-1-k][d-1-m]: negative strides from element (d-1, d-1)
    GemmP g = gemm_params();
    const double* last = f.A + (long long)(d - 1) * dp + (d - 1);
    g.A = last;  // A(m, k) = U[k][m]
    g.a_m = -1;
    g.a_k = -(long long)dp;
    g.a_batch = pp;
    g.B = last;  // B(k, n) = U[k][n]
    g.b_k = -(long long)dp;
    g.b_n = -1;
    g.b_batch = pp;
    g.C = Hinv;
    g.ldc = d;
    g.c_batch = (long long)d * d;
    g.M = d;
    g.N = d;
    g.K = d;
    g.n_batch = n_batch;
    g.btrim = 1;  // U(k, n) = 0 for k > n
    g.atrim = 1;  // U(k, m) = 0 for k > m
    TB_TRY((gemm_launch<double, double, float, double, true, true>(g, st)));
  }
  return TB_OK;
}

// P and C: T1 = R U^T, C = T1 U, P = (strictly upper part of T1) U, three double-precision products on the integer
// tensor cores (tb_i8.cuh).  R U^T U cancels heavily at large widths (a split-bf16 version, good to a few 1e-7 of
// sum |a||b|, missed by 1.5e-5 of the result at 4096 columns); these products are as good as the FP64 pipe's.  The
// contraction of R U^T runs over columns whose scales R and U have in opposite directions: the exponents of U's
// diagonal take them out.  4096 columns: 6.8 ms on the FP64 pipe, 1.85 ms now.
struct PrepWs {
  double* T1;
  int* exps;
  unsigned long long *ma, *mb;
  I8Mat A, B;
  size_t total;
};
static PrepWs prep_ws(int d, void* ws) {
  PrepWs w;
  Bump b(ws);
  w.T1 = b.take<double>((size_t)d * d);
  w.exps = b.take<int>((size_t)d);
  w.ma = b.take<unsigned long long>((size_t)d);
  w.mb = b.take<unsigned long long>((size_t)d);
  w.A.row_blocks = w.B.row_blocks = (d + I8_RB - 1) / I8_RB;
  w.A.k_blocks = w.B.k_blocks = (d + I8_KB - 1) / I8_KB;
  w.A.data = b.take<unsigned char>(i8_bytes(w.A.row_blocks, w.A.k_blocks));
  w.B.data = b.take<unsigned char>(i8_bytes(w.B.row_blocks, w.B.k_blocks));
  w.total = b.total();
  return w;
}

extern "C" size_t tb_prepare_correction_workspace(int n_batch, int d) {
  if (n_batch <= 0 || d <= 0) return 0;
  return prep_ws(d, nullptr).total;
}

extern "C" tb_status tb_prepare_correction(const float* R, const float* U_in, int n_batch, int d,
                                           float* P, float* C, void* ws, size_t ws_bytes,
                                           void* stream) {
  if (!R || !U_in || !P || !C || n_batch <= 0 || d <= 0) return TB_ERR_INVALID_ARG;
  if (!ws || !aligned(ws, 256) || ws_bytes < tb_prepare_correction_workspace(n_batch, d))
    return TB_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  PrepWs w = prep_ws(d, ws);
  const long long dd = (long long)d * d;
  // what the vector accesses of the digit kernels need; other widths and pointers take the strided engine
  const bool digits = d % 4 == 0 && d <= 16384 && aligned(R, 16) && aligned(U_in, 16) && aligned(P, 16) && aligned(C, 16);
  for (int i = 0; i < n_batch; ++i) {
    const float* Rb = R + i * dd;
    const float* Ub = U_in + i * dd;
    if (digits) {
      TB_TRY(i8_diag_exp(Ub, w.exps, d, st));
      const I8Src r{Rb, d, 0, d, d, 1, true, true, 0, w.exps, 1};
      const I8Src ut{Ub, d, 0, d, d, 1, true, true, 2, w.exps, -1};  // row n of the operand: U[n][k], zero for k < n
      TB_TRY(i8_row_max(r, w.ma, d, st));
      TB_TRY(i8_row_max(ut, w.mb, d, st));
      TB_TRY(i8_slice(r, w.ma, d, 0, w.A, 0, 0, 0, st));
      TB_TRY(i8_slice(ut, w.mb, d, 0, w.B, 0, 0, 0, st));
      I8Gemm g = i8_gemm_params();
      g.A = w.A;
      g.B = w.B;
      g.k_blocks = w.A.k_blocks;
      g.a_max = w.ma;
      g.b_max = w.mb;
      g.C = w.T1;
      g.ldc = d;
      g.M = g.N = d;
      g.zeros = 2;
      g.order = 1;
      TB_TRY(i8_gemm(g, st));
      const I8Src u{Ub, d, 0, d, d, 1, true, false, 1, nullptr, 0};  // row n of the operand: U[k][n], zero for k > n
      TB_TRY(i8_row_max(u, w.mb, d, st));
      TB_TRY(i8_slice(u, w.mb, d, 0, w.B, 0, 0, 0, st));
      for (int upper = 0; upper < 2; ++upper) {
        const I8Src t{w.T1, d, 0, d, d, 1, false, true, upper ? 3 : 0, nullptr, 0};
        TB_TRY(i8_row_max(t, w.ma, d, st));
        TB_TRY(i8_slice(t, w.ma, d, 0, w.A, 0, 0, 0, st));
        g.C = nullptr;
        g.Cf = (upper ? P : C) + i * dd;
        g.zeros = upper ? 8 + 16 : 8;
        g.order = 0;
        TB_TRY(i8_gemm(g, st));
      }
      continue;
    }
    GemmP g = gemm_params();  // T1 = R U^T
    g.A = Rb;
    g.a_m = d;
    g.a_k = 1;
    g.B = Ub;  // B(k, n) = U[n][k], zero for k < n
    g.b_k = 1;
    g.b_n = d;
    g.C = w.T1;
    g.ldc = d;
    g.M = d;
    g.N = d;
    g.K = d;
    g.btrim = 2;
    TB_TRY((gemm_launch<float, float, double, double, false, false>(g, st)));
    GemmP c = gemm_params();  // C = T1 U
    c.A = w.T1;
    c.a_m = d;
    c.a_k = 1;
    c.B = Ub;  // B(k, n) = U[k][n], zero for k > n
    c.b_k = d;
    c.b_n = 1;
    c.C = C + i * dd;
    c.ldc = d;
    c.M = d;
    c.N = d;
    c.K = d;
    c.btrim = 1;
    TB_TRY((gemm_launch<double, float, float, double, false, true>(c, st)));
    double* T2 = reinterpret_cast<double*>(w.A.data);  // 2 x 7 bytes per entry: room for a double
    const int eb = (int)((dd + 255) / 256 < 148 * 8 ? (dd + 255) / 256 : 148 * 8);
    k_mask_strict_upper<<<eb, 256, 0, st>>>(w.T1, T2, d);
    TB_LAUNCH_CHECK();
    GemmP p = c;  // P = (strictly upper part of T1) U
    p.A = T2;
    p.C = P + i * dd;
    p.atrim = 2;  // T2(m, k) = 0 for k < m + 1
    p.aoff = 1;
    TB_TRY((gemm_launch<double, float, float, double, false, true>(p, st)));
  }
  return TB_OK;
}
