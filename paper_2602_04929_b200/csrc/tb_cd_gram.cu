// Coordinate descent on the scales (Proposition 3.3 / Algorithm 3) of heads with few coordinates, as a triangular solve.
//
// A step delta_a on coordinate a = (row j, group g2) of a head changes the numerator of coordinate b = (row i, group g) by
//   delta_a K[a][b],   K[a][b] = H_out[i][j] W_j,g2 H_in[G_g2, G_g] W_i,g^T      (W = W_int - z),
// so a Gauss-Seidel pass in order (rows ascending, groups inside a row) is a forward substitution with the head's matrix
// K.  The pass that walks the rows with a vector of d_in columns per row (k_cd_head_cols) costs 6 us a row whatever the number
// of groups; K costs n d_head d_in multiply-adds to form (n = d_head n_groups coordinates) and the solve reads it once:
//   k_cd_gram    K, one group of columns b at a time, FP64 tensor steps from Yw = W H_in blockwise
//   k_cd_start   numerators before the pass, n0[g][i] = W_i,g . (H_out Dm)_i,g
//   k_cd_solve   one CTA per head, 32 coordinates at a time: their chain in one warp, then the rest of the vector
//   k_cd_apply   Dm_j += sum_g2 delta Yw[j][g2], and the scales
// The whole refinement, one pass, walking the rows and here: 8 heads x 128 rows x 1024 columns, one scale per row 0.64 and
// 0.25 ms; 8 x 512 rows, 4 groups of 256 columns 3.90 and 1.90 ms.  The solve costs 10 us per 32 coordinates at 1024 of
// them (reading K), and so with many groups a row the walk is the better one (cd_gram_pays).
#include "tb_gemm.cuh"
#include "tb_rows.cuh"

namespace tb {

// K[a][g dh + i] for i >= j(a) (other entries are not read).  CTA: 64 coordinates a x 64 rows i of one group g.
template <typename TY>
__global__ void __launch_bounds__(256) k_cd_gram(const TY* __restrict__ Yw, const float* __restrict__ Wb,
                                                 const float* __restrict__ Hout, double* __restrict__ K, int d, int seg,
                                                 int ng, int dh) {
  constexpr int KC = 32, LD = KC + 4;
  __shared__ double As[64][LD], Bs[64][LD];
  const int n = dh * ng, tiles_i = (dh + 63) / 64, tiles_a = (n + 63) / 64;
  const int head = blockIdx.z, g = blockIdx.y, a0 = (blockIdx.x % tiles_a) * 64, i0 = (blockIdx.x / tiles_a) * 64;
  if (i0 + 63 < a0 / ng) return;  // all rows i before the first row j
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, fr = lane >> 2, fk = lane & 3;
  const TY* Y = Yw + (long long)head * n * d + (long long)g * seg;
  const float* W = Wb + (long long)head * dh * d + (long long)g * seg;
  double acc[8][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0.0;
  for (int c0 = 0; c0 < seg; c0 += KC) {  // seg is a multiple of 32
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int r = warp * 8 + q;
      As[r][lane] = (a0 + r < n) ? (double)Y[(long long)(a0 + r) * d + c0 + lane] : 0.0;
      Bs[r][lane] = (i0 + r < dh) ? (double)W[(long long)(i0 + r) * d + c0 + lane] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < KC / 4; ++q) {
      const double av = As[8 * warp + fr][4 * q + fk];
#pragma unroll
      for (int t = 0; t < 8; ++t)
        dmma(acc[t], av, Bs[8 * t + fr][4 * q + fk]);
    }
    __syncthreads();
  }
  const int a = a0 + 8 * warp + fr, j = a / ng;
  if (a >= n) return;
  const float* H = Hout + (long long)head * dh * dh;
  double* Ka = K + ((long long)head * n + a) * n + (long long)g * dh;
#pragma unroll
  for (int t = 0; t < 8; ++t)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int i = i0 + 8 * t + 2 * fk + e;
      if (i < dh) Ka[i] = acc[t][e] * (double)H[(long long)i * dh + j];
    }
}

// n0[head][g dh + i] = sum over the group of Wb[i] G[i]; a warp per (row, group)
__global__ void __launch_bounds__(256) k_cd_start(const double* __restrict__ G, const float* __restrict__ Wb,
                                                  double* __restrict__ n0, long long lines, int d, int seg, int ng, int dh) {
  const long long line = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (line >= lines) return;
  const long long row = line / ng;
  const int g = (int)(line % ng);
  const double* gr = G + row * d + (long long)g * seg;
  const float* w = Wb + row * d + (long long)g * seg;
  double v = 0.0;
#pragma unroll 4
  for (int c = lane; c < seg; c += 32) v = fma((double)w[c], gr[c], v);
  v = warp_sum(v);
  if (lane == 0) n0[(row / dh) * (long long)dh * ng + (long long)g * dh + row % dh] = v;
}

// delta[head][a], a = j ng + g.  The numerators stay in shared memory, [g][i].  Block k of 32 coordinates: warp 0 walks its
// chain and applies it to block k + 1 alone, while the other warps apply block k to everything behind; the
// two 32 x 32 parts of K that warp 0 needs next are copied ahead.
__global__ void __launch_bounds__(512) k_cd_solve(const double* __restrict__ K, const double* __restrict__ n0,
                                                  double* __restrict__ delta, int ng, int dh) {
  extern __shared__ double cs_num[];  // [n]
  __shared__ double Kd[2][32][33], Kx[2][32][33], dl[2][32];
  const int n = dh * ng, head = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* Kh = K + (long long)head * n * n;
  for (int i = tid; i < n; i += 512) cs_num[i] = n0[(long long)head * n + i];
  auto place = [&](int a) { return (a % ng) * dh + a / ng; };
  // block starting at a0: its triangle and its effect on the next block (zero outside the matrix)
  auto copy_ahead = [&](int a0, int buf, int w, int nw) {
    const int c = lane;
    const int pd = (a0 + c < n) ? place(a0 + c) : -1, px = (a0 + 32 + c < n) ? place(a0 + 32 + c) : -1;
    for (int r = w; r < 32; r += nw) {
      const long long row = (long long)(a0 + r) * n;
      const bool in = a0 + r < n;
      double vd = 0.0, vx = 0.0;
      if (in && pd >= 0 && c >= r) vd = Kh[row + pd];
      if (in && px >= 0) vx = Kh[row + px];
      Kd[buf][r][c] = vd;
      Kx[buf][r][c] = vx;
    }
  };
  copy_ahead(0, 0, warp, 16);
  __syncthreads();
  for (int a0 = 0, k = 0; a0 < n; a0 += 32, ++k) {
    const int buf = k & 1, cnt = min(32, n - a0);
    if (warp == 0) {
      // lane c holds the numerator of coordinate a0 + c: -n_r / K_rr carried through one shuffle and one multiply-add
      double nm = (lane < cnt) ? cs_num[place(a0 + lane)] : 0.0;
      const double den = Kd[buf][lane][lane], rinv = (den == 0.0) ? 0.0 : 1.0 / den;
      double mine = 0.0;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const double f = -__shfl_sync(0xffffffffu, rinv, r) * Kd[buf][r][lane];
        const double nr = __shfl_sync(0xffffffffu, nm, r);
        if (lane == r) mine = -nr * rinv;
        if (lane > r) nm = fma(nr, f, nm);
      }
      dl[buf][lane] = (lane < cnt) ? mine : 0.0;
      if (lane < cnt) delta[(long long)head * n + a0 + lane] = mine;
    }
    __syncthreads();  // also: block k - 1 has been applied to everything
    if (a0 + 32 >= n) break;
    if (warp == 0) {
      if (a0 + 32 + lane < n) {
        const int b = place(a0 + 32 + lane);
        double v = cs_num[b], v1 = 0.0;
#pragma unroll
        for (int r = 0; r < 32; r += 2) {
          v = fma(dl[buf][r], Kx[buf][r][lane], v);
          v1 = fma(dl[buf][r + 1], Kx[buf][r + 1][lane], v1);
        }
        cs_num[b] = v + v1;
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");  // the next block's copies have landed
    } else {
      copy_ahead(a0 + 32, buf ^ 1, warp - 1, 15);
      asm volatile("bar.arrive 1, 512;" ::: "memory");
      // coordinates behind the next block: all rows beyond the one it ends in, and the rest of that row
      const int first = a0 + 64, i_min = first / ng, left = dh - i_min;
      for (int t = tid - 32; t < left * ng; t += 480) {
        const int g = t / left, i = i_min + t % left;
        if (i * ng + g < first) continue;  // (part of the next block)
        const int b = g * dh + i;
        double v = cs_num[b], v1 = 0.0;
        const double* kc = Kh + (long long)a0 * n + b;
#pragma unroll
        for (int r = 0; r < 32; r += 2) {  // a full block: another one follows it
          v = fma(dl[buf][r], __ldg(kc + (long long)r * n), v);
          v1 = fma(dl[buf][r + 1], __ldg(kc + (long long)(r + 1) * n), v1);
        }
        cs_num[b] = v + v1;
      }
    }
  }
}

// Dm_j += sum_g2 delta[j][g2] Yw[j][g2][:] and s += delta.  A CTA per row (along x, which holds any
// number of them) and 1024 columns.
template <typename TY>
__global__ void __launch_bounds__(256) k_cd_apply(double* __restrict__ Dm, const TY* __restrict__ Yw,
                                                  const double* __restrict__ delta, double* __restrict__ sD, int d, int ng) {
  const long long row = blockIdx.x;
  const double* dr = delta + row * ng;  // [head][j ng + g] is [row][g]
  if (blockIdx.y == 0)
    for (int g = threadIdx.x; g < ng; g += 256) sD[row * ng + g] += dr[g];
  const TY* y = Yw + row * ng * d;
  for (int c = blockIdx.y * 1024 + threadIdx.x; c < min(d, (int)(blockIdx.y + 1) * 1024); c += 256) {
    double v = Dm[row * d + c];
#pragma unroll 8
    for (int g = 0; g < ng; ++g) v = fma(dr[g], (double)y[(long long)g * d + c], v);
    Dm[row * d + c] = v;
  }
}

// Measured, walk / triangular solve, one pass, in us.  Up to 4 groups the solve is ahead wherever it fits: 2048 coordinates
// as 512 rows x 4 groups of 512 columns 3746 / 1031 (1 head), 4641 / 2697 (8), 7768 / 6927 (32); with 64 heads of 256 rows x 4
// groups of 256 2632 / 2268, with 128 they meet.  5 to 7 groups do not divide over the walk's cluster of 4 or 8 CTAs: 128 rows x
// 5 groups of 256 1489 / 342 (8 heads), 1959 / 814 (32), 3096 / 2323 (128).  8 groups do, and reading the heads' matrices
// decides, which grows with their number: 128 rows x 8 groups of 128, 642 / 400 (4 heads), 672 / 530 (8), 1260 / 729 (16),
// 920 / 1043 (32), 1326 / 1656 (64); 64 rows, 586 / 291 (16), 455 / 459 (32), 644 / 732 (64).  With 16 groups it is behind at 8
// heads: 64 rows, 451 / 627.
bool cd_gram_pays(int heads, int dh, int ng) {
  const long long n = (long long)dh * ng;
  return (ng <= 4 && n <= CD_GRAM_MAX) || (ng <= 8 && n <= 1024 && (ng < 8 || heads * n <= 16384));
}

size_t cd_gram_doubles(int heads, int dh, int ng) {  // K, n0, delta
  const size_t n = (size_t)dh * ng;
  return (size_t)heads * (n * n + 2 * n);
}

template <typename TY>
static tb_status gram_form(const CdGram& p, cudaStream_t st) {
  const int n = p.dh * p.ng;
  const dim3 grid(((n + 63) / 64) * ((p.dh + 63) / 64), p.ng, p.heads);
  k_cd_gram<TY><<<grid, 256, 0, st>>>(static_cast<const TY*>(p.Yw), p.Wb, p.Hout, p.scratch, p.d, p.seg, p.ng, p.dh);
  TB_LAUNCH_CHECK();
  return TB_OK;
}
tb_status cd_gram_form(const CdGram& p, cudaStream_t st) {
  return p.yw_float ? gram_form<float>(p, st) : gram_form<double>(p, st);
}

// one pass; G = H_out Dm on entry
tb_status cd_gram_pass(const CdGram& p, const double* G, double* Dm, double* sD, cudaStream_t st) {
  const long long n = (long long)p.dh * p.ng, rows = (long long)p.heads * p.dh;
  double* n0 = p.scratch + p.heads * n * n;
  double* delta = n0 + p.heads * n;
  k_cd_start<<<(unsigned)((rows * p.ng + 7) / 8), 256, 0, st>>>(G, p.Wb, n0, rows * p.ng, p.d, p.seg, p.ng, p.dh);
  TB_LAUNCH_CHECK();
  static bool configured[64] = {false};
  TB_TRY(allow_smem(k_cd_solve, CD_GRAM_MAX * sizeof(double), configured));
  k_cd_solve<<<p.heads, 512, (size_t)n * sizeof(double), st>>>(p.scratch, n0, delta, p.ng, p.dh);
  TB_LAUNCH_CHECK();
  const dim3 grid((unsigned)rows, (p.d + 1023) / 1024);
  if (p.yw_float)
    k_cd_apply<float><<<grid, 256, 0, st>>>(Dm, static_cast<const float*>(p.Yw), delta, sD, p.d, p.ng);
  else
    k_cd_apply<double><<<grid, 256, 0, st>>>(Dm, static_cast<const double*>(p.Yw), delta, sD, p.d, p.ng);
  TB_LAUNCH_CHECK();
  return TB_OK;
}

}  // namespace tb
