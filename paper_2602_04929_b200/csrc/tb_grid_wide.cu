// Grid search for column groups wider than 128 columns (one scale per row, or groups of 256 and more), few rows (with
// many rows: tb_grid_digits.cu).
//
// For every (row, group): n_cand clipped min-max grids, p_k = 1 - k/32, score e H_in[G,G] e^T with e the
// round-to-nearest error on that grid, lowest score wins, lowest k on ties.  H_in[G,G] is symmetric, so
// e H e^T = 2 e T e^T with T its upper triangle (diagonal halved); the factor 2 is dropped, scores are only
// compared.  Three launches:
//   k_row_range    minimum and maximum of every (row, group)
//   k_grid_score   partial scores: a CTA takes a tile of candidate rows (rows x candidates) and a tile of
//                  columns, forms E T for its columns (contraction over the rows of T from the group's first
//                  one to the tile's last) and the row dots with E
//   k_grid_pick    adds the partial scores of a group in column order, takes the lowest
// The work is FP64 tensor steps (half of d_group^2 per candidate row); what a step of few rows lacks is
// CTAs, hence the column split, and tiles of 32 x 32 instead of 128 x 128 while the large ones would not
// fill the SMs (0.49 of the FP64 rate with large ones).  32 searches of 8 rows x 256 columns, against one CTA that walks
// all columns of its rows with the full product: 3.44 ms before, 0.67 ms now.
#include "tb_gemm.cuh"
#include "tb_grid.cuh"
#include "tb_rows.cuh"

namespace tb {

enum { GW_KC = 64 };  // contraction rows per chunk

template <int CR>
struct GwSmem {  // CR candidate rows x CR columns
  static constexpr int LDE = CR + 4, LDT = CR + 8;
  double E[GW_KC][LDE];
  float T[2][GW_KC][LDT];
  double s[CR], rs[CR], z[CR];
  double part[8][CR];
  long long src[CR];  // element offset of the candidate's row in W~, or -1
};

__global__ void __launch_bounds__(256) k_row_range(GridP p, int m0, double2* range) {
  __shared__ double smn[8], smx[8];
  pdl_wait();
  const int m = m0 + blockIdx.y, grp = blockIdx.x;
  const double* w = p.Wt + p.rm.row(m) * p.d + (long long)grp * p.seg;
  double mn = 0.0, mx = 0.0;
  for (int a = threadIdx.x; a < p.seg; a += 256) {
    const double v = w[a];
    mn = fmin(mn, v);
    mx = fmax(mx, v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  pdl_trigger();
  if ((threadIdx.x & 31) == 0) {
    smn[threadIdx.x >> 5] = mn;
    smx[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) {
      mn = fmin(mn, smn[i]);
      mx = fmax(mx, smx[i]);
    }
    range[(long long)blockIdx.y * p.ng + grp] = make_double2(mn, mx);
  }
}

// Candidate rows: row m of the chunk and candidate k at m * ncp + k; tiles never cross units (rows of one H_in).
// CR = 128: 16 warps of 32 x 32; CR = 32: 8 warps, four of 16 x 16 times two halves of every chunk.
template <int CR>
__global__ void __launch_bounds__(CR == 128 ? 512 : 256, 1)
    k_grid_score(GridP p, int m0, int unit_rows, int tiles_per_unit, int col_tiles, const double2* range, double* partial) {
  extern __shared__ __align__(16) unsigned char gw_raw[];
  using Smem = GwSmem<CR>;
  constexpr int THREADS = (CR == 128) ? 512 : 256;
  constexpr int NF = (CR == 128) ? 4 : 2;   // 8 x 8 fragments per warp and direction
  constexpr int KSPLIT = (CR == 128) ? 1 : 2;
  constexpr int WPR = (CR == 128) ? 4 : 2;  // warps along a direction
  Smem& sm = *reinterpret_cast<Smem*>(gw_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int fr = lane >> 2, fk = lane & 3;
  const int kh = (KSPLIT == 2) ? warp >> 2 : 0;
  const int wr = (warp % (WPR * WPR)) / WPR, wc = warp % WPR;
  // the last column tiles have the longest contraction: they start first
  const int grp = blockIdx.x / col_tiles, ct = col_tiles - 1 - blockIdx.x % col_tiles;
  const int unit = blockIdx.y / tiles_per_unit, tile = blockIdx.y % tiles_per_unit;
  const int rt = CR / p.ncp;
  const int seg = p.seg, d = p.d;
  const long long seg0 = (long long)grp * seg;
  const int n0 = ct * CR, k_end = min(seg, n0 + CR);
  const float* H = p.Hin + ((p.units > 1) ? (long long)(p.rm.row(m0 + unit * unit_rows) / p.rm.d_head) * d * d : 0);

  pdl_wait();
  if (tid < CR) {
    const int r = tile * rt + tid / p.ncp, k = tid % p.ncp;
    const bool valid = r < unit_rows && k < p.n_cand;
    double s = 1.0, z = 0.0;
    long long src = -1;
    if (valid) {
      const int m = unit * unit_rows + r;
      gw_candidate(range[(long long)m * p.ng + grp], k, p.maxq, &s, &z);
      src = p.rm.row(m0 + m) * d + seg0;
    }
    sm.s[tid] = s;
    sm.rs[tid] = 1.0 / s;
    sm.z[tid] = z;
    sm.src[tid] = src;
  }
  // T chunk: rows k0 .. +63, columns n0 .. +CR-1 of the upper triangle (diagonal halved)
  constexpr int TPT = GW_KC * CR / 4 / THREADS;  // float4 per thread
  float4 tv[TPT];
  auto fetch_t = [&](int k0) {
#pragma unroll
    for (int i = 0; i < TPT; ++i) {
      const int idx = tid + i * THREADS, kk = idx / (CR / 4), c4 = (idx % (CR / 4)) * 4;
      tv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k0 + kk < k_end && n0 + c4 < seg)  // groups are multiples of 32 columns
        tv[i] = *reinterpret_cast<const float4*>(H + (seg0 + k0 + kk) * d + seg0 + n0 + c4);
    }
  };
  auto store_t = [&](int k0, int buf) {
#pragma unroll
    for (int i = 0; i < TPT; ++i) {
      const int idx = tid + i * THREADS, kk = idx / (CR / 4), c4 = (idx % (CR / 4)) * 4;
      const int k = k0 + kk;
      float v[4] = {tv[i].x, tv[i].y, tv[i].z, tv[i].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int n = n0 + c4 + e;
        v[e] = (k > n) ? 0.0f : (k == n) ? 0.5f * v[e] : v[e];
      }
      *reinterpret_cast<float4*>(&sm.T[buf][kk][c4]) = make_float4(v[0], v[1], v[2], v[3]);
    }
  };
  // E chunk: thread = (candidate row, every THREADS / CR -th k)
  constexpr int EPT = GW_KC * CR / THREADS, ESTEP = THREADS / CR;
  const int e_cr = tid % CR, e_k = tid / CR;
  fetch_t(0);
  __syncthreads();
  const double es = sm.s[e_cr], ers = sm.rs[e_cr], ez = sm.z[e_cr];
  const long long e_src = sm.src[e_cr];
  double acc[NF][NF][2];
#pragma unroll
  for (int i = 0; i < NF * NF * 2; ++i) (&acc[0][0][0])[i] = 0.0;
  int buf = 0;
  for (int k0 = 0; k0 < k_end; k0 += GW_KC, buf ^= 1) {
    store_t(k0, buf);
#pragma unroll 8
    for (int i = 0; i < EPT; ++i) {
      const int kk = e_k + i * ESTEP;
      double e = 0.0;
      if (e_src >= 0 && k0 + kk < k_end) e = gw_error(p.Wt[e_src + k0 + kk], es, ers, ez, p.maxq);
      sm.E[kk][e_cr] = e;
    }
    __syncthreads();
    if (k0 + GW_KC < k_end) fetch_t(k0 + GW_KC);
    const double* ap = &sm.E[fk][wr * NF * 8 + fr];
    const float* bp = &sm.T[buf][fk][wc * NF * 8 + fr];
#pragma unroll 4
    for (int q = kh; q < GW_KC / 4; q += KSPLIT) {
      double a[NF], b[NF];
#pragma unroll
      for (int i = 0; i < NF; ++i) a[i] = ap[q * 4 * Smem::LDE + 8 * i];
#pragma unroll
      for (int j = 0; j < NF; ++j) b[j] = (double)bp[q * 4 * Smem::LDT + 8 * j];
#pragma unroll
      for (int i = 0; i < NF; ++i)
#pragma unroll
        for (int j = 0; j < NF; ++j)
          dmma(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
  pdl_trigger();
  // row dots of (E T) with E: quads by shuffle, warps through shared memory in a fixed order
#pragma unroll
  for (int i = 0; i < NF; ++i) {
    const int cr = wr * NF * 8 + i * 8 + fr;
    const long long src = sm.src[cr];
    double v = 0.0;
    if (src >= 0) {
#pragma unroll
      for (int j = 0; j < NF; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int n = n0 + wc * NF * 8 + j * 8 + 2 * fk + e;
          if (n < seg) v = fma(acc[i][j][e], gw_error(p.Wt[src + n], sm.s[cr], sm.rs[cr], sm.z[cr], p.maxq), v);
        }
    }
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (fk == 0) sm.part[kh * WPR + wc][cr] = v;
  }
  __syncthreads();
  if (tid < CR && sm.src[tid] >= 0) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < KSPLIT * WPR; ++i) t += sm.part[i][tid];
    const long long m = unit * unit_rows + tile * rt + tid / p.ncp;
    partial[((m * p.ng + grp) * col_tiles + ct) * p.ncp + tid % p.ncp] = t;
  }
}

// one warp per (row, group), one lane per candidate; strict '<' and the lower k on ties
__global__ void __launch_bounds__(256) k_grid_pick(GridP p, int m0, long long lines, int col_tiles,
                                                   const double2* range, const double* partial) {
  const long long line = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  pdl_wait();
  pdl_trigger();
  if (line >= lines) return;
  double t = 0.0;
  if (lane < p.n_cand)
    for (int c = 0; c < col_tiles; ++c) t += partial[(line * col_tiles + c) * p.ncp + lane];
  // a candidate that scores no number never beats another one, and candidate 0 is only beaten by '<'
  if (t != t) t = (lane == 0) ? -INFINITY : INFINITY;
  if (lane >= p.n_cand) t = INFINITY;
  int best = lane;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ot = __shfl_xor_sync(0xffffffffu, t, o);
    const int ob = __shfl_xor_sync(0xffffffffu, best, o);
    if (ot < t || (ot == t && ob < best)) {
      t = ot;
      best = ob;
    }
  }
  if (lane == 0) {
    double s, z;
    gw_candidate(range[line], best, p.maxq, &s, &z);
    const long long o = p.rm.row(m0 + (int)(line / p.ng)) * p.ng + line % p.ng;
    p.sD[o] = s;
    p.s_out[o] = (float)s;
    p.z_out[o] = (int)z;
    if (p.cand_out) p.cand_out[o] = (unsigned char)best;
  }
}

// a row's ranges (2 ng doubles) and partial scores (ncp per column tile; the narrow tiles are the most)
size_t grid_wide_row_doubles(int d, int ng, int ncp) {
  return (size_t)2 * ng + (size_t)ng * ((d / ng + 31) / 32) * ncp;
}

tb_status grid_wide(const GridP& p, double* scratch, size_t scratch_doubles, cudaStream_t st) {
  const size_t per_row = grid_wide_row_doubles(p.d, p.ng, p.ncp);
  static bool conf128[64] = {false}, conf32[64] = {false};
  TB_TRY(allow_smem(k_grid_score<128>, sizeof(GwSmem<128>), conf128));
  TB_TRY(allow_smem(k_grid_score<32>, sizeof(GwSmem<32>), conf32));
  // chunks of rows whose scratch fits: whole units when every head has its own H_in, else a part of a unit
  long long fit = (long long)(scratch_doubles / per_row);
  if (fit > 32768) fit = 32768;  // rows are a grid dimension of k_row_range
  if (fit < 1) return TB_ERR_WORKSPACE;
  for (int u0 = 0; u0 < p.M;) {
    // rows u0 .. u0 + cnt - 1, all units of `rows` rows
    int cnt, rows;
    const int in_unit = u0 % p.rows_per_unit;
    if (in_unit == 0 && fit >= p.rows_per_unit) {
      long long units = fit / p.rows_per_unit, left = (p.M - u0) / p.rows_per_unit;
      if (units > left) units = left;
      cnt = (int)(units * p.rows_per_unit);
      rows = p.rows_per_unit;
    } else {
      const int left = p.rows_per_unit - in_unit;
      cnt = rows = (fit < left) ? (int)fit : left;
    }
    double2* range = reinterpret_cast<double2*>(scratch);
    double* partial = scratch + (size_t)2 * cnt * p.ng;
    const int units = cnt / rows;
    TB_CUDA_CHECK(launch_pdl(k_row_range, dim3(p.ng, cnt), dim3(256), 0, st, p, u0, range));
    TB_LAUNCH_CHECK();
    // 128 x 128 tiles when they fill the SMs, else 32 x 32
    const int rt128 = 128 / p.ncp, rt32 = 32 / p.ncp;
    const long long t128 = (long long)units * ((rows + rt128 - 1) / rt128), c128 = (p.seg + 127) / 128;
    const bool small = t128 * c128 * p.ng < 148;
    const int rt = small ? rt32 : rt128, col_tiles = small ? (p.seg + 31) / 32 : (int)c128;
    const int tiles = (rows + rt - 1) / rt;
    if ((long long)units * tiles > 65535) return TB_ERR_UNSUPPORTED;
    const dim3 grid((unsigned)(p.ng * col_tiles), (unsigned)(units * tiles));
    if (small)
      TB_CUDA_CHECK(launch_pdl(k_grid_score<32>, grid, dim3(256), sizeof(GwSmem<32>), st, p, u0, rows, tiles, col_tiles, range, partial));
    else
      TB_CUDA_CHECK(launch_pdl(k_grid_score<128>, grid, dim3(512), sizeof(GwSmem<128>), st, p, u0, rows, tiles, col_tiles, range, partial));
    TB_LAUNCH_CHECK();
    const long long lines = (long long)cnt * p.ng;
    TB_CUDA_CHECK(launch_pdl(k_grid_pick, dim3((unsigned)((lines + 7) / 8)), dim3(256), 0, st, p, u0, lines, col_tiles, range, partial));
    TB_LAUNCH_CHECK();
    u0 += cnt;
  }
  return TB_OK;
}

}  // namespace tb
