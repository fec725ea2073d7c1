// Grid search with many rows on the integer tensor cores.
//
// Score of candidate grid (s, z) with codes q, n = q - z, error e = w - s n, up to the common (w H w) / 2:
//   J = s^2 n T n - s n (H w),    T: upper triangle of H, diagonal halved.
// n holds integers of at most 8 bits, so n T n is a sum of exact int8 products once T is cut into six signed base-256
// digits, where the errors e themselves (k_grid_tri, k_grid_score) need double precision; H w is one product per row
// instead of one per candidate.  (8 bits: n does not fit a byte, m = q - 128 = n - k does, and
// n T n = m T m + k sum_j (n_j - k / 2) (H 1)_j.)
//
// The difference cancels, so J has a rounding error of its own; it is bounded (k_gd_pick), and so is the error of
// the direct evaluation e T e.  A candidate is taken when no other one's interval reaches its own: then the direct
// evaluation has the same winner.  Otherwise the candidates left are evaluated directly, e T e in double
// (k_gd_rescore), so that the choice is always that of the direct evaluation, ties to the lowest candidate included.
//
//   k_gd_hmax, k_gd_slice  digits of T, once per call for all steps
//   k_gd_h                 H w of the rows, FP64 tensor steps
//   k_gd_codes             ranges, candidates, integers n (in the products' operand layout), n (H w)
//   k_gd_score             n T n: 128 candidate rows x a column tile x two digits at a time
//   k_gd_pick, k_gd_rescore, k_gd_repick
// 4096 rows x 4096 columns, groups of 128, 16 candidates: 1.93 ms directly (0.48 of the FP64 pipe's rate), 0.84 ms
// here: k_gd_score 0.30 (the tensor pipe 0.32 busy, reading its results 0.36, integer instructions of the epilogue 0.33),
// k_gd_codes 0.25 (0.61 of the issue slots), k_gd_h 0.22 (FP64 tensor steps 0.56 busy), k_gd_pick 0.04.
// Groups of 64: 2.44 -> 1.08 ms; of 32: 3.76 -> 1.88; 208 rows x one group of 1664: 0.63 -> 0.22 ms a step.
#include "tb_grid.cuh"
#include "tb_gemm.cuh"
#include "tb_rows.cuh"
#include "tb_tma.cuh"

namespace tb {

enum {
  GD_PAIRS = 3,  // digit pairs of T
  GD_CHUNK_MB = 128,
  GD_EPI = 16,   // epilogue warps of k_gd_score: 32 rows x a quarter of the columns each
  GD_THREADS = 32 * (GD_EPI + 2),
  GD_A_STAGES = 6,
  GD_B_STAGES = 3,
  GD_A_BYTES = 128 * 128,
  GD_B_BYTES = 128 * 256,
  GD_SMEM = GD_A_STAGES * GD_A_BYTES + GD_B_STAGES * GD_B_BYTES + 2 * 4 * 128 * 8 + 512 + 128
};

__device__ int g_gd_error = 0;

int grid_digits_error_read_clear() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_gd_error, sizeof(int)) != cudaSuccess) return -1;
  if (v) {
    int z = 0;
    cudaMemcpyToSymbol(g_gd_error, &z, sizeof(int));
  }
  return v;
}

// Column tiles of a group: ct columns of 128 (the last may hold fewer), kc of them when the group is narrower.
struct GdGeom {
  int seg, ng, d, cts, kc;
  long long blocks;  // digit blocks per group
};
__host__ __device__ inline GdGeom gd_geom(int d, int seg) {
  GdGeom g;
  g.seg = seg;
  g.d = d;
  g.ng = d / seg;
  g.cts = (seg + 127) / 128;
  g.kc = seg < 128 ? seg : 128;
  g.blocks = (long long)GD_PAIRS * g.cts * (g.cts + 1) / 2;
  return g;
}
// digit block of (column tile, pair, contraction chunk): [chunk columns / 16][2 x tile columns][16]
__host__ __device__ inline long long gd_block(const GdGeom& g, int ct, int pr, int c) {
  return (long long)GD_PAIRS * ct * (ct + 1) / 2 + (long long)pr * (ct + 1) + c;
}
__device__ __forceinline__ int gd_exponent(unsigned int bits) { return (int)(bits >> 23) - 126; }  // |x| < 2^E

__global__ void __launch_bounds__(256) k_gd_hmax(const float* __restrict__ H, int d, int seg, unsigned int* hmax) {
  const float* Hg = H + (long long)blockIdx.z * d * d + (long long)blockIdx.y * seg * (d + 1);
  unsigned int m = 0;
  for (int k = blockIdx.x; k < seg; k += gridDim.x)
    for (int n = k + threadIdx.x; n < seg; n += 256)
      m = max(m, __float_as_uint(Hg[(long long)k * d + n]) & 0x7fffffffu);  // a NaN is larger than everything
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(hmax + (long long)blockIdx.z * gridDim.y + blockIdx.y, m);
}

// one digit block position (column tile, chunk) of one group, all three pairs
__global__ void __launch_bounds__(256) k_gd_slice(const float* __restrict__ H, GdGeom g, const unsigned int* __restrict__ hmax,
                                                  unsigned char* __restrict__ dst) {
  int ct = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while (ct * (ct + 1) / 2 > (int)blockIdx.x) --ct;
  while ((ct + 1) * (ct + 2) / 2 <= (int)blockIdx.x) ++ct;
  const int c = blockIdx.x - ct * (ct + 1) / 2;
  const long long gi = (long long)blockIdx.z * g.ng + blockIdx.y;
  const float* Hg = H + (long long)blockIdx.z * g.d * g.d + (long long)blockIdx.y * g.seg * (g.d + 1);
  const int n0 = ct * 128, k0 = c * 128, nt = min(128, g.seg - n0), kn = min(128, g.seg - k0);
  const int n = threadIdx.x & 127;
  if (n >= nt) return;
  const double scale = pow2d(46 - gd_exponent(hmax[gi]));
  const long long blk_bytes = 2ll * g.kc * g.kc;
  unsigned char* base = dst + gi * g.blocks * blk_bytes;
  for (int kb = threadIdx.x >> 7; kb < kn / 16; kb += 2) {
    unsigned int w[6][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int i = 0; i < 6; ++i) w[i][q] = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = k0 + 16 * kb + 4 * q + j;
        float v = (k <= n0 + n) ? Hg[(long long)k * g.d + n0 + n] : 0.0f;
        double x = (double)v * scale;
        if (k == n0 + n) x *= 0.5;
        // |x| <= 2^46: adding 128 to every digit makes the bytes of the sum the digits plus 128
        const unsigned long long y = (unsigned long long)__double2ll_rn(x) + 0x808080808080ull;
#pragma unroll
        for (int i = 0; i < 6; ++i) w[i][q] |= (unsigned int)((y >> (8 * (5 - i))) & 0xff) << (8 * j);
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) w[i][q] ^= 0x80808080u;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
      *reinterpret_cast<uint4*>(base + gd_block(g, ct, i >> 1, c) * blk_bytes + ((long long)kb * 2 * nt + (i & 1) * nt + n) * 16) =
          make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
  }
}

// r = H 1 of every group (8 bits only), from the upper triangle: a warp per column
__global__ void __launch_bounds__(256) k_gd_rsum(const float* __restrict__ H, int d, int seg, double* __restrict__ r) {
  const int col = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (col >= d) return;
  const int n = col % seg;
  const float* Hg = H + (long long)blockIdx.y * d * d + (long long)(col - n) * (d + 1);
  double t = 0.0;
  for (int k = lane; k < seg; k += 32) t += (double)Hg[(long long)min(k, n) * d + max(k, n)];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) r[(long long)blockIdx.y * d + col] = t;
}

// rows m0 .. of the step, `units` units of unit_rows rows (the first is unit u0 of H_in)
struct GdP {
  GridP p;
  GdGeom g;
  int m0, u0, units, unit_rows, tiles;  // tiles of 128 candidate rows per unit
  int ncp, eight;
  const unsigned int* hmax;
  const unsigned char* B;
  unsigned char* A;
  double* h;       // [row][d]
  const double* r;  // [unit][d] (8 bits)
  double4* range;  // [line], line = row ng + group: minimum, maximum, sum of magnitudes
  double* lin;     // [line][cts][ncp]
  double* part;    // [line][cts][ncp]: m T m in units of 2^(E - 46)
  int *count, *list;
};

// h = w H of RT rows x NT columns of one group; H from its upper triangle.  8 warps of RT / 2 x NT / 4.
template <int RT, int NT>
__global__ void __launch_bounds__(256, NT == 128 ? 2 : 3) k_gd_h(GdP q) {
  constexpr int MF = RT / 16, NF = NT / 32, AV = RT / 8, BV = NT / 8;
  __shared__ double As[RT][36];
  __shared__ float Bs[32][NT + 8];
  const GdGeom& g = q.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, fr = lane >> 2, fk = lane & 3;
  const int cpg = (g.seg + NT - 1) / NT;  // column tiles per group
  const int grp = blockIdx.x / cpg, n0 = (blockIdx.x % cpg) * NT;
  const int rpt = (q.unit_rows + RT - 1) / RT;
  const int unit = blockIdx.y / rpt, r0 = (blockIdx.y % rpt) * RT;
  const int rows = min(RT, q.unit_rows - r0), mb = q.m0 + unit * q.unit_rows + r0;
  const float* Hg = q.p.Hin + (q.p.units > 1 ? (long long)(q.u0 + unit) * g.d * g.d : 0) + (long long)grp * g.seg * (g.d + 1);
  const int wr = (warp >> 2) * (RT / 2), wc = (warp & 3) * (NT / 4);
  double acc[MF][NF][2];
#pragma unroll
  for (int i = 0; i < MF * NF * 2; ++i) (&acc[0][0][0])[i] = 0.0;
  double av[AV];
  float bv[BV];
  auto fetch = [&](int k0) {  // the next contraction chunk, while this one is multiplied
#pragma unroll
    for (int i = 0; i < AV; ++i) {
      const int rr = warp + 8 * i;
      av[i] = (rr < rows) ? q.p.Wt[q.p.rm.row(mb + rr) * g.d + (long long)grp * g.seg + k0 + lane] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < BV; ++i) {
      // on or above the diagonal (mostly) along the row of H, below it the mirrored entry, along its row
      const int n = (k0 <= n0) ? tid % NT : warp + 8 * i, kk = (k0 <= n0) ? tid / NT + 256 / NT * i : lane;
      const int lo = min(k0 + kk, n0 + n), hi = max(k0 + kk, n0 + n);
      bv[i] = (n0 + n < g.seg) ? Hg[(long long)lo * g.d + hi] : 0.0f;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < g.seg; k0 += 32) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < AV; ++i) As[warp + 8 * i][lane] = av[i];
#pragma unroll
    for (int i = 0; i < BV; ++i) {
      if (k0 <= n0)
        Bs[tid / NT + 256 / NT * i][tid % NT] = bv[i];
      else
        Bs[lane][warp + 8 * i] = bv[i];
    }
    __syncthreads();
    if (k0 + 32 < g.seg) fetch(k0 + 32);
#pragma unroll
    for (int k4 = 0; k4 < 8; ++k4) {
      double a[MF], b[NF];
#pragma unroll
      for (int i = 0; i < MF; ++i) a[i] = As[wr + 8 * i + fr][4 * k4 + fk];
#pragma unroll
      for (int j = 0; j < NF; ++j) b[j] = (double)Bs[4 * k4 + fk][wc + 8 * j + fr];
#pragma unroll
      for (int i = 0; i < MF; ++i)
#pragma unroll
        for (int j = 0; j < NF; ++j)
          dmma(acc[i][j], a[i], b[j]);
    }
  }
#pragma unroll
  for (int i = 0; i < MF; ++i)
#pragma unroll
    for (int j = 0; j < NF; ++j) {
      const int rr = wr + 8 * i + fr, n = n0 + wc + 8 * j + 2 * fk;
      if (rr < rows && n < g.seg)
        *reinterpret_cast<double2*>(q.h + (long long)(mb - q.m0 + rr) * g.d + (long long)grp * g.seg + n) =
            make_double2(acc[i][j][0], acc[i][j][1]);
    }
}

// minimum, maximum and sum of magnitudes of a wide group
__global__ void __launch_bounds__(256) k_gd_range(GdP q) {
  __shared__ double red[3][8];
  const int tid = threadIdx.x;
  const double* w = q.p.Wt + q.p.rm.row(q.m0 + blockIdx.y) * q.g.d + (long long)blockIdx.x * q.g.seg;
  double mn = 0.0, mx = 0.0, sum = 0.0;
  for (int a = tid; a < q.g.seg; a += 256) {
    const double v = w[a];
    mn = fmin(mn, v);
    mx = fmax(mx, v);
    sum += fabs(v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
  }
  if ((tid & 31) == 0) {
    red[0][tid >> 5] = mn;
    red[1][tid >> 5] = mx;
    red[2][tid >> 5] = sum;
  }
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < 8; ++i) {
      mn = fmin(mn, red[0][i]);
      mx = fmax(mx, red[1][i]);
      sum += red[2][i];
    }
    q.range[(long long)blockIdx.y * q.g.ng + blockIdx.x] = make_double4(mn, mx, sum, 0.0);
  }
}

// A warp per (row, group, chunk of 128 columns).  Lane: columns 8 (lane / 2) .., every second candidate: it makes 8 codes at
// a time, half a 16-byte piece of the operand, and its share of n (H w).  The shares of NR candidates are summed over
// the lanes together, half of them handed over at every step.
template <bool EIGHT, int NR>
__global__ void __launch_bounds__(256) k_gd_codes(GdP q) {
  const GdGeom& g = q.g;
  if (blockIdx.x == 0 && threadIdx.x == 0) *q.count = 0;
  const int lane = threadIdx.x & 31, blk = lane >> 1, sub = lane & 1;
  const long long item = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int c = (int)(item % g.cts);
  const int line = (int)(item / g.cts);
  const int grp = line % g.ng, rl = line / g.ng;  // row of the chunk
  if (rl >= q.units * q.unit_rows) return;
  const bool on = 8 * blk < min(128, g.seg - 128 * c);
  const long long col = (long long)grp * g.seg + 128 * c + 8 * blk;
  const int unit = rl / q.unit_rows, ru = rl - unit * q.unit_rows;
  double w[8], h[8], r[EIGHT ? 8 : 1];
  {
    const double* wp = q.p.Wt + q.p.rm.row(q.m0 + rl) * g.d + col;
    const double* hp = q.h + (long long)rl * g.d + col;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      const double2 a = on ? *reinterpret_cast<const double2*>(wp + j) : make_double2(0.0, 0.0);
      const double2 b = on ? *reinterpret_cast<const double2*>(hp + j) : make_double2(0.0, 0.0);
      w[j] = a.x;
      w[j + 1] = a.y;
      h[j] = b.x;
      h[j + 1] = b.y;
    }
    if (EIGHT) {
      const double* rp = q.r + (q.p.units > 1 ? (long long)(q.u0 + unit) * g.d : 0) + col;
#pragma unroll
      for (int j = 0; j < 8; ++j) r[EIGHT ? j : 0] = on ? rp[j] : 0.0;
    }
  }
  double2 mnmx;
  if (g.cts > 1) {
    const double4 t = q.range[line];
    mnmx = make_double2(t.x, t.y);
  } else {
    double mn = 0.0, mx = 0.0, sum = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      mn = fmin(mn, w[j]);
      mx = fmax(mx, w[j]);
      sum += fabs(w[j]);
    }
#pragma unroll
    for (int o = 2; o < 32; o <<= 1) {
      mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    mnmx = make_double2(mn, mx);
    if (lane == 0) q.range[line] = make_double4(mn, mx, sum, 0.0);
  }
  double cs, cz;
  gw_candidate(mnmx, lane, q.p.maxq, &cs, &cz);  // a lane per candidate
  const double crs = 1.0 / cs;
  const int rt = 128 / q.ncp, tile = ru / rt, pr0 = (ru - tile * rt) * q.ncp;
  unsigned char* Ab = q.A + ((((long long)unit * q.tiles + tile) * g.ng + grp) * g.cts + c) * (128ll * g.kc) +
                      (blk >> 1) * 2048 + (blk & 1) * 8;
  for (int rd0 = 0; rd0 < q.ncp; rd0 += 2 * NR) {
    double dot[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      const int cand = rd0 + 2 * i + sub;
      const double rs = __shfl_sync(0xffffffffu, crs, cand), z = __shfl_sync(0xffffffffu, cz, cand);
      const double zm = z + 6755399441055744.0;
      const int off = EIGHT ? 128 : (int)z;
      const double hk = 0.5 * (128.0 - z);
      double d0 = 0.0, d1 = 0.0, d2 = 0.0;
      int n[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        n[j] = gw_code(w[j], rs, zm, q.p.maxq);
        const double dn = __hiloint2double(0x43380000, n[j]) - zm;  // q - z, exact
        if (j & 1)
          d1 = fma(dn, h[j], d1);
        else
          d0 = fma(dn, h[j], d0);
        if (EIGHT) d2 = fma(dn - hk, r[EIGHT ? j : 0], d2);
        n[j] -= off;
      }
      d0 += d1;
      if (EIGHT) d0 = fma(-__shfl_sync(0xffffffffu, cs, cand) * (128.0 - z), d2, d0);
      dot[i] = d0;
      if (on) {
        const int pr = pr0 + cand;
        *reinterpret_cast<uint2*>(Ab + (pr >> 3) * 128 + (pr & 7) * 16) =
            make_uint2(__byte_perm(__byte_perm(n[0], n[1], 0x0040), __byte_perm(n[2], n[3], 0x0040), 0x5410),
                       __byte_perm(__byte_perm(n[4], n[5], 0x0040), __byte_perm(n[6], n[7], 0x0040), 0x5410));
      }
    }
    int mine = 0, o = 2;
#pragma unroll
    for (int half = NR / 2; half > 0; half >>= 1, o <<= 1) {
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < half; ++i) {
        const double give = up ? dot[i] : dot[i + half], keep = up ? dot[i + half] : dot[i];
        dot[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
      if (up) mine += half;
    }
    for (; o < 32; o <<= 1) dot[0] += __shfl_xor_sync(0xffffffffu, dot[0], o);
    if (lane < 2 * NR) q.lin[((long long)line * g.cts + c) * q.ncp + rd0 + 2 * mine + sub] = dot[0];
  }
}

__device__ __forceinline__ void gd_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
               "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ int gd_sbyte(uint32_t v, int i) {  // byte i with its sign
  int r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(v), "r"(0x8880 + 0x1111 * i));
  return r;
}
__device__ __forceinline__ void gd_tmem_ld8(uint32_t taddr, int (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}

// One work unit: 128 candidate rows x one column tile, contraction over the group's columns up to the tile's end, two
// digits of T at a time into one of two accumulators of 256 columns; the epilogue takes the row dots with the integers
// themselves (the last chunk of the operand).  Narrow groups: a CTA takes a run of row tiles against the same digits,
// which stay in shared memory, and the integers are loaded once for the three digit pairs.  Wide groups: CTAs next to
// one another take row tiles of the same column tile, longest contraction first.
template <bool WIDE>
__global__ void __launch_bounds__(GD_THREADS, 1) k_gd_score(GdP q, int n_work) {
  extern __shared__ __align__(128) unsigned char gd_raw[];
  const GdGeom& g = q.g;
  const uint32_t base = smem_u32(gd_raw);
  const uint32_t b_base = base + GD_A_STAGES * GD_A_BYTES;
  double* red = reinterpret_cast<double*>(gd_raw + GD_A_STAGES * GD_A_BYTES + GD_B_STAGES * GD_B_BYTES);  // [2][4][128]
  uint64_t* bars = reinterpret_cast<uint64_t*>(red + 2 * 4 * 128);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * GD_A_STAGES + 2 * GD_B_STAGES + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t bar0 = smem_u32(bars);
  auto a_full = [&](int s) { return bar0 + 8u * s; };
  auto a_empty = [&](int s) { return bar0 + 8u * (GD_A_STAGES + s); };
  auto b_full = [&](int s) { return bar0 + 8u * (2 * GD_A_STAGES + s); };
  auto b_empty = [&](int s) { return bar0 + 8u * (2 * GD_A_STAGES + GD_B_STAGES + s); };
  auto acc_full = [&](int s) { return bar0 + 8u * (2 * GD_A_STAGES + 2 * GD_B_STAGES + s); };
  auto acc_empty = [&](int s) { return bar0 + 8u * (2 * GD_A_STAGES + 2 * GD_B_STAGES + 2 + s); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < GD_A_STAGES; ++s) {
      mbar_init(a_full(s), 1);
      mbar_init(a_empty(s), 1 + GD_EPI);
    }
    for (int s = 0; s < GD_B_STAGES; ++s) {
      mbar_init(b_full(s), 1);
      mbar_init(b_empty(s), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(acc_full(s), 1);
      mbar_init(acc_empty(s), GD_EPI);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == GD_EPI) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // this CTA's work
  const int t_first = WIDE ? blockIdx.x : (int)((long long)n_work * blockIdx.x / gridDim.x);
  const int t_end = WIDE ? n_work : (int)((long long)n_work * (blockIdx.x + 1) / gridDim.x);
  const int t_step = WIDE ? gridDim.x : 1;
  struct Work {
    int unit, grp, ct, tile, item;
  };
  auto decode = [&](int t, Work& w) {
    if (!WIDE && t != t_first && ++w.tile < q.tiles) return;  // the next row tile of the same item
    w.tile = t % q.tiles;
    w.item = t / q.tiles;
    w.grp = w.item % g.ng;
    w.unit = w.item / g.ng;
    w.ct = 0;
    if (WIDE) {  // [column tile descending][unit][group]
      w.ct = g.cts - 1 - w.unit / q.units;
      w.unit %= q.units;
    }
  };
  const long long a_blk = 128ll * g.kc, b_blk = 2ll * g.kc * g.kc;

  if (warp == GD_EPI) {
    if (lane == 0) {
      uint32_t ai = 0, bi = 0;
      int last = -1;
      Work w;
      for (int t = t_first; t < t_end && !*abort_flag; t += t_step) {
        decode(t, w);
        const int nt = min(128, g.seg - 128 * w.ct);
        const unsigned char* A = q.A + ((((long long)w.unit * q.tiles + w.tile) * g.ng + w.grp) * g.cts) * a_blk;
        const unsigned char* B = q.B + ((long long)(q.p.units > 1 ? q.u0 + w.unit : 0) * g.ng + w.grp) * g.blocks * b_blk +
                                 gd_block(g, w.ct, 0, 0) * b_blk;
        for (int pr = 0; pr < GD_PAIRS; ++pr)
          for (int c = 0; c <= w.ct; ++c) {
            const int kn = min(128, g.seg - 128 * c);
            if (WIDE || w.item != last) {
              const int s = bi % GD_B_STAGES;
              if (!mbar_wait(b_empty(s), ((bi / GD_B_STAGES) & 1u) ^ 1u, abort_flag, &g_gd_error)) break;
              mbar_expect_tx(b_full(s), kn * 2 * nt);
              gd_bulk(b_base + s * GD_B_BYTES, B + (pr * (w.ct + 1) + c) * b_blk, kn * 2 * nt, b_full(s));
              ++bi;
            }
            if (WIDE || pr == 0) {
              const int s = ai % GD_A_STAGES;
              if (!mbar_wait(a_empty(s), ((ai / GD_A_STAGES) & 1u) ^ 1u, abort_flag, &g_gd_error)) break;
              mbar_expect_tx(a_full(s), kn * 128);
              gd_bulk(base + s * GD_A_BYTES, A + c * a_blk, kn * 128, a_full(s));
              ++ai;
            }
          }
        last = w.item;
      }
    }
  } else if (warp == GD_EPI + 1) {
    if (lane == 0) {
      uint32_t ai = 0, bi = 0, u = 0;  // stages taken so far, accumulators filled
      int last = -1;
      bool ok = true;
      Work w;
      for (int t = t_first; t < t_end && ok; t += t_step) {
        decode(t, w);
        const int nt = min(128, g.seg - 128 * w.ct);
        const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * nt >> 3) << 17) | ((128u >> 4) << 24);
        const bool fresh = w.item != last, done = t + t_step >= t_end || w.tile == q.tiles - 1;
        if (!WIDE && fresh) bi += GD_PAIRS;
        for (int pr = 0; pr < GD_PAIRS && ok; ++pr, ++u) {
          const int buf = u & 1;
          ok = mbar_wait(acc_empty(buf), ((u >> 1) & 1u) ^ 1u, abort_flag, &g_gd_error);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int c = 0; c <= w.ct && ok; ++c) {
            const int kn = min(128, g.seg - 128 * c);
            const uint32_t bt = WIDE ? bi : bi - GD_PAIRS + pr;
            const int s = ai % GD_A_STAGES, sb = bt % GD_B_STAGES;
            if (WIDE || fresh) ok = mbar_wait(b_full(sb), (bt / GD_B_STAGES) & 1u, abort_flag, &g_gd_error);
            if (WIDE || pr == 0) ok = ok && mbar_wait(a_full(s), (ai / GD_A_STAGES) & 1u, abort_flag, &g_gd_error);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int k = 0; k < kn / 32; ++k)
              umma_i8(tmem + 256 * buf, smem_desc_k(base + s * GD_A_BYTES + k * 4096, 2048),
                     smem_desc_k(b_base + sb * GD_B_BYTES + k * 64 * nt, 32 * nt), idesc, (c > 0 || k > 0) ? 1u : 0u);
            if (WIDE || pr == GD_PAIRS - 1) {
              umma_commit(a_empty(s));
              ++ai;
            }
            if (WIDE || done) umma_commit(b_empty(sb));
            if (WIDE) ++bi;
          }
          if (ok) umma_commit(acc_full(buf));
        }
        last = w.item;
      }
    }
  } else {
    // epilogue: rows 32 (warp % 4) .., quarter warp / 4 of the columns
    const int rq = warp & 3, cq = warp >> 2, row = rq * 32 + lane;
    const int lg = 31 - __clz(q.ncp), row_line = row >> lg;
    uint32_t ai = 0, u = 0, n_work_done = 0;
    Work w;
    for (int t = t_first; t < t_end; t += t_step, ++n_work_done) {  // no early exit: every warp meets every barrier
      decode(t, w);
      const int nt = min(128, g.seg - 128 * w.ct), per = nt / 4;  // 8, 16, 24 or 32 columns
      int m[32];
      double sum = 0.0;
      for (int pr = 0; pr < GD_PAIRS; ++pr, ++u) {
        const int buf = u & 1;
        if (WIDE || pr == 0) {
          for (int c = 0; c <= w.ct; ++c, ++ai) {
            const int s = ai % GD_A_STAGES;
            mbar_wait(a_full(s), (ai / GD_A_STAGES) & 1u, abort_flag, &g_gd_error);
            if (pr == 0 && c == w.ct) {
              const unsigned char* a = gd_raw + s * GD_A_BYTES + (row >> 3) * 128 + (row & 7) * 16;
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int n = cq * per + 8 * j;
                uint2 v = make_uint2(0, 0);
                if (8 * j < per) v = *reinterpret_cast<const uint2*>(a + (n >> 4) * 2048 + (n & 8));
#pragma unroll
                for (int e = 0; e < 8; ++e) m[8 * j + e] = gd_sbyte(e < 4 ? v.x : v.y, e & 3);
              }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(a_empty(s));
          }
        }
        mbar_wait(acc_full(buf), (u >> 1) & 1u, abort_flag, &g_gd_error);
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t ta = tmem + ((uint32_t)(rq * 32) << 16) + (uint32_t)(256 * buf + cq * per);
        long long sa = 0, sb = 0;
#pragma unroll
        for (int h = 0; h < 4; h += 2) {
          if (8 * h >= per) break;
          int va[2][8], vb[2][8];
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (8 * (h + j) < per) {
              gd_tmem_ld8(ta + 8 * (h + j), va[j]);
              gd_tmem_ld8(ta + nt + 8 * (h + j), vb[j]);
            }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (8 * (h + j) < per) {
              int ia = 0, ib = 0;  // 8 products of 2^21 (128 digit products) and 2^7
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                if (WIDE) {
                  sa += (long long)m[8 * (h + j) + e] * va[j][e];
                  sb += (long long)m[8 * (h + j) + e] * vb[j][e];
                } else {
                  ia += m[8 * (h + j) + e] * va[j][e];
                  ib += m[8 * (h + j) + e] * vb[j][e];
                }
              }
              if (!WIDE) {
                sa += ia;
                sb += ib;
              }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty(buf));
        sum = fma(sum, 65536.0, (double)(sa * 256 + sb));
      }
      double* rd = red + (n_work_done & 1) * 512;
      rd[cq * 128 + row] = sum;
      // the four warps of these rows; the other half of the buffer is free once all have passed
      asm volatile("bar.sync %0, 128;" ::"r"(1 + rq) : "memory");
      if (cq == 0) {
        const int ru = (w.tile << (7 - lg)) + row_line;
        if (ru < q.unit_rows) {
          const long long line = (long long)(w.unit * q.unit_rows + ru) * g.ng + w.grp;
          q.part[(line * g.cts + w.ct) * q.ncp + (row & (q.ncp - 1))] =
              (rd[row] + rd[128 + row]) + (rd[256 + row] + rd[384 + row]);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == GD_EPI) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// A lane per candidate, a warp for 32 / ncp (row, group) pairs: J, its error bound, the winner or an entry of the list.
//
// With eps = 2^-53, Hm = max |H| of the group, W = sum |w|, every sum over i, j is bounded by Hm times the product of
// absolute sums.  sum s |n| <= S = W + seg s / 2, since |s n - w| <= s / 2 or n was clamped, towards zero.  (8 bits: S gets
// another 192 seg s for the integers moved by 128 and their k sum (n - k / 2).)
//   digits       T is rounded at 2^-47 2^E <= 2^-46 Hm:                      2^-46 Hm S^2
//   n T n        exact, ten roundings to double per column tile:              (10 cts + 2) eps Hm S^2
//   n (H w)      seg + 2 terms twice (each dot, H w before that):            (2 seg + 8) eps Hm S W
//   n (H 1)      8 bits, the same with s n for w:                            (2 seg + 8) eps Hm S^2
//   direct e T e: e rounded twice, |e| <= |w| + s |n|:  2 eps Hm (S + W)^2, its sums: (seg + 8) eps Hm (S + W)^2
// in all below Hm (S + W)^2 (2^-45 + (6 seg + 64) eps), with room for the roundings of the bound itself.
__global__ void __launch_bounds__(256) k_gd_pick(GdP q, long long lines) {
  const GdGeom& g = q.g;
  const int lane = threadIdx.x & 31, lg = 31 - __clz(q.ncp), cand = lane & (q.ncp - 1), first = lane - cand;
  const long long line_ = ((((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) << (5 - lg)) + (lane >> lg));
  const bool valid = line_ < lines, in = valid && cand < q.p.n_cand;
  const long long line = valid ? line_ : lines - 1;
  const int rl = (int)line / g.ng, grp = (int)line % g.ng, unit = rl / q.unit_rows;
  const unsigned int hb = q.hmax[(q.p.units > 1 ? (long long)(q.u0 + unit) * g.ng : 0) + grp];
  const double4 range = q.range[line];
  double s, z;
  gw_candidate(make_double2(range.x, range.y), cand, q.p.maxq, &s, &z);
  double P = 0.0, L = 0.0;
  if (in)
    for (int c = 0; c < g.cts; ++c) {
      P += q.part[(line * g.cts + c) * q.ncp + cand];
      L += q.lin[(line * g.cts + c) * q.ncp + cand];
    }
  const double J = s * fma(s * pow2d(gd_exponent(hb) - 46), P, -L);
  const double seg = (double)g.seg;
  const double SW = 2.0 * range.z + seg * s * (q.eight ? 192.5 : 0.5);
  const double delta = (double)__uint_as_float(hb) * SW * SW * (0x1p-45 + (6.0 * seg + 64.0) * 0x1p-53);
  const bool number = fabs(J) <= 1.7e308 && delta <= 1.7e308;  // false for NaN as well
  const unsigned int mine = (q.ncp == 32 ? 0xffffffffu : (1u << q.ncp) - 1u) << first;
  const bool numbers = (__ballot_sync(0xffffffffu, in && !number) & mine) == 0;
  double hi = in ? J + delta : INFINITY;
  for (int o = q.ncp >> 1; o > 0; o >>= 1) hi = fmin(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  bool keep = in && (!numbers || !(J - delta > hi));
  if (range.x == 0.0 && range.y == 0.0) keep = in && cand == 0;  // all candidates are the same grid
  const unsigned int left = (__ballot_sync(0xffffffffu, keep) & mine) >> first;
  const int best = __ffs(left) - 1;
  if (valid && cand == best) {
    const long long o = q.p.rm.row(q.m0 + rl) * g.ng + grp;
    q.p.sD[o] = s;
    q.p.s_out[o] = (float)s;
    q.p.z_out[o] = (int)z;
    if (q.p.cand_out) q.p.cand_out[o] = (unsigned char)best;
    if (left & (left - 1)) {
      const int at = atomicAdd(q.count, 1);
      q.list[2 * at] = (int)line;
      q.list[2 * at + 1] = (int)left;
    }
  }
}

// The candidates that k_gd_pick could not tell apart: e T e in double, a CTA per entry and column tile (the partial
// scores take the place of the sums that k_gd_pick has read).  A thread per column and eighth of up to 1024 contraction rows.
__global__ void __launch_bounds__(1024) k_gd_rescore(GdP q) {
  __shared__ double e_sm[1024], red[32];
  const GdGeom& g = q.g;
  const int tid = threadIdx.x, jt = tid & 127, kq = tid >> 7;
  const long long n_items = (long long)*q.count * g.cts;
  for (long long i = blockIdx.x; i < n_items; i += gridDim.x) {
    const int ct = (int)(i % g.cts), line = q.list[2 * (i / g.cts)];
    const unsigned int left = (unsigned int)q.list[2 * (i / g.cts) + 1];
    const int rl = line / g.ng, grp = line % g.ng, unit = rl / q.unit_rows;
    const double* w = q.p.Wt + q.p.rm.row(q.m0 + rl) * g.d + (long long)grp * g.seg;
    const float* Hg = q.p.Hin + (q.p.units > 1 ? (long long)(q.u0 + unit) * g.d * g.d : 0) + (long long)grp * g.seg * (g.d + 1);
    const double4 range = q.range[line];
    const int j = 128 * ct + jt, k_end = min(g.seg, 128 * ct + 128);
    const bool in = j < g.seg;
    for (unsigned int rest = left; rest; rest &= rest - 1) {
      const int cand = __ffs(rest) - 1;
      double s, z;
      gw_candidate(make_double2(range.x, range.y), cand, q.p.maxq, &s, &z);
      const double rs = 1.0 / s;
      double t = 0.0;
      for (int i0 = 0; i0 < k_end; i0 += 1024) {
        __syncthreads();
        e_sm[tid] = (i0 + tid < k_end) ? gw_error(w[i0 + tid], s, rs, z, q.p.maxq) : 0.0;
        __syncthreads();
        const int per = min(1024, k_end - i0) / 8, k0 = kq * per;  // groups are multiples of 32 columns
        const float* hp = Hg + (long long)(i0 + k0) * g.d + min(j, g.seg - 1);
        double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
        for (int k = 0; k < per; k += 4) {
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = hp[(long long)(k + e) * g.d];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int ii = i0 + k0 + k + e;
            a[e] = fma(ii < j ? (double)v[e] : ii == j ? 0.5 * (double)v[e] : 0.0, e_sm[k0 + k + e], a[e]);
          }
        }
        if (in) t = fma((a[0] + a[1]) + (a[2] + a[3]), gw_error(w[j], s, rs, z, q.p.maxq), t);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if ((tid & 31) == 0) red[tid >> 5] = t;
      __syncthreads();
      if (tid == 0) {
        for (int k = 1; k < 32; ++k) t += red[k];
        q.part[((long long)line * g.cts + ct) * q.ncp + cand] = t;
      }
    }
  }
}
// and the choice among them: strict '<', the lowest candidate wins ties; one that scores no number never beats another
__global__ void __launch_bounds__(256) k_gd_repick(GdP q) {
  const GdGeom& g = q.g;
  const int n_list = *q.count;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n_list; i += gridDim.x * 256) {
    const int line = q.list[2 * i];
    int best = -1;
    double bj = 0.0;
    for (unsigned int rest = (unsigned int)q.list[2 * i + 1]; rest; rest &= rest - 1) {
      const int cand = __ffs(rest) - 1;
      double t = 0.0;
      for (int c = 0; c < g.cts; ++c) t += q.part[((long long)line * g.cts + c) * q.ncp + cand];
      if (best < 0 || t < bj) {
        best = cand;
        bj = t;
      }
    }
    const double4 range = q.range[line];
    double s, z;
    gw_candidate(make_double2(range.x, range.y), best, q.p.maxq, &s, &z);
    const long long o = q.p.rm.row(q.m0 + line / g.ng) * g.ng + line % g.ng;
    q.p.sD[o] = s;
    q.p.s_out[o] = (float)s;
    q.p.z_out[o] = (int)z;
    if (q.p.cand_out) q.p.cand_out[o] = (unsigned char)best;
  }
}

// From which size the launches pay (three and more candidates: a lane of k_gd_codes steps by two, and rounds go in
// pairs).  Measured with 16 candidates, the direct search against this one: groups of 128, 4096 columns, 128 rows
// 76 us / 87 us, 256 rows 127 / 102; 512 columns, 1024 rows 75 / 81, 2048 rows 127 / 97; groups of 32, 4096 columns,
// 128 rows 123 / 102; one group of 1664 columns, 32 rows 119 / 163, 64 rows 192 / 167; groups of 256, 4096 columns,
// 32 rows 65 / 71, 64 rows 110 / 80: a line in the elements of all candidates, lower for wide groups.  Digits of H_in
// that would not fit half a gigabyte stay with the direct search.
bool grid_wants_digits(int M, int units, int d, int seg, int ncp) {
  const GdGeom g = gd_geom(d, seg);
  return ncp >= 4 && (double)M * ncp * d >= (seg > 128 ? 2.5e6 : 1.2e7) &&
         (double)units * g.ng * g.blocks * 2.0 * g.kc * g.kc <= 512.0 * 1024 * 1024;
}

// Rows per chunk: operands of GD_CHUNK_MB, a multiple of the rows of a tile.  4096 rows, groups of 128, 4096 columns:
// 0.99 ms in chunks of 32 MB, which stay in L2 between the launches, 0.89 of 64, 0.83 of 128 (longer launches).
static int gd_chunk_rows(int M, int d, int ncp) {
  const int rt = 128 / ncp;
  long long tiles = ((long long)GD_CHUNK_MB << 20) / (128ll * d);
  if (tiles < 1) tiles = 1;
  long long rows = tiles * rt;
  if (rows > 32768) rows = 32768;  // rows are a grid dimension of k_row_range
  return rows < M ? (int)rows : M;
}

void grid_digits_scratch(Bump& b, int M, int units, int d, int seg, int ncp, int bits, GridDigits* s) {
  const GdGeom g = gd_geom(d, seg);
  const int rows = gd_chunk_rows(M, d, ncp), rpu = M / units, rt = 128 / ncp;
  // tiles end with their unit: at most one part tile per unit of a chunk
  const long long tiles = (rows >= rpu) ? (long long)(rows / rpu) * ((rpu + rt - 1) / rt) : (rows + rt - 1) / rt;
  const size_t lines = (size_t)rows * g.ng;
  s->rows = rows;
  s->A = b.take<unsigned char>((size_t)tiles * g.ng * g.cts * g.kc * 128);
  s->B = b.take<unsigned char>((size_t)units * g.ng * g.blocks * 2 * g.kc * g.kc);
  s->h = b.take<double>((size_t)rows * d);
  s->r = bits == 8 ? b.take<double>((size_t)units * d) : nullptr;
  s->range = b.take<double>(4 * lines);
  s->lin = b.take<double>(lines * g.cts * ncp);
  s->part = b.take<double>(lines * g.cts * ncp);
  s->hmax = b.take<unsigned int>((size_t)units * g.ng);
  s->list = b.take<int>(2 * lines + 64);  // the count, then the entries
}

tb_status grid_digits_prepare(const float* H, int units, int d, int seg, const GridDigits& s, cudaStream_t st) {
  const GdGeom g = gd_geom(d, seg);
  if (units > 65535 || g.ng > 65535) return TB_ERR_UNSUPPORTED;
  TB_CUDA_CHECK(cudaMemsetAsync(s.hmax, 0, (size_t)units * g.ng * sizeof(unsigned int), st));
  k_gd_hmax<<<dim3(seg < 64 ? seg : 64, g.ng, units), 256, 0, st>>>(H, d, seg, s.hmax);
  TB_LAUNCH_CHECK();
  k_gd_slice<<<dim3(g.cts * (g.cts + 1) / 2, g.ng, units), 256, 0, st>>>(H, g, s.hmax, s.B);
  TB_LAUNCH_CHECK();
  if (s.r) {
    k_gd_rsum<<<dim3((d + 7) / 8, units), 256, 0, st>>>(H, d, seg, s.r);
    TB_LAUNCH_CHECK();
  }
  return TB_OK;
}

tb_status grid_digits(const GridP& p, const GridDigits& s, cudaStream_t st) {
  static bool conf_n[64] = {false}, conf_w[64] = {false};
  TB_TRY(allow_smem(k_gd_score<false>, GD_SMEM, conf_n));
  TB_TRY(allow_smem(k_gd_score<true>, GD_SMEM, conf_w));
  GdP q;
  q.p = p;
  q.g = gd_geom(p.d, p.seg);
  q.ncp = p.ncp;
  q.eight = s.r != nullptr;
  q.hmax = s.hmax;
  q.A = s.A;
  q.B = s.B;
  q.h = s.h;
  q.r = s.r;
  q.range = reinterpret_cast<double4*>(s.range);
  q.lin = s.lin;
  q.part = s.part;
  q.count = s.list;
  q.list = s.list + 64;
  const int rt = 128 / p.ncp;
  for (int m0 = 0; m0 < p.M;) {
    const int in_unit = m0 % p.rows_per_unit;
    if (in_unit == 0 && s.rows >= p.rows_per_unit) {
      q.units = min(s.rows / p.rows_per_unit, (p.M - m0) / p.rows_per_unit);
      q.unit_rows = p.rows_per_unit;
    } else {
      q.units = 1;
      q.unit_rows = min(s.rows, p.rows_per_unit - in_unit);
    }
    const int cnt = q.units * q.unit_rows;
    q.m0 = m0;
    q.u0 = m0 / p.rows_per_unit;
    q.tiles = (q.unit_rows + rt - 1) / rt;
    const long long lines = (long long)cnt * q.g.ng;
    if (q.g.cts > 1) {
      k_gd_range<<<dim3(q.g.ng, cnt), 256, 0, st>>>(q);
      TB_LAUNCH_CHECK();
    }
    const long long work = (long long)q.units * q.g.ng * q.g.cts * q.tiles;
    if ((long long)q.units * ((q.unit_rows + 31) / 32) > 65535 || work > 0x7fffffff || lines * q.g.cts > 0x7fffffffll)
      return TB_ERR_UNSUPPORTED;
    // large tiles where they fill the SMs twice (groups of up to 64 columns have no 128)
    const long long t64 = (long long)q.units * ((q.unit_rows + 63) / 64), c64 = (long long)q.g.ng * ((p.seg + 63) / 64);
    if (p.seg > 64 && p.seg <= 128)
      k_gd_h<64, 128><<<dim3(q.g.ng, (unsigned)t64), 256, 0, st>>>(q);
    else if (p.seg <= 64 || t64 * c64 >= 296)
      k_gd_h<64, 64><<<dim3((unsigned)c64, (unsigned)t64), 256, 0, st>>>(q);
    else
      k_gd_h<32, 64><<<dim3((unsigned)c64, (unsigned)(q.units * ((q.unit_rows + 31) / 32))), 256, 0, st>>>(q);
    TB_LAUNCH_CHECK();
    const unsigned cg = (unsigned)((lines * q.g.cts + 7) / 8);
    switch ((q.eight ? 8 : 0) + (p.ncp == 4 ? 0 : p.ncp == 8 ? 1 : 2)) {
      case 0: k_gd_codes<false, 2><<<cg, 256, 0, st>>>(q); break;
      case 1: k_gd_codes<false, 4><<<cg, 256, 0, st>>>(q); break;
      case 2: k_gd_codes<false, 8><<<cg, 256, 0, st>>>(q); break;
      case 8: k_gd_codes<true, 2><<<cg, 256, 0, st>>>(q); break;
      case 9: k_gd_codes<true, 4><<<cg, 256, 0, st>>>(q); break;
      default: k_gd_codes<true, 8><<<cg, 256, 0, st>>>(q); break;
    }
    TB_LAUNCH_CHECK();
    const unsigned grid = work < 148 ? (unsigned)work : 148u;
    if (q.g.cts > 1)
      k_gd_score<true><<<grid, GD_THREADS, GD_SMEM, st>>>(q, (int)work);
    else
      k_gd_score<false><<<grid, GD_THREADS, GD_SMEM, st>>>(q, (int)work);
    TB_LAUNCH_CHECK();
    k_gd_pick<<<(unsigned)((lines * p.ncp + 255) / 256), 256, 0, st>>>(q, lines);
    TB_LAUNCH_CHECK();
    k_gd_rescore<<<296, 1024, 0, st>>>(q);
    TB_LAUNCH_CHECK();
    k_gd_repick<<<64, 256, 0, st>>>(q);
    TB_LAUNCH_CHECK();
    m0 += cnt;
  }
  return TB_OK;
}

}  // namespace tb
