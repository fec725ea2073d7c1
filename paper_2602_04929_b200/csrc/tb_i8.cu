// Double-precision products on the integer tensor cores: rounding to digits, and the product kernel.
//
// k_i8_gemm: one 128 x 64 tile of C at a time.  Seven int32 accumulators of 64 columns (one per digit weight
// s = i + j) take 448 of the 512 TMEM columns.  The digits j of B lie behind one another in shared memory as
// rows of one operand, so digit i of A meets digits 0 .. 6-i of B in one tcgen05.mma (two where that is more
// than 256 columns), whose result columns are the accumulators s = i .. 6: ten MMAs per 32 contraction steps,
// 920 clocks measured (896 at the peak rate), 43 KB of operands a stage, five stages.
// Bound: 43 KB of operands per 920 clocks and SM from L2 (47 B a clock; about 36 arrive when every SM asks),
// then the MMA rate; with short contractions the reading of the accumulators, which the next tile's products
// wait for.  Scaling and writing C overlaps them, and C's old values are fetched while they run.
// Measured (B200): 4096^3 1.15 ms = 119 TFLOP/s (FP64 pipe 4.1 ms), lower half of 8192 x 8192 with 256 steps 0.24 ms
// (0.61 ms), 1024 x 4096 x 4096 0.31 ms (1.20 ms).
#include "tb_i8.cuh"

namespace tb {

enum {
  I8_BM = 128,
  I8_BN = 64,
  I8_STAGES = 5,
  I8_A_BYTES = 2 * I8_BLOCK,
  I8_B_BYTES = I8_BLOCK,
  I8_STAGE_BYTES = I8_A_BYTES + I8_B_BYTES,
  I8_SMEM = I8_STAGES * I8_STAGE_BYTES + 1024 + 128,
  I8_EPI = 16,  // epilogue warps: 32 rows x 16 columns each
  I8_THREADS = 32 * (I8_EPI + 2)  // and a TMA warp, an MMA warp
};

__device__ int g_i8_error = 0;

int i8_error_read_clear() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_i8_error, sizeof(int)) != cudaSuccess) return -1;
  if (v) {
    int z = 0;
    cudaMemcpyToSymbol(g_i8_error, &z, sizeof(int));
  }
  return v;
}

// smallest E with |x| < 2^E for the largest magnitude of a row (zero rows: any)
__device__ __forceinline__ int i8_exponent(unsigned long long bits) {
  const int e = (int)(bits >> 52) - 1022;
  return e < -900 ? -900 : (e > 900 ? 900 : e);
}
// A row with an entry that is no finite number has no digits: its largest magnitude (a bit pattern, a NaN's above
// infinity's, both above every number's) is kept as it is, and the scale of its results is no number.
__device__ __forceinline__ double i8_result_scale(unsigned long long bits) {
  return (bits >> 52) >= 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : pow2d(i8_exponent(bits) - 54 + 24);
}
__device__ __forceinline__ unsigned long long i8_magnitude(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

__device__ __forceinline__ bool i8_masked(int mask, int k, int row) {
  return (mask == 1 && k > row) || (mask == 2 && k < row) || (mask == 3 && k <= row);
}

template <typename T, bool KCONTIG>
__global__ void __launch_bounds__(256) k_i8_row_max(I8Src s, unsigned long long* out, long long out_batch) {
  const T* X = static_cast<const T*>(s.X) + blockIdx.z * s.batch;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long m = 0;
  if (KCONTIG) {  // a warp per row, 512 contraction steps
    const int row = blockIdx.x * 8 + warp, k0 = blockIdx.y * 512;
    if (row >= s.rows) return;
    const T* x = X + (long long)row * s.ld;
    const int k_hi = min(s.K, k0 + 512);
#pragma unroll 4
    for (int k = k0 + lane; k < k_hi; k += 32)
      if (!i8_masked(s.mask, k, row)) {
        double v = (double)x[k];
        if (s.k_exp) v *= pow2d(s.k_sign * s.k_exp[k]);
        m = max(m, i8_magnitude(v));
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) atomicMax(out + blockIdx.z * out_batch + row, m);
  } else {  // a lane per row, 8 warps x 16 contraction steps
    const int row = blockIdx.x * 32 + lane, k0 = blockIdx.y * 128 + warp * 16;
    if (row >= s.rows) return;
    const T* x = X + row;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int k = k0 + i;
      if (k < s.K && !i8_masked(s.mask, k, row)) {
        double v = (double)x[(long long)k * s.ld];
        if (s.k_exp) v *= pow2d(s.k_sign * s.k_exp[k]);
        m = max(m, i8_magnitude(v));
      }
    }
    if (m) atomicMax(out + blockIdx.z * out_batch + row, m);
  }
}

// 128 threads: 64 rows x 2 halves of a 32-step block; a thread writes 16 contraction steps of its row, one
// 16-byte store per digit
template <typename T, bool KCONTIG>
__global__ void __launch_bounds__(128) k_i8_slice(I8Src s, const unsigned long long* max_bits, long long max_batch,
                                                  int fixed_exp, unsigned char* dst, int dst_k_blocks, long long rb0,
                                                  long long rb_batch, int kb0, int* bad) {
  const int r = threadIdx.x & 63, kc = threadIdx.x >> 6;
  const int row = blockIdx.y * 64 + r, k0 = blockIdx.x * 32 + kc * 16;
  const T* X = static_cast<const T*>(s.X) + blockIdx.z * s.batch;
  T x[16];
  if (KCONTIG && row < s.rows && k0 + 16 <= s.K) {
    const T* p = X + (long long)row * s.ld + k0;  // 16-byte aligned (checked by the launcher)
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        const double2 v = *reinterpret_cast<const double2*>(p + i);
        x[i] = v.x;
        x[i + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(p + i);
        x[i] = v.x;
        x[i + 1] = v.y;
        x[i + 2] = v.z;
        x[i + 3] = v.w;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const bool in = row < s.rows && k0 + i < s.K;
      x[i] = in ? X[KCONTIG ? (long long)row * s.ld + k0 + i : (long long)(k0 + i) * s.ld + row] : (T)0;
    }
  }
  int e = fixed_exp;
  if (max_bits) e = row < s.rows ? i8_exponent(max_bits[blockIdx.z * max_batch + row]) : 0;
  const double scale = pow2d(54 - e), limit = pow2d(fixed_exp);
  unsigned int w[I8_DIGITS][4];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    unsigned int lo[4], hi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = k0 + 4 * g + i;
      double v = (double)x[4 * g + i];
      if (i8_masked(s.mask, k, row)) v = 0.0;
      if (s.k_exp && k < s.K) v *= pow2d(s.k_sign * s.k_exp[k]);
      if (bad && !(fabs(v) < limit)) bad[blockIdx.z * max_batch + row] = 1;
      // |v scale| <= 2^54: adding 128 to every digit makes the bytes of the sum the digits plus 128
      const unsigned long long y = (unsigned long long)__double2ll_rn(v * scale) + 0x0080808080808080ull;
      lo[i] = (unsigned int)y;
      hi[i] = (unsigned int)(y >> 32);
    }
    auto bytes = [](const unsigned int (&v)[4], unsigned int (&b)[4]) {  // b[n] = byte n of the four values
      const unsigned int t0 = __byte_perm(v[0], v[1], 0x5140), t1 = __byte_perm(v[2], v[3], 0x5140);
      const unsigned int t2 = __byte_perm(v[0], v[1], 0x7362), t3 = __byte_perm(v[2], v[3], 0x7362);
      b[0] = __byte_perm(t0, t1, 0x5410) ^ 0x80808080u;
      b[1] = __byte_perm(t0, t1, 0x7632) ^ 0x80808080u;
      b[2] = __byte_perm(t2, t3, 0x5410) ^ 0x80808080u;
      b[3] = __byte_perm(t2, t3, 0x7632) ^ 0x80808080u;
    };
    unsigned int bl[4], bh[4];
    bytes(lo, bl);
    bytes(hi, bh);
#pragma unroll
    for (int n = 0; n < 4; ++n) w[6 - n][g] = bl[n];
#pragma unroll
    for (int n = 0; n < 3; ++n) w[2 - n][g] = bh[n];
  }
  unsigned char* blk =
      dst + ((rb0 + blockIdx.z * rb_batch + blockIdx.y) * dst_k_blocks + kb0 + blockIdx.x) * (long long)I8_BLOCK +
      kc * (I8_BLOCK / 2) + (r >> 3) * 128 + (r & 7) * 16;
#pragma unroll
  for (int n = 0; n < I8_DIGITS; ++n)
    *reinterpret_cast<uint4*>(blk + n * 1024) = make_uint4(w[n][0], w[n][1], w[n][2], w[n][3]);
}

__global__ void k_i8_diag_exp(const float* __restrict__ U, int* __restrict__ exps, int d) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= d) return;
  const float u = fabsf(U[(long long)k * (d + 1)]);
  int e = 0;
  if (u > 0.0f && u < INFINITY) frexpf(u, &e);
  exps[k] = e;
}
tb_status i8_diag_exp(const float* U, int* exps, int d, cudaStream_t st) {
  k_i8_diag_exp<<<(d + 255) / 256, 256, 0, st>>>(U, exps, d);
  TB_LAUNCH_CHECK();
  return TB_OK;
}

tb_status i8_row_max(const I8Src& s, unsigned long long* max_bits, long long max_batch, cudaStream_t st) {
  if (s.rows <= 0 || s.K <= 0) return TB_OK;
  if (s.n_batch == 1)
    TB_CUDA_CHECK(cudaMemsetAsync(max_bits, 0, (size_t)s.rows * 8, st));
  else
    TB_CUDA_CHECK(cudaMemset2DAsync(max_bits, (size_t)max_batch * 8, 0, (size_t)s.rows * 8, s.n_batch, st));
  if (s.k_contig) {
    const dim3 g((s.rows + 7) / 8, (s.K + 511) / 512, s.n_batch);
    if (s.is_float)
      k_i8_row_max<float, true><<<g, 256, 0, st>>>(s, max_bits, max_batch);
    else
      k_i8_row_max<double, true><<<g, 256, 0, st>>>(s, max_bits, max_batch);
  } else {
    const dim3 g((s.rows + 31) / 32, (s.K + 127) / 128, s.n_batch);
    if (s.is_float)
      k_i8_row_max<float, false><<<g, 256, 0, st>>>(s, max_bits, max_batch);
    else
      k_i8_row_max<double, false><<<g, 256, 0, st>>>(s, max_bits, max_batch);
  }
  TB_LAUNCH_CHECK();
  return TB_OK;
}

tb_status i8_slice(const I8Src& s, const unsigned long long* max_bits, long long max_batch, int fixed_exp,
                   const I8Mat& dst, long long rb0, long long rb_batch, int kb0, cudaStream_t st, int* bad) {
  if (s.rows <= 0 || s.K <= 0) return TB_OK;
  const size_t es = s.is_float ? 4 : 8;
  if (s.k_contig && (!aligned(s.X, 16) || (s.ld * es) % 16 || (s.batch * es) % 16)) return TB_ERR_INVALID_ARG;
  const dim3 g((s.K + 31) / 32, (s.rows + 63) / 64, s.n_batch);
  if (s.is_float) {
    if (s.k_contig)
      k_i8_slice<float, true><<<g, 128, 0, st>>>(s, max_bits, max_batch, fixed_exp, dst.data, dst.k_blocks, rb0, rb_batch, kb0, bad);
    else
      k_i8_slice<float, false><<<g, 128, 0, st>>>(s, max_bits, max_batch, fixed_exp, dst.data, dst.k_blocks, rb0, rb_batch, kb0, bad);
  } else {
    if (s.k_contig)
      k_i8_slice<double, true><<<g, 128, 0, st>>>(s, max_bits, max_batch, fixed_exp, dst.data, dst.k_blocks, rb0, rb_batch, kb0, bad);
    else
      k_i8_slice<double, false><<<g, 128, 0, st>>>(s, max_bits, max_batch, fixed_exp, dst.data, dst.k_blocks, rb0, rb_batch, kb0, bad);
  }
  TB_LAUNCH_CHECK();
  return TB_OK;
}

// ------------------------------------------------------------------------------------------ the product

__device__ __forceinline__ uint32_t i8_idesc(uint32_t n) {  // D = s32, A = B = s8, M = 128
  return (2u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ void i8_tma(uint32_t dst, const CUtensorMap* map, int rb, int kb, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(
          dst),
      "l"(map), "r"(0), "r"(rb), "r"(0), "r"(kb), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void i8_tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void i8_ld4(const double* p, double& a, double& b, double& c, double& d) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(p));
}
__device__ __forceinline__ void i8_st4(double* p, double a, double b, double c, double d) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
}

struct I8K {
  double* C;
  float* Cf;
  long long ldc, c_batch;
  const unsigned long long *a_max, *b_max;
  long long a_max_batch, b_max_batch;
  long long a_rb, b_rb, a_rb_batch, b_rb_batch;
  int a_kb, b_kb, k_blocks, a_exp, b_exp;
  int M, N, tiles_m, tiles_n, tiles_per_matrix, n_tiles;
  int negate, add, zeros, order;
};

__device__ __forceinline__ void i8_tile(const I8K& p, int t, int& batch, int& tm, int& tn) {
  batch = t / p.tiles_per_matrix;
  int i = t % p.tiles_per_matrix;
  if (p.zeros & 4) {
    // row tile tm has min(tiles_n, 2 tm + 2) tiles; the rows up to q - 1 are not yet full
    const int q = p.tiles_n / 2, head = q * (q + 1);
    if (i < head) {
      tm = (int)((sqrtf(4.0f * (float)i + 1.0f) - 1.0f) * 0.5f);
      while (tm * (tm + 1) > i) --tm;
      while ((tm + 1) * (tm + 2) <= i) ++tm;
      tn = i - tm * (tm + 1);
    } else {
      tm = q + (i - head) / p.tiles_n;
      tn = (i - head) % p.tiles_n;
    }
  } else if (p.order == 1) {
    tn = i / p.tiles_m;
    tm = i % p.tiles_m;
  } else {
    tm = i / p.tiles_n;
    tn = i % p.tiles_n;
    if (p.order == 2) tm = p.tiles_m - 1 - tm;
  }
}
__device__ __forceinline__ void i8_k_range(const I8K& p, int tm, int tn, int& kb, int& ke) {
  kb = 0;
  ke = p.k_blocks;
  if (p.zeros & 1) ke = min(ke, (tm + 1) * (I8_BM / I8_KB));
  if (p.zeros & 8) ke = min(ke, (tn + 1) * (I8_BN / I8_KB));
  if (p.zeros & 2) kb = tn * (I8_BN / I8_KB);
  if (p.zeros & 16) kb = max(kb, tm * (I8_BM / I8_KB));
  kb = min(kb, ke);
}

__global__ void __launch_bounds__(I8_THREADS, 1) k_i8_gemm(const I8K p, const __grid_constant__ CUtensorMap map_a,
                                                           const __grid_constant__ CUtensorMap map_b) {
  extern __shared__ unsigned char i8_raw[];
  const uint32_t raw = smem_u32(i8_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint64_t* bars = reinterpret_cast<uint64_t*>(i8_raw + (base - raw) + I8_STAGES * I8_STAGE_BYTES);
  // full, empty per stage, then accumulators full / empty, then the TMEM address and the abort flag
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * I8_STAGES + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (I8_STAGES + s); };
  const uint32_t accf_bar = bar0 + 8u * (2 * I8_STAGES), acce_bar = accf_bar + 8u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < I8_STAGES; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(accf_bar, 1);
    mbar_init(acce_bar, I8_EPI);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == I8_EPI) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == I8_EPI) {
    if (lane == 0) {
      uint32_t it = 0;
      for (int t = blockIdx.x; t < p.n_tiles && !*abort_flag; t += gridDim.x) {
        int b, tm, tn, kb, ke;
        i8_tile(p, t, b, tm, tn);
        i8_k_range(p, tm, tn, kb, ke);
        const int rb_a = (int)(p.a_rb + b * p.a_rb_batch) + 2 * tm, rb_b = (int)(p.b_rb + b * p.b_rb_batch) + tn;
        for (int k = kb; k < ke; ++k, ++it) {
          const int s = it % I8_STAGES;
          if (!mbar_wait(empty_bar(s), ((it / I8_STAGES) & 1u) ^ 1u, abort_flag, &g_i8_error)) break;
          mbar_expect_tx(full_bar(s), I8_STAGE_BYTES);
          i8_tma(base + s * I8_STAGE_BYTES, &map_a, rb_a, p.a_kb + k, full_bar(s));
          i8_tma(base + s * I8_STAGE_BYTES + I8_A_BYTES, &map_b, rb_b, p.b_kb + k, full_bar(s));
        }
      }
    }
  } else if (warp == I8_EPI + 1) {
    if (lane == 0) {
      uint32_t it = 0, tile_it = 0;
      for (int t = blockIdx.x; t < p.n_tiles && !*abort_flag; t += gridDim.x, ++tile_it) {
        int b, tm, tn, kb, ke;
        i8_tile(p, t, b, tm, tn);
        i8_k_range(p, tm, tn, kb, ke);
        if (!mbar_wait(acce_bar, (tile_it & 1u) ^ 1u, abort_flag, &g_i8_error)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        bool ok = true;
        for (int k = kb; k < ke; ++k, ++it) {
          const int s = it % I8_STAGES;
          if (!mbar_wait(full_bar(s), (it / I8_STAGES) & 1u, abort_flag, &g_i8_error)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = base + s * I8_STAGE_BYTES, sb = sa + I8_A_BYTES;
#pragma unroll
          for (int i = 0; i < I8_DIGITS; ++i) {
            const int n = I8_BN * (I8_DIGITS - i);
            const uint64_t a = smem_desc_k(sa + i * 2048, I8_A_BYTES / 2);
            const uint32_t acc = (k > kb || i > 0) ? 1u : 0u;
            umma_i8(tmem + I8_BN * i, a, smem_desc_k(sb, I8_B_BYTES / 2), i8_idesc(n > 256 ? 256 : n), acc);
            if (n > 256)
              umma_i8(tmem + I8_BN * i + 256, a, smem_desc_k(sb + 4 * 1024, I8_B_BYTES / 2), i8_idesc(n - 256), acc);
          }
          umma_commit(empty_bar(s));
        }
        if (!ok) break;
        umma_commit(accf_bar);
      }
    }
  } else {
    // epilogue warps: TMEM lanes 32 (w % 4) .., columns 16 (w / 4) .. of every accumulator
    const int q = warp & 3, hf = warp >> 2;
    const int row = q * 32 + lane;
    uint32_t tile_it = 0;
    for (int t = blockIdx.x; t < p.n_tiles && !*abort_flag; t += gridDim.x, ++tile_it) {
      int b, tm, tn, kb, ke;
      i8_tile(p, t, b, tm, tn);
      i8_k_range(p, tm, tn, kb, ke);
      const int m = tm * I8_BM + row, n0 = tn * I8_BN + hf * 16;
      const bool in_m = m < p.M;
      const long long at = b * p.c_batch + (in_m ? m : 0) * p.ldc + n0;
      double* c = p.C + at;
      // while the products run: the old values, and the scales of the row and (a lane each) of the columns
      double o[16];
#pragma unroll
      for (int j = 0; j < 16; j += 4) {  // N is a multiple of 4
        o[j] = o[j + 1] = o[j + 2] = o[j + 3] = 0.0;
        if (p.add && in_m && n0 + j < p.N) i8_ld4(c + j, o[j], o[j + 1], o[j + 2], o[j + 3]);
      }
      double sa = (p.a_max && in_m) ? i8_result_scale(p.a_max[b * p.a_max_batch + m]) : pow2d(p.a_exp - 54 + 24);
      const double sb_mine = (p.b_max && lane < 16 && n0 + lane < p.N) ? i8_result_scale(p.b_max[b * p.b_max_batch + n0 + lane])
                                                                       : pow2d(p.b_exp - 54 + 24);
      if (p.negate) sa = -sa;
      if (!mbar_wait(accf_bar, tile_it & 1u, abort_flag, &g_i8_error)) break;
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (ke > kb) {  // otherwise the accumulators were not written
        const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hf * 16);
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          uint32_t r[I8_DIGITS][8];
#pragma unroll
          for (int s = 0; s < I8_DIGITS; ++s) i8_tmem_ld8(ta + I8_BN * s + 8 * g, r[s]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            // sum of acc_s 256^(6 - s), exact in two 64-bit integers
            long long hi = (int)r[0][j], lo = (int)r[4][j];
            hi = hi * 256 + (int)r[1][j];
            hi = hi * 256 + (int)r[2][j];
            hi = hi * 256 + (int)r[3][j];
            lo = lo * 256 + (int)r[5][j];
            lo = lo * 256 + (int)r[6][j];
            const double v = fma((double)hi, 16777216.0, (double)lo);
            const double sb = __shfl_sync(0xffffffffu, sb_mine, 8 * g + j);
            o[8 * g + j] = fma(v * sa, sb, o[8 * g + j]);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acce_bar);  // the accumulators may be overwritten
      if (!in_m) continue;
      if (p.Cf) {
#pragma unroll
        for (int j = 0; j < 16; j += 4)
          if (n0 + j < p.N)
            *reinterpret_cast<float4*>(p.Cf + at + j) =
                make_float4((float)o[j], (float)o[j + 1], (float)o[j + 2], (float)o[j + 3]);
        continue;
      }
#pragma unroll
      for (int j = 0; j < 16; j += 4)
        if (n0 + j < p.N) i8_st4(c + j, o[j], o[j + 1], o[j + 2], o[j + 3]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == I8_EPI) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

static tb_status i8_map(CUtensorMap* map, const I8Mat& m, unsigned box_blocks) {
  EncodeTiledFn enc = encode_tiled_fn();
  if (!enc) return TB_ERR_CUDA;
  // 128 doubles = one digit of 64 rows x 16 steps; row blocks; 14 (half, digit) pairs; k blocks
  const cuuint64_t dims[4] = {128, (cuuint64_t)m.row_blocks, 14, (cuuint64_t)m.k_blocks};
  const cuuint64_t strides[3] = {(cuuint64_t)m.k_blocks * I8_BLOCK, 1024, I8_BLOCK};
  const cuuint32_t box[4] = {128, box_blocks, 14, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  if (enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, m.data, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return TB_ERR_CUDA;
  return TB_OK;
}

tb_status i8_gemm(const I8Gemm& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.n_batch <= 0) return TB_OK;
  // vectors of four doubles on C
  if (g.N % 4 || g.ldc % 4 || g.c_batch % 4 || !aligned(g.C, 32) || !aligned(g.Cf, 16) || (g.Cf && g.beta != 0.0) || g.k_blocks > I8_MAX_K_BLOCKS) return TB_ERR_INVALID_ARG;
  CUtensorMap ma, mb;
  TB_TRY(i8_map(&ma, g.A, 2));
  TB_TRY(i8_map(&mb, g.B, 1));
  I8K p;
  p.C = g.C;
  p.Cf = g.Cf;
  p.ldc = g.ldc;
  p.c_batch = g.c_batch;
  p.a_max = g.a_max;
  p.b_max = g.b_max;
  p.a_max_batch = g.a_max_batch;
  p.b_max_batch = g.b_max_batch;
  p.a_rb = g.a_rb;
  p.b_rb = g.b_rb;
  p.a_rb_batch = g.a_rb_batch;
  p.b_rb_batch = g.b_rb_batch;
  p.a_kb = g.a_kb;
  p.b_kb = g.b_kb;
  p.k_blocks = g.k_blocks;
  p.a_exp = g.a_exp;
  p.b_exp = g.b_exp;
  p.M = g.M;
  p.N = g.N;
  p.tiles_m = (g.M + I8_BM - 1) / I8_BM;
  p.tiles_n = (g.N + I8_BN - 1) / I8_BN;
  long long per = (long long)p.tiles_m * p.tiles_n;
  if (g.zeros & 4) {
    const long long q = p.tiles_n / 2;
    per = (p.tiles_m <= q) ? (long long)p.tiles_m * (p.tiles_m + 1) : q * (q + 1) + (p.tiles_m - q) * p.tiles_n;
  }
  if (per * g.n_batch > 0x7fffffffll) return TB_ERR_UNSUPPORTED;
  p.tiles_per_matrix = (int)per;
  p.n_tiles = (int)(per * g.n_batch);
  p.negate = g.alpha < 0.0;
  p.add = g.beta != 0.0;
  p.zeros = g.zeros;
  p.order = g.order;
  static bool configured[64] = {false};
  TB_TRY(allow_smem(k_i8_gemm, I8_SMEM, configured));
  const int sms = 148;
  const int rounds = (p.n_tiles + sms - 1) / sms;
  // as many CTAs as fill the rounds of tiles evenly, unless the tiles differ in length
  int grid = (g.zeros & ~4) ? (p.n_tiles < sms ? p.n_tiles : sms) : (p.n_tiles + rounds - 1) / rounds;
  // short-lived CTAs: a kernel of higher priority gets SMs soon
  if (g.tiles_per_cta > 0 && rounds > g.tiles_per_cta) grid = (p.n_tiles + g.tiles_per_cta - 1) / g.tiles_per_cta;
  k_i8_gemm<<<grid, I8_THREADS, I8_SMEM, st>>>(p, ma, mb);
  TB_LAUNCH_CHECK();
  return TB_OK;
}

}  // namespace tb
