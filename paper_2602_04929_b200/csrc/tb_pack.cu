// Bit-packed storage of the integer weights W_int in {0 .. 2^b - 1} (Section 2.1:
// Q = diag(s) W_int) and the fused unpack + dequantize + compare.
//
// Format: every row is a little-endian bit stream, code j of the row in bits
// [j b, (j + 1) b) counted from the least significant bit of 32-bit word 0; rows
// are d_in * b / 32 words long (d_in is a multiple of 32, so rows end on a word
// boundary).  A code may straddle two words when b does not divide 32.
//
// Rows end on a word, so the whole matrix is one bit stream, and a column group divides its row, so element e of
// the matrix has the scale e / quant_group.  Both kernels are pure data movement, bound by HBM and, once the accesses
// are contiguous, nearly by the instructions per code.  Packing: a lane loads 16 codes, joins them four
// at a time, and its BITS half-words go through shared memory.  Unpacking: a lane makes eight values, one 32-byte
// store; the words it needs are its neighbours' too and come from L1.  (A thread per 32 codes touched 32 lines with
// every 16-byte store.)  4096 x 4096, 3 bits: packing 6.6 -> 6.4 us (8 bits: 21 -> 7.6), unpacking into float 25.5 -> 14.5
// (the bytes alone: 3.5 and 11.3).
#include "tb_common.cuh"

namespace tb {

constexpr int PACK_PER = 2;    // pieces of 512 codes a warp has in flight
constexpr int UNPACK_PER = 2;  // pieces of 256 values

template <int BITS>
__global__ void __launch_bounds__(256) k_pack_codes(const unsigned char* __restrict__ codes,
                                                    unsigned int* __restrict__ packed, long long n) {
  __shared__ __align__(16) unsigned short stage[8][PACK_PER * 32 * BITS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // n is a multiple of 32: 16 codes are inside together
  const long long e0 = (blockIdx.x * 8ll + warp) * (512 * PACK_PER);
  if (e0 >= n) return;
  const int left = n - e0 < 512 * PACK_PER ? (int)(n - e0) : 512 * PACK_PER;
  uint4 a[PACK_PER];
#pragma unroll
  for (int k = 0; k < PACK_PER; ++k)
    a[k] = 512 * k + 16 * lane < left ? __ldcs(reinterpret_cast<const uint4*>(codes + e0 + 512 * k + 16 * lane))
                                      : make_uint4(0, 0, 0, 0);
#pragma unroll
  for (int k = 0; k < PACK_PER; ++k) {
    const unsigned int w4[4] = {a[k].x, a[k].y, a[k].z, a[k].w};
    constexpr unsigned int M = ((1u << BITS) - 1u) * 0x01010101u;
    unsigned long long acc = 0;  // bits of the stream not yet written
    int have = 0, o = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned int x = w4[i] & M;
      const unsigned int y = (x & 0x00ff00ffu) | ((x & 0xff00ff00u) >> (8 - BITS));
      const unsigned int z = (y & 0xffffu) | ((y & 0xffff0000u) >> (16 - 2 * BITS));  // four codes, 4 BITS bits
      acc |= (unsigned long long)z << have;
      have += 4 * BITS;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (have >= 16) {
          stage[warp][(32 * k + lane) * BITS + o++] = (unsigned short)acc;
          acc >>= 16;
          have -= 16;
        }
    }
  }
  __syncwarp();
  const int words = left / 32 * BITS;
  unsigned int* dst = packed + e0 / 32 * BITS;
  const unsigned int* src = reinterpret_cast<const unsigned int*>(stage[warp]);
#pragma unroll
  for (int i = 0; i < PACK_PER * 16 * BITS; i += 32)
    if (i + lane < words) dst[i + lane] = src[i + lane];
}

struct UnpackP {
  const unsigned int* packed;
  const float* scales;
  const int* zeros;
  unsigned char* codes_out;
  float* what_out;
  const unsigned char* codes_ref;
  const float* what_ref;
  unsigned long long* mismatch;  // [0] codes that differ from codes_ref, [1] values beyond tol of what_ref
  long long n;
  unsigned long long seg_inv;  // ceil(2^64 / (seg / 32)), 0 for groups of 32 columns
  int wide;                    // W_hat_out is 32-byte aligned
  float tol;
};

template <int BITS>
__global__ void __launch_bounds__(256) k_unpack_dequant(UnpackP p) {
  unsigned int bad_codes = 0, bad_vals = 0;
  const int lane = threadIdx.x & 31;
  const long long w0 = (blockIdx.x * 8ll + (threadIdx.x >> 5)) * (256 * UNPACK_PER);
#pragma unroll
  for (int k = 0; k < UNPACK_PER; ++k) {
    const long long e = w0 + 256 * k + 8 * lane;
    if (e >= p.n) break;  // n is a multiple of 32: eight elements are inside together
    // (e / 32) / (seg / 32): exact while their product stays below 2^64
    const unsigned long long e32 = (unsigned long long)e >> 5;
    const long long so = p.seg_inv ? (long long)__umul64hi(e32, p.seg_inv) : (long long)e32;
    const float s = __ldg(p.scales + so);
    const int z = __ldg(p.zeros + so);
    const long long bit = e * BITS;
    const unsigned int* src = p.packed + (bit >> 5);
    const int sh = (int)bit & 31;
    // the 8 BITS bits in lo, hi: they start on a byte and span up to three words
    const unsigned int x0 = __ldg(src);
    const unsigned int x1 = sh + 8 * BITS > 32 ? __ldg(src + 1) : 0u;
    const unsigned int x2 = sh + 8 * BITS > 64 ? __ldg(src + 2) : 0u;
    const unsigned int lo = __funnelshift_r(x0, x1, sh), hi = __funnelshift_r(x1, x2, sh);
    unsigned int out[2] = {0, 0};
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      constexpr unsigned int M = (1u << BITS) - 1u;
      const int b = i * BITS;
      const unsigned int c = (b >= 32 ? hi >> (b & 31) : b + BITS <= 32 ? lo >> (b & 31) : __funnelshift_r(lo, hi, b & 31)) & M;
      out[i >> 2] |= c << (8 * (i & 3));
      v[i] = s * (float)((int)c - z);
    }
    if (p.codes_out) *reinterpret_cast<uint2*>(p.codes_out + e) = make_uint2(out[0], out[1]);
    if (p.codes_ref) {
      const uint2 r = *reinterpret_cast<const uint2*>(p.codes_ref + e);
      const unsigned int x[2] = {r.x ^ out[0], r.y ^ out[1]};
#pragma unroll
      for (int i = 0; i < 2; ++i)
        bad_codes += ((x[i] & 0xffu) != 0) + ((x[i] & 0xff00u) != 0) + ((x[i] & 0xff0000u) != 0) + ((x[i] & 0xff000000u) != 0);
    }
    if (p.what_out) {
      float* dst = p.what_out + e;
      if (p.wide) {
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                     "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                     : "memory");
      } else {
        reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
      }
    }
    if (p.what_ref) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 r = reinterpret_cast<const float4*>(p.what_ref + e)[h];
        const float rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          // !(<=) so that a NaN on either side counts as a deviation
          if (!(fabsf(v[4 * h + i] - rr[i]) <= p.tol * fabsf(rr[i]))) ++bad_vals;
      }
    }
  }
  if (p.mismatch) {
    bad_codes = __reduce_add_sync(0xffffffffu, bad_codes);
    bad_vals = __reduce_add_sync(0xffffffffu, bad_vals);
    if ((threadIdx.x & 31) == 0) {
      if (bad_codes) atomicAdd(&p.mismatch[0], (unsigned long long)bad_codes);
      if (bad_vals) atomicAdd(&p.mismatch[1], (unsigned long long)bad_vals);
    }
  }
}

}  // namespace tb

using namespace tb;

extern "C" size_t tb_packed_bytes(int d_out, int d_in, int bits) {
  if (d_out <= 0 || d_in <= 0 || (d_in % 32) || bits < 2 || bits > 8) return 0;
  return (size_t)d_out * (size_t)(d_in / 32) * (size_t)bits * sizeof(unsigned int);
}

extern "C" tb_status tb_pack_codes(const unsigned char* codes, int d_out, int d_in, int bits, unsigned int* packed,
                                   void* stream) {
  if (!codes || !packed || d_out <= 0 || d_in <= 0 || bits < 2 || bits > 8) return TB_ERR_INVALID_ARG;
  if (d_in % 32) return TB_ERR_UNSUPPORTED;
  if (!aligned(codes, 16) || !aligned(packed, 4)) return TB_ERR_INVALID_ARG;
  const long long n = (long long)d_out * d_in;
  cudaStream_t st = as_stream(stream);
  const unsigned nb = (unsigned)((n + 4096 * PACK_PER - 1) / (4096 * PACK_PER));
  switch (bits) {
    case 2: k_pack_codes<2><<<nb, 256, 0, st>>>(codes, packed, n); break;
    case 3: k_pack_codes<3><<<nb, 256, 0, st>>>(codes, packed, n); break;
    case 4: k_pack_codes<4><<<nb, 256, 0, st>>>(codes, packed, n); break;
    case 5: k_pack_codes<5><<<nb, 256, 0, st>>>(codes, packed, n); break;
    case 6: k_pack_codes<6><<<nb, 256, 0, st>>>(codes, packed, n); break;
    case 7: k_pack_codes<7><<<nb, 256, 0, st>>>(codes, packed, n); break;
    default: k_pack_codes<8><<<nb, 256, 0, st>>>(codes, packed, n); break;
  }
  TB_LAUNCH_CHECK();
  return TB_OK;
}

extern "C" tb_status tb_unpack_dequant(const unsigned int* packed, const float* scales, const int* zeros, int d_out,
                                       int d_in, int bits, int quant_group, unsigned char* codes_out,
                                       float* W_hat_out, const unsigned char* codes_ref, const float* W_hat_ref,
                                       float tol, unsigned long long* mismatch, void* stream) {
  if (!packed || !scales || !zeros || d_out <= 0 || d_in <= 0 || bits < 2 || bits > 8) return TB_ERR_INVALID_ARG;
  if (quant_group < 0 || (quant_group > 0 && d_in % quant_group)) return TB_ERR_INVALID_ARG;
  if ((d_in % 32) || (quant_group > 0 && quant_group % 32)) return TB_ERR_UNSUPPORTED;
  if ((codes_ref || W_hat_ref) && !mismatch) return TB_ERR_INVALID_ARG;
  if (!(tol >= 0.0f)) return TB_ERR_INVALID_ARG;
  if (!aligned(packed, 4) || !aligned(codes_out, 16) || !aligned(codes_ref, 16) || !aligned(W_hat_out, 16) ||
      !aligned(W_hat_ref, 16))
    return TB_ERR_INVALID_ARG;
  UnpackP p;
  p.packed = packed;
  p.scales = scales;
  p.zeros = zeros;
  p.codes_out = codes_out;
  p.what_out = W_hat_out;
  p.codes_ref = codes_ref;
  p.what_ref = W_hat_ref;
  p.mismatch = mismatch;
  p.n = (long long)d_out * d_in;
  const unsigned long long seg32 = (unsigned)(quant_group > 0 ? quant_group : d_in) / 32;
  p.seg_inv = seg32 > 1 ? ~0ull / seg32 + 1 : 0;
  p.wide = aligned(W_hat_out, 32);
  p.tol = tol;
  cudaStream_t st = as_stream(stream);
  if (mismatch) TB_CUDA_CHECK(cudaMemsetAsync(mismatch, 0, 2 * sizeof(unsigned long long), st));
  const unsigned nb = (unsigned)((p.n + 2048 * UNPACK_PER - 1) / (2048 * UNPACK_PER));
  switch (bits) {
    case 2: k_unpack_dequant<2><<<nb, 256, 0, st>>>(p); break;
    case 3: k_unpack_dequant<3><<<nb, 256, 0, st>>>(p); break;
    case 4: k_unpack_dequant<4><<<nb, 256, 0, st>>>(p); break;
    case 5: k_unpack_dequant<5><<<nb, 256, 0, st>>>(p); break;
    case 6: k_unpack_dequant<6><<<nb, 256, 0, st>>>(p); break;
    case 7: k_unpack_dequant<7><<<nb, 256, 0, st>>>(p); break;
    default: k_unpack_dequant<8><<<nb, 256, 0, st>>>(p); break;
  }
  TB_LAUNCH_CHECK();
  return TB_OK;
}
