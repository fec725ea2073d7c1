// Shared host/device helpers of the TurboBoA CUDA library (sm_100a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "turboboa.h"

// A failed runtime call leaves its code in the runtime's last-error slot; it is cleared here so
// that the next, unrelated launch check does not report it again.
#define TB_CUDA_CHECK(expr)                      \
  do {                                           \
    cudaError_t tb_e_ = (expr);                  \
    if (tb_e_ != cudaSuccess) {                  \
      (void)cudaGetLastError();                  \
      return TB_ERR_CUDA;                        \
    }                                            \
  } while (0)

// Follows every kernel launch of the library (one check per launch); also counts them.
#define TB_LAUNCH_CHECK()                                   \
  do {                                                      \
    ++tb::g_launch_count;                                   \
    if (cudaGetLastError() != cudaSuccess) return TB_ERR_CUDA; \
  } while (0)

#define TB_TRY(expr)                   \
  do {                                 \
    tb_status tb_s_ = (expr);          \
    if (tb_s_ != TB_OK) return tb_s_;  \
  } while (0)

namespace tb {

extern unsigned long long g_launch_count;  // kernels launched by the library in this process (tb_api.cu)

// Bump allocator over a caller-provided workspace.  With base == nullptr it
// only measures (used by the *_workspace queries), so sizes and carving can
// never disagree.
struct Bump {
  char* base;
  size_t off;
  explicit Bump(void* b) : base(static_cast<char*>(b)), off(0) {}
  template <typename T>
  T* take(size_t n) {
    off = (off + 255) & ~static_cast<size_t>(255);
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += n * sizeof(T);
    return p;
  }
  size_t total() const { return (off + 255) & ~static_cast<size_t>(255); }
};

inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

// Short kernels that follow one another (a step's grid search, sweep, update and compensation) are launched so that the next
// one's CTAs start while the last of the one before still run (programmatic dependent launch).  Every kernel launched this
// way calls pdl_wait() before it touches anything that an earlier kernel writes or reads back (it returns when the kernel
// before has completed, which waited in turn), and pdl_trigger() shortly before its end: earlier, the next kernel's CTAs
// would hold places that another stream's kernels could use.  (k_rank_rows calls it earlier where the
// next kernel's CTAs leave half of the SMs free: that one may then start before the kernel before this one has ended, and has
// to wait for all it did not find at the call's start.)  None of their parameters is `const __restrict__`, and __ldg is
// for what the whole call leaves alone (U, P): both promise that the data does not change while the kernel lives, which
// here begins before the kernel that writes it has ended, and free the compiler to load it ahead of the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// One FP64 tensor step: c (8 x 8, two entries of a lane) += a (8 x 4) b (4 x 8); lane: row / column lane / 4, k lane % 4, entries
// of c at columns 2 (lane % 4), + 1.
__device__ __forceinline__ void dmma(double (&c)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(c[0]), "+d"(c[1])
               : "d"(a), "d"(b));
}
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }  // -1022 .. 1023

inline cudaStream_t as_stream(void* s) { return static_cast<cudaStream_t>(s); }

template <typename TO, typename TI>
__device__ __forceinline__ TO cvt(TI v) {
  return static_cast<TO>(v);
}
template <>
__device__ __forceinline__ float cvt<float, __nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <>
__device__ __forceinline__ double cvt<double, __nv_bfloat16>(__nv_bfloat16 v) {
  return static_cast<double>(__bfloat162float(v));
}

template <typename T>
__device__ __forceinline__ T zero_of() {
  return T(0);
}
template <>
__device__ __forceinline__ __nv_bfloat16 zero_of<__nv_bfloat16>() {
  return __float2bfloat16(0.0f);
}

__device__ __forceinline__ double shfl_d(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Round to nearest integer, ties to even, for |x| < 2^51 (two full-rate adds).
__device__ __forceinline__ double rne(double x) {
  const double magic = 6755399441055744.0;  // 1.5 * 2^52
  return __dadd_rn(__dadd_rn(x, magic), -magic);
}

}  // namespace tb
