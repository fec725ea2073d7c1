// A candidate grid of the search and the codes and errors on it, shared by the search kernels.
#pragma once

#include "tb_common.cuh"

namespace tb {

__device__ __forceinline__ void gw_candidate(double2 mnmx, int k, int maxq, double* s_out, double* z_out) {
  const double pk = 1.0 - (double)k / 32.0;
  const double lo = pk * mnmx.x, hi = pk * mnmx.y;
  double s = 1.0, z = 0.0;
  if (hi != lo) {
    s = (hi - lo) / (double)maxq;
    z = fmin(fmax(rne(-lo / s), 0.0), (double)maxq);
  }
  *s_out = s;
  *z_out = z;
}

// The fused multiply-add into zm = z + 1.5 * 2^52 rounds to nearest-even and leaves the integer in the low
// word (|w / s + z| < 2^31), where the clamp is one integer instruction
__device__ __forceinline__ int gw_code(double w, double rs, double zm, int maxq) {
  return __vimin_s32_relu(__double2loint(fma(w, rs, zm)), maxq);
}
__device__ __forceinline__ double gw_error(double w, double s, double rs, double z, int maxq) {
  const double magic = 6755399441055744.0;
  return w - s * ((__hiloint2double(0x43380000, gw_code(w, rs, z + magic, maxq)) - magic) - z);
}

}  // namespace tb
