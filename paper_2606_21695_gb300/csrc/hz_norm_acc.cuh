// Sums of squares for the WaveHoltz stopping test, ||u^{m+1} - u^m||^2 and
// ||u^{m+1}||^2, of a thread's FP32 iterates without the FP64 pipe (a
// conversion or an addition there takes a warp as long as 64 FP32
// instructions).  Each sum is three floats, hi + mid + lo, to which squares are
// added by error-free transformations (Dekker, Knuth: FMA products and
// two-sums); what is rounded off is below 2^-48 of a term and is itself added
// in FP32, so a sum of up to 128 squares is good to about 2^-65 of its value and
// becomes FP64 once per thread.  FP64 sums round to 2^-53 at every addition.
// Entries are scaled by a power of two to the largest of the thread's entries,
// old and new, so that nothing overflows; what underflows is below 2^-140 of
// the largest entry's square.
// 64 subdomains of 129 x 129 nodes, P = 4, WaveHoltz to 1e-4: 7.3 ms with FP64
// sums, 5.2 ms; 1024 of 25 x 25, P = 3, N_t = 37: 1040 us, 944 us (two floats, 2^-46:
// 5.2 ms, 867 us).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

namespace hz {
namespace norm_acc {

// Two entries at a time: the packed instructions halve the issue slots and the
// code (which a warp runs once per iteration, out of the instruction cache's
// reach).  Every operation is rounded (host: compile without contraction).
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma3(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ unsigned bits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ float from_bits(unsigned b) { return __uint_as_float(b); }
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }
#else
inline float2 add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
inline float2 sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
inline float2 mul(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
inline float2 fma3(float2 a, float2 b, float2 c) { return make_float2(std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y)); }
inline unsigned bits(float x) {
  unsigned b;
  std::memcpy(&b, &x, 4);
  return b;
}
inline float from_bits(unsigned b) {
  float x;
  std::memcpy(&x, &b, 4);
  return x;
}
inline double pow2(int e) { return std::ldexp(1.0, e); }
#endif
__host__ __device__ __forceinline__ float2 twice(float2 a) { return add(a, a); }
__host__ __device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }

// a + b = the returned sum + err, exactly
__host__ __device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2& err) {
  const float2 t = add(a, b), z = sub(t, a);
  err = add(sub(a, sub(t, z)), sub(b, z));
  return t;
}

struct ThreeFloat {
  float2 hi = {0.f, 0.f}, mid = {0.f, 0.f}, lo = {0.f, 0.f};
  __host__ __device__ __forceinline__ void add_second(float2 s) {  // a term of the second order
    float2 e;
    mid = two_sum(mid, s, e);
    lo = add(lo, e);
  }
  // += x^2
  __host__ __device__ __forceinline__ void add_square(float2 x) {
    const float2 p = mul(x, x), e = fma3(x, x, neg(p));  // x^2 = p + e
    float2 c, d;
    hi = two_sum(hi, p, c);
    add_second(two_sum(c, e, d));
    lo = add(lo, d);
  }
  // += (x + r)^2, |r| <= half a unit in the last place of x
  __host__ __device__ __forceinline__ void add_square(float2 x, float2 r) {
    add_square(x);
    const float2 x2 = twice(x), q = mul(x2, r), e = fma3(x2, r, neg(q));
    add_second(q);
    lo = add(lo, fma3(r, r, e));
  }
  __host__ __device__ __forceinline__ double value() const {  // of both
    float2 e;
    const float2 t = two_sum(hi, make_float2(hi.y, hi.x), e);  // its first entries
    return (double)t.x + (((double)mid.x + (double)mid.y) + ((double)e.x + (double)(lo.x + lo.y)));
  }
};

}  // namespace norm_acc

struct NormAcc {
  float2 scale = {1.f, 1.f};
  int exp = 127;
  norm_acc::ThreeFloat d, u;
  // largest: the largest |entry| of the thread's new and old iterate
  __host__ __device__ __forceinline__ void start(float largest) {
    const unsigned e = norm_acc::bits(largest) >> 23;
    exp = e < 253u ? (int)e : 253;
    scale.x = scale.y = norm_acc::from_bits((unsigned)(254 - exp) << 23);  // 2^(127 - exp)
  }
  __host__ __device__ __forceinline__ void add(float2 now, float2 before) {
    const float2 a = norm_acc::mul(now, scale), b = norm_acc::mul(before, scale);
    float2 r;
    const float2 x = norm_acc::two_sum(a, norm_acc::neg(b), r);  // a - b = x + r
    d.add_square(x, r);
    u.add_square(a);
  }
  __host__ __device__ __forceinline__ void finish(double& dn, double& un) const {
    const double f = norm_acc::pow2(2 * (exp - 127));
    dn = d.value() * f;
    un = u.value() * f;
  }
};

}  // namespace hz
