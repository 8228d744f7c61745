// Complex entries of the caller's arrays.  The C ABI takes plain double
// pointers, which promise 8-byte alignment and no more (a contiguous view at
// an odd offset of a double buffer is valid), and a 16-byte access to an
// address that is not a multiple of 16 ends the CUDA context.  So an entry is
// read and written as two doubles, or, where the pair access pays (kernels
// that move every entry of such an array once per few FP64 instructions), as
// a pair in an instantiation that the launch chooses by is_pair_aligned.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace hz {

template <bool PAIR = false>
__device__ __forceinline__ double2 load_complex(const double* p, int64_t k) {
  if constexpr (PAIR) return reinterpret_cast<const double2*>(p)[k];
  else return make_double2(p[2 * k], p[2 * k + 1]);
}
template <bool PAIR = false>  // of an array that the kernel does not write
__device__ __forceinline__ double2 load_complex_ro(const double* p, int64_t k) {
  if constexpr (PAIR) return __ldg(reinterpret_cast<const double2*>(p) + k);
  else return make_double2(__ldg(p + 2 * k), __ldg(p + 2 * k + 1));
}
template <bool PAIR = false>
__device__ __forceinline__ void store_complex(double* p, int64_t k, double2 v) {
  if constexpr (PAIR) {
    reinterpret_cast<double2*>(p)[k] = v;
  } else {
    p[2 * k] = v.x;
    p[2 * k + 1] = v.y;
  }
}
inline bool is_pair_aligned(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

}  // namespace hz
