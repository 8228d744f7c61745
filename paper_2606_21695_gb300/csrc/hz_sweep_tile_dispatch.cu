// Dispatch of the element-tile sweep over the compiled degrees, and the rules
// by size.
#include <cstdlib>

#include "hz_internal.h"

namespace hz {
namespace tile_sweep {
hz_status tile_f32_p1(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f32_p2(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f32_p3(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f32_p4(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f32_p5(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f64_p1(const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f64_p2(const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f64_p3(const SweepArgs& a, int count, cudaStream_t st, int* warps);
hz_status tile_f64_p4(const SweepArgs& a, int count, cudaStream_t st, int* warps);
}  // namespace tile_sweep

namespace {
// Threads of a subdomain's tiles in the one-element shape.
int one_element_lanes(int sxe, int sye) { return tile_pow2(sxe) * sye; }
}  // namespace

// Two paired elements per tile halve the instructions per node (packed FMAs)
// but leave half the warps: better once one-element tiles fill the SMs'
// resident blocks.  Sweeps of 5 WaveHoltz iterations at 14 node spacings per
// wavelength (N_t = 21, 24, 32, 38 and 44 for P = 1 to 5; all timings of this file, taken before
// fixed-count sweeps had kernels of their own), one / two elements: P = 3, 8 x 8 elements: 40 / 62 us at 9 subdomains, 57 / 63 at 256, 69 / 64 at
// 576, 131 / 104 at 1024; P = 2, 16 x 16: 73 / 55 at 256; P = 3, 32 x 32: 103 /
// 157 at 9, 202 / 157 at 64.  Degrees 1 and 2 gain earlier (P = 2, 12 x 10: 36 /
// 29 at 9, 16 x 16: 38 / 37); P = 4 loses (see launch_tile_f32), and P = 3 where
// the tiles do not fill whole warps (12 x 10 at 1024: 278 / 325).
int tile_shape(bool fp32, int P, int sxe, int sye, int L) {
  if (!fp32 || P > 3 || sye % 2) return 1;
  const int lanes1 = one_element_lanes(sxe, sye), lanes2 = lanes1 / 2;
  if (lanes1 <= 32 && sxe + sye <= 32) return 1;  // one warp either way
  if (P == 1) return 2;
  const int cap = tile_max_threads(false, P, 1) / 32;
  if (P == 2 && lanes2 > 32 && (lanes2 + 31) / 32 + 2 <= cap) return 2;
  if (lanes2 > 32 && lanes2 % 32) return 1;
  const int warps = (lanes1 + 31) / 32 + (sxe + sye + 31) / 32;
  const int ctas = (warps + cap - 1) / cap;           // CTAs per subdomain
  const int res = cap / ((warps + ctas - 1) / ctas);  // and per SM
  return 4LL * L * ctas > 3LL * sm_count() * (res > 0 ? res : 1) ? 2 : 1;
}

// Where the tiles beat the other kernels (5 WaveHoltz iterations, best other
// kernel / tiles).  FP32: nearly everywhere (P = 3, 8 x 8 at 1024 subdomains
// 172 / 104 us; P = 4, 8 x 8 at 64: 157 / 76; P = 4, 32 x 32 at 144: 2145 / 652),
// except
//  - degrees 1 and 2 with many idle lanes and many subdomains (P = 1, 12 x 10
//    at 1024: 50 / 57; P = 2, 5 x 7 at 1024: 70 / 75);
//  - few one-warp subdomains of degree 5, where 25 nodes in a row on one lane
//    are the longer chain (4 x 4, one warp by node columns / tiles: 149 / 177 us
//    at 64, 155 / 178 at 576, 250 / 180 at 1024).
// FP64 (bound by the FP64 pipe; 3 iterations): with a subdomain per SM and
// whole tiles (P = 3, 8 x 8 at 256: 915 / 648, at 64: 466 / 501; P = 4,
// 16 x 16 at 16: 2364 / 1458; P = 3, 32 x 32 at 64: 3905 / 2354).  P = 2 and other
// sye were not timed by themselves: the limits are those of whole tiles per warp.
bool tile_default(bool fp32, int P, int sxe, int sye, int L) {
  if (sxe > 32 || sye > 32 || P > (fp32 ? 5 : 4)) return false;
  const int lanes = one_element_lanes(sxe, sye), sms = sm_count();
  const bool one_warp = lanes / (tile_shape(fp32, P, sxe, sye, L)) <= 32 && sxe + sye <= 32;
  if (!fp32) {
    if (P < 2 || sxe < 8 || sxe != tile_pow2(sxe) || sye % 4) return false;
    return sxe == 32 || (P == 4 && sxe == 16) || L >= sms;
  }
  if (P == 1 && !one_warp && sxe != tile_pow2(sxe)) return false;
  if (P <= 2 && !one_warp && 3 * sxe * sye < 2 * ((lanes + 31) / 32) * 32 && L > 4 * sms) return false;
  if (P == 5 && one_warp && 2 * L <= 9 * sms) return false;
  return true;
}

hz_status launch_sweep_tile(bool fp32, int P, const SweepArgs& a, int count, cudaStream_t st, int* warps, int* elements) {
  if (a.round_mode != 0 || a.eta != 0.0 || a.u0) return HZ_ERR_UNSUPPORTED;
  if (a.sxe > 32 || a.sye > 32) return HZ_ERR_UNSUPPORTED;
  int shape = a.ty_force;
  if (shape == 0) {
    const char* v = std::getenv("HZ_TILE_SHAPE");  // 1 or 2 forces the shape (tests)
    shape = v ? std::atoi(v) : tile_shape(fp32, P, a.sxe, a.sye, a.Sx * a.Sy);
  }
  if (shape == 2 && (!fp32 || P > 3 || a.sye % 2)) return HZ_ERR_UNSUPPORTED;
  *elements = shape == 2 ? 2 : 1;
  if (fp32) {
    switch (P) {
      case 1: return tile_sweep::tile_f32_p1(shape, a, count, st, warps);
      case 2: return tile_sweep::tile_f32_p2(shape, a, count, st, warps);
      case 3: return tile_sweep::tile_f32_p3(shape, a, count, st, warps);
      case 4: return tile_sweep::tile_f32_p4(shape, a, count, st, warps);
      case 5: return tile_sweep::tile_f32_p5(shape, a, count, st, warps);
      default: return HZ_ERR_UNSUPPORTED;
    }
  }
  switch (P) {
    case 1: return tile_sweep::tile_f64_p1(a, count, st, warps);
    case 2: return tile_sweep::tile_f64_p2(a, count, st, warps);
    case 3: return tile_sweep::tile_f64_p3(a, count, st, warps);
    case 4: return tile_sweep::tile_f64_p4(a, count, st, warps);
    default: return HZ_ERR_UNSUPPORTED;
  }
}
}  // namespace hz
