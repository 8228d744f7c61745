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
// but leave half the warps: better once one-element tiles fill half of the
// SMs' resident blocks.  Sweeps of 5 WaveHoltz iterations, one / two elements:
// P = 3, 8 x 8 elements: 52 / 67 us at 9 subdomains, 69 / 69 at 256, 87 / 70
// at 576, 165 / 118 at 1024; P = 2, 16 x 16: 46 / 60 at 64, 89 / 76 at 256;
// P = 3, 32 x 32: 143 / 185 at 9, 276 / 186 at 64.  P = 4 gains only where a
// subdomain is one warp (8 x 8: 337 / 249 at 1024; 16 x 16: 337 / 364 at 256:
// 255 registers a thread leave 8 warps an SM).  Tiles that do not fill whole
// warps lose it again (P = 3, 12 x 10 at 1024: 315 / 386).
int tile_shape(bool fp32, int P, int sxe, int sye, int L) {
  if (!fp32 || P > 4 || sye % 2) return 1;
  const int lanes1 = one_element_lanes(sxe, sye), lanes2 = lanes1 / 2;
  if (lanes1 <= 32 && sxe + sye <= 32) return 1;  // one warp either way
  if (lanes2 > 32 && (P == 4 || lanes2 % 32)) return 1;
  if (P == 1) return 2;
  const int cap = tile_max_threads(false, P, 1) / 32;
  const int warps = (lanes1 + 31) / 32 + (sxe + sye + 31) / 32;
  const int ctas = (warps + cap - 1) / cap;                     // CTAs per subdomain
  const int res = cap / ((warps + ctas - 1) / ctas);            // and per SM
  return (long long)L * ctas * 2 > (long long)sm_count() * (res > 0 ? res : 1) ? 2 : 1;
}

// Where the tiles beat the other kernels (5 WaveHoltz iterations, other
// kernel / tiles).  FP32: nearly everywhere (P = 3, 8 x 8 at 1024 subdomains
// 171 / 118 us; P = 4, 32 x 32 at 144: 2140 / 810), except
//  - degree 1 on more than one warp (16 x 16 at 64: 28 / 37), and tiles that
//    leave more than a third of the lanes idle (P = 2, 5 x 7 at 1024: 70 / 80);
//  - few small subdomains of high degree, where P^2 nodes in a row on one
//    lane is the longer chain (block kernel: P = 4, 6 x 6 at 64: 89 / 124;
//    P = 5, 4 x 4 at 64: 120 / 182, one warp at 576: 155 / 182, 1024: 250 / 185).
// FP64 (bound by the FP64 pipe; 3 iterations): with a subdomain per SM and
// whole tiles (P = 3, 8 x 8 at 256: 917 / 685, at 64: 466 / 528; P = 4,
// 16 x 16 at 16: 2364 / 1458; P = 3, 32 x 32 at 64: 3914 / 2384).
bool tile_default(bool fp32, int P, int sxe, int sye, int L) {
  if (sxe > 32 || sye > 32 || P > (fp32 ? 5 : 4)) return false;
  const int lanes = one_element_lanes(sxe, sye);
  const bool one_warp = lanes / (tile_shape(fp32, P, sxe, sye, L)) <= 32 && sxe + sye <= 32;
  if (!fp32) {
    if (P < 2 || sxe < 8 || sxe != tile_pow2(sxe) || sye % 4) return false;
    return sxe == 32 || (P == 4 && sxe == 16) || L >= sm_count();
  }
  if (P == 1 && !one_warp) return false;
  if (!one_warp && 3 * sxe * sye < 2 * ((lanes + 31) / 32) * 32) return false;
  const int block = (sxe * P + 1) * (sye + 1);  // threads of the block kernel
  if (P >= 4 && block <= 192 && 5 * L <= 13 * sm_count()) return false;
  if (P == 5 && one_warp && 2 * L <= 9 * sm_count()) return false;
  return true;
}

hz_status launch_sweep_tile(bool fp32, int P, const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  if (a.round_mode != 0 || a.eta != 0.0 || a.u0) return HZ_ERR_UNSUPPORTED;
  if (a.sxe > 32 || a.sye > 32) return HZ_ERR_UNSUPPORTED;
  int shape = a.ty_force;
  if (shape == 0) {
    const char* v = std::getenv("HZ_TILE_SHAPE");  // 1 or 2 forces the shape (tests)
    shape = v ? std::atoi(v) : tile_shape(fp32, P, a.sxe, a.sye, a.Sx * a.Sy);
  }
  if (shape == 2 && (!fp32 || P > 4 || a.sye % 2)) return HZ_ERR_UNSUPPORTED;
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
