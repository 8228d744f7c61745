// Launch of the element-tile sweep (hz_sweep_tile.cuh) for one degree and
// precision: the tile grid, the slabs and the launch shape by subdomain size.
#pragma once

#include <cstdlib>

#include "hz_sweep_tile.cuh"

namespace hz {
namespace tile_sweep {

// Dynamic shared memory that a launch may ask for.  A kernel's limit is set to
// this constant and not to the launch's own size: another thread that launches
// the same kernel with less would lower the limit between the two calls.
constexpr int kMaxSmem = 220 * 1024;

template <typename Real, int P, int H, bool SRC, bool ISO, bool TOL>
hz_status launch_tile_iso(const SweepArgs& a0, int count, cudaStream_t st, int* warps) {
  const int sxe = a0.sxe, sye = a0.sye;
  if (sxe > 32 || sye > 32 || sye % H) return HZ_ERR_UNSUPPORTED;
  TileArgs x{};
  x.base = a0;
  x.count = count;
  x.LX = tile_pow2(sxe);
  while ((1 << x.lxs) < x.LX) ++x.lxs;
  x.nbt = sye / H;
  for (int k = 0; k < P; ++k) {
    const double wk = a0.w[k] + (k == 0 ? a0.w[P] : 0.0);
    x.wx[k] = a0.hx2 * wk;
    x.wy[k] = a0.hy2 * wk;
  }
  const char* mute = std::getenv("HZ_TILE_MUTE");  // 1: data that never comes (tests)
  x.mute = mute ? std::atoi(mute) : 0;
  const bool tol = a0.wh_tol > 0.0;
  const int lanes = x.LX * x.nbt, need = lanes > sxe + sye ? lanes : sxe + sye;
  if (need <= 32) {  // the whole subdomain in (part of) one warp
    x.nb = x.nbt;
    x.gs = tile_pow2(need);
    x.spw = 32 / x.gs;
    x.offB = sye;
    const Lay y = make_lay<P, Real>(H, x.LX, x.nb, x.gs, SRC, tol);
    const size_t smem = (size_t)x.spw * y.total * sizeof(Real);
    auto kern = x.spw > 1 ? sweep_tile_kernel<Real, P, H, 2, SRC, ISO, false, TOL, 32>
                          : sweep_tile_kernel<Real, P, H, 1, SRC, ISO, false, TOL, 32>;
    if (smem > 48 * 1024) HZ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    kern<<<(count + x.spw - 1) / x.spw, 32, smem, st>>>(x);
    note_launch();
    HZ_CUDA(cudaGetLastError());
    *warps = 1;
    return HZ_OK;
  }
  constexpr int MAXT = tile_max_threads(sizeof(Real) == 8, P, H);
  for (int CL = 1; CL <= 8; ++CL) {
    x.nb = (x.nbt + CL - 1) / CL;
    if (x.nbt - (CL - 1) * x.nb < 1) break;
    x.wm = (x.LX * x.nb + 31) / 32;
    const int nA = x.nb * H;
    x.offB = nA + sxe <= 32 ? nA : 32;
    const int threads = 32 * (x.wm + (x.offB + sxe + 31) / 32);
    if (threads > MAXT) continue;
    const Lay y = make_lay<P, Real>(H, x.LX, x.nb, threads, SRC, tol);
    const size_t smem = (size_t)y.total * sizeof(Real);
    if (smem > kMaxSmem) continue;
    auto kern = CL > 1 ? sweep_tile_kernel<Real, P, H, 0, SRC, ISO, true, TOL, MAXT>
                       : sweep_tile_kernel<Real, P, H, 0, SRC, ISO, false, TOL, MAXT>;
    if (smem > 48 * 1024) HZ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(count * CL));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    HZ_CUDA(cudaLaunchKernelEx(&cfg, kern, x));
    note_launch();
    *warps = CL > 1 ? 0 : threads / 32;  // 0: a cluster
    return HZ_OK;
  }
  return HZ_ERR_UNSUPPORTED;
}

template <typename Real, int P, int H, bool SRC>
hz_status launch_tile(const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  const bool iso = a.hx2 == a.hy2;
  if constexpr (sizeof(Real) == 4) {
    if (!(a.wh_tol > 0.0))
      return iso ? launch_tile_iso<Real, P, H, SRC, true, false>(a, count, st, warps)
                 : launch_tile_iso<Real, P, H, SRC, false, false>(a, count, st, warps);
  }
  return iso ? launch_tile_iso<Real, P, H, SRC, true, true>(a, count, st, warps)
             : launch_tile_iso<Real, P, H, SRC, false, true>(a, count, st, warps);
}

// FP32, shape 1: one element per tile, shape 2: two, paired (P <= 3: the state
// of two larger elements leaves too few warps; P = 4, N_t = 38, 8 x 8 elements at 1024
// subdomains: 235 us one by one, 241 paired, 16 x 16 at 256: 239, 264).
template <int P>
hz_status launch_tile_f32(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  if constexpr (P <= 3) {
    if (shape == 2)
      return a.rhs ? launch_tile<float, P, 2, true>(a, count, st, warps) : launch_tile<float, P, 2, false>(a, count, st, warps);
  }
  return a.rhs ? launch_tile<float, P, 1, true>(a, count, st, warps) : launch_tile<float, P, 1, false>(a, count, st, warps);
}

template <int P>
hz_status launch_tile_f64(const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  return a.rhs ? launch_tile<double, P, 1, true>(a, count, st, warps) : launch_tile<double, P, 1, false>(a, count, st, warps);
}

}  // namespace tile_sweep
}  // namespace hz
