// Element-tile sweep instantiations for degree 2.
#include "hz_sweep_tile_launch.cuh"

namespace hz {
namespace tile_sweep {
hz_status tile_f32_p2(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  return launch_tile_f32<2>(shape, a, count, st, warps);
}
hz_status tile_f64_p2(const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  return launch_tile_f64<2>(a, count, st, warps);
}
}  // namespace tile_sweep
}  // namespace hz
