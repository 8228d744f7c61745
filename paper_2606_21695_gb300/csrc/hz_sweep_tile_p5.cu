// Element-tile sweep instantiations for degree 5.
#include "hz_sweep_tile_launch.cuh"

namespace hz {
namespace tile_sweep {
hz_status tile_f32_p5(int shape, const SweepArgs& a, int count, cudaStream_t st, int* warps) {
  return launch_tile_f32<5>(shape, a, count, st, warps);
}
}  // namespace tile_sweep
}  // namespace hz
