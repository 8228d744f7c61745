// One-element-per-thread sweep on curved quadrilaterals: instantiations, and
// the rule by size.
#include <algorithm>

#include "hz_sweep_mapped_tile.cuh"

namespace hz {
// One thread per element runs (P+1)^2 nodes in a row, the other kernel one
// node per thread: the tiles win once the node kernel's blocks fill the SMs
// (about 900 of its threads an SM) or need more than one pass over a block.
// Node kernel / tiles, 5 WaveHoltz iterations at 14 node spacings per wavelength
// (N_t about a third above that of square elements): P = 3, 8 x 8 elements: 196 / 119
// us at 9 subdomains, 388 / 127 at 256, 1343 / 349 at 1024; P = 3, 4 x 4: 106 /
// 130 at 256, 270 / 135 at 1024; P = 4, 4 x 4: 231 / 324 at 256, 809 / 330 at
// 1024; P = 2, 16 x 12: 338 / 102 at 9.  Tiles that leave half of the lanes
// idle lose (P = 1, 6 x 5 at 1024: 67 / 81).
bool mapped_tile_default(int P, int snx, int sny, int L) {
  if (P > 4 || snx > 32 || tile_pow2(snx) * sny > 256) return false;
  const int nodes = std::max((snx * P + 1) * (sny * P + 1), snx * sny * (P + 1) * (P + 1));
  const int lanes = tile_pow2(snx) * sny;
  if (lanes > 32 && 3 * snx * sny < 2 * ((lanes + 31) / 32) * 32) return false;
  const int threads = std::min((nodes + 31) / 32 * 32, 1024);
  return nodes >= 1024 || (P <= 2 && threads >= 512) || (long long)threads * L >= 920LL * sm_count();
}

hz_status launch_sweep_mapped_tile(int P, const MappedSweepArgs& a, int count, cudaStream_t st) {
  switch (P) {
    case 1: return mapped_tile::launch<1>(a, count, st);
    case 2: return mapped_tile::launch<2>(a, count, st);
    case 3: return mapped_tile::launch<3>(a, count, st);
    case 4: return mapped_tile::launch<4>(a, count, st);
    default: return HZ_ERR_UNSUPPORTED;
  }
}
}  // namespace hz
