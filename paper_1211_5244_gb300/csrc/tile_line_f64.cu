// Instances of the tile line kernels.
#include "tile_pass.cuh"

namespace ps {

namespace {
template <int DIR, bool HALF>
const void* pick(int cls) {
  using tile::k_tile_line;
  return cls == 0 ? (const void*)k_tile_line<double, DIR, HALF, 0> : cls == 1 ? (const void*)k_tile_line<double, DIR, HALF, 1> : (const void*)k_tile_line<double, DIR, HALF, 2>;
}
}  // namespace

template <>
const void* tile_line_kernel<double>(int dir, bool half, int cls) {
  if (dir < 0) return half ? pick<-1, true>(cls) : pick<-1, false>(cls);
  return half ? pick<1, true>(cls) : pick<1, false>(cls);
}

}  // namespace ps
