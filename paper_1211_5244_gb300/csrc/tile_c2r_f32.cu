// Instances of the real tile kernels (c2r).
#include "tile_pass.cuh"

namespace ps {

namespace {
template <bool PAIR, bool HALF>
const void* pick(int cls) {
  using tile::k_tile_c2r;
  return cls == 0 ? (const void*)k_tile_c2r<float, PAIR, HALF, 0> : cls == 1 ? (const void*)k_tile_c2r<float, PAIR, HALF, 1> : (const void*)k_tile_c2r<float, PAIR, HALF, 2>;
}
}  // namespace

template <>
const void* tile_c2r_kernel<float>(bool pair, bool half, int cls) {
  if (pair) return half ? pick<true, true>(cls) : pick<true, false>(cls);
  return half ? pick<false, true>(cls) : pick<false, false>(cls);
}

}  // namespace ps
