// Instances of the fused forward, K^F, inverse tile kernels.
#include "tile_pass.cuh"

namespace ps {

namespace {
template <bool HALF>
const void* pick(int cls) {
  using tile::k_tile_conv;
  return cls == 0 ? (const void*)k_tile_conv<float, HALF, 0> : cls == 1 ? (const void*)k_tile_conv<float, HALF, 1> : (const void*)k_tile_conv<float, HALF, 2>;
}
}  // namespace

template <>
const void* tile_conv_kernel<float>(bool half, int cls) {
  return half ? pick<true>(cls) : pick<false>(cls);
}

}  // namespace ps
