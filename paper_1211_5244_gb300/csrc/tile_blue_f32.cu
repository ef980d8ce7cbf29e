// Instances of the tile kernels in Bluestein form (radices up to 16).
#include "tile_pass.cuh"

namespace ps {

template <>
const void* tile_blue_kernel<float>(int pass, bool pair) {
  using namespace tile;
  switch (pass) {
    case P1: return pair ? (const void*)k_blue_r2c<float, true, 1> : (const void*)k_blue_r2c<float, false, 1>;
    case P2: return (const void*)k_blue_line<float, -1, 1>;
    case P3: return (const void*)k_blue_conv<float, 1>;
    case P4: return (const void*)k_blue_line<float, 1, 1>;
    default: return pair ? (const void*)k_blue_c2r<float, true, 1> : (const void*)k_blue_c2r<float, false, 1>;
  }
}

}  // namespace ps
