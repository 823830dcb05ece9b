// k_tile_f32.cu -- k_tile compiled for float storage.
#include "k_tile.cuh"

namespace lbk {

int launch_tile_f32(const TileArgs &a, dim3 grid, cudaStream_t s) {
  return launch_tile_t<float, 1>(a, grid, s);
}

}  // namespace lbk
