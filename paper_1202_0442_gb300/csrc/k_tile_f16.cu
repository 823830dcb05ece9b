// k_tile_f16.cu -- k_tile compiled for __half storage.
#include "k_tile.cuh"

namespace lbk {

int launch_tile_f16(const TileArgs &a, dim3 grid, cudaStream_t s) {
  return a.sr ? launch_tile_t<__half, 2>(a, grid, s) : launch_tile_t<__half, 1>(a, grid, s);
}

}  // namespace lbk
