// k_tile_bf16.cu -- k_tile compiled for __nv_bfloat16 storage.
#include "k_tile.cuh"

namespace lbk {

int launch_tile_bf16(const TileArgs &a, dim3 grid, cudaStream_t s) {
  return a.sr ? launch_tile_t<__nv_bfloat16, 2>(a, grid, s) : launch_tile_t<__nv_bfloat16, 1>(a, grid, s);
}

}  // namespace lbk
