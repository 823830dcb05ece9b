// k_march_f16.cu -- k_march compiled for __half storage.
#include "k_march.cuh"

namespace lbk {

int launch_march_f16(const MarchArgs &a, dim3 grid, dim3 block, cudaStream_t s) {
  return a.sr ? launch_march_t<__half, 2>(a, grid, block, s) : launch_march_t<__half, 1>(a, grid, block, s);
}

int launch_march_batch_f16(const MarchBatch &b, int parity, cudaStream_t s) {
  return b.sr ? launch_march_batch_t<__half, 2>(b, parity, s) : launch_march_batch_t<__half, 1>(b, parity, s);
}

}  // namespace lbk
