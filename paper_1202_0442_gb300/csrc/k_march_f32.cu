// k_march_f32.cu -- k_march compiled for float storage.
#include "k_march.cuh"

namespace lbk {

int launch_march_f32(const MarchArgs &a, dim3 grid, dim3 block, cudaStream_t s) {
  return launch_march_t<float, 1>(a, grid, block, s);
}

int launch_march_batch_f32(const MarchBatch &b, int parity, cudaStream_t s) {
  return launch_march_batch_t<float, 1>(b, parity, s);
}

}  // namespace lbk
