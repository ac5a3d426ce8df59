// Launches of the exact tensor-core kernel for blocks of 32^3 (dense_exact.cuh).
#include "dense_exact_launch.cuh"

namespace cfd {
cfd_status dense_exact_launch32(const DenseParams &P, bool f32_in, bool f32_out, unsigned grid, cudaStream_t st) {
  return launch_exact<32>(P, f32_in, f32_out, grid, st);
}
}  // namespace cfd
