// Halo passes of the hybrid iteration through the exact tensor-core kernel (dense_exact.cuh).
#include "dense_exact_launch.cuh"

namespace cfd {
cfd_status dense_exact_halo(const DenseParams &P, bool f32_in, unsigned grid, cudaStream_t st) {
  if (P.N == 32) return f32_in ? launch_exact_halo<float, 32>(P, grid, st) : launch_exact_halo<double, 32>(P, grid, st);
  return f32_in ? launch_exact_halo<float, 16>(P, grid, st) : launch_exact_halo<double, 16>(P, grid, st);
}
}  // namespace cfd
