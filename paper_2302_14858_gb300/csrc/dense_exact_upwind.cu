// Upwinded stages of the shift advection through the exact tensor-core kernel (dense_exact.cuh).
#include "dense_exact_launch.cuh"

namespace cfd {
cfd_status dense_exact_upwind(const DenseParams &P, bool f32, unsigned grid, cudaStream_t st) {
  if (P.N == 32)
    return f32 ? launch_exact_types<float, float, 32, kUpwind>(P, grid, st)
               : launch_exact_types<double, double, 32, kUpwind>(P, grid, st);
  return f32 ? launch_exact_types<float, float, 16, kUpwind>(P, grid, st)
             : launch_exact_types<double, double, 16, kUpwind>(P, grid, st);
}
}  // namespace cfd
