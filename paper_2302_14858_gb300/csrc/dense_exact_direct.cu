// Outer stages of mixed derivatives that read the inner derivative from its output slot
// (dense_exact.cuh, DIRECT), and their halo passes.
#include "dense_exact_launch.cuh"

namespace cfd {
namespace {
template <int N, int MODE>
cfd_status launch_direct(const DenseParams &P, unsigned grid, cudaStream_t st) {
  const bool it = P.halo_in != nullptr;
  if (P.axis == 2)
    return it ? launch_one<double, double, N, 2, true, MODE>(P, grid, st) : launch_one<double, double, N, 2, false, MODE>(P, grid, st);
  return it ? launch_one<double, double, N, 1, true, MODE>(P, grid, st) : launch_one<double, double, N, 1, false, MODE>(P, grid, st);
}
}  // namespace
cfd_status dense_exact_direct(const DenseParams &P, bool halo, unsigned grid, cudaStream_t st) {
  if (P.N == 32) return halo ? launch_direct<32, kHaloDirect>(P, grid, st) : launch_direct<32, kDirect>(P, grid, st);
  return halo ? launch_direct<16, kHaloDirect>(P, grid, st) : launch_direct<16, kDirect>(P, grid, st);
}
}  // namespace cfd
