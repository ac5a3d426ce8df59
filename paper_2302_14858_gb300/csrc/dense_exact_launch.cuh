// Host side of the exact tensor-core kernel: shared-memory plan and instantiation choice.
#pragma once
#include <algorithm>
#include <atomic>

#include "dense_exact.cuh"

namespace cfd {
namespace {

constexpr size_t kSmemMax = 227 * 1024;

// Shared memory of a launch: two A digit buffers, the operator digits, the staging buffers (two where
// they fit), the epilogue's output boxes (x stages), row exponents, the pencil-scale ring and the barriers.  At least 116 KB, so that one CTA
// (holding all TMEM columns) occupies an SM.
template <typename TI, int N>
size_t plan_smem(DenseParams &P) {
  constexpr int KP = N == 32 ? 48 : 32;
  const int E = N + 2 * P.g;
  const size_t fixed = ((2 * (size_t)kSl * kTile * KP * 2 + (size_t)kSl * P.rows * KP * 2 + 1023) & ~(size_t)1023) +
                       64 * 4 + kXEtau * kTile * 2 + 28 * 8 + 16;
  const size_t rows = P.axis == 2 ? (size_t)((E * (int)sizeof(TI) + kXRowBytes - 1) / kXRowBytes) * kTile * kXRowBytes
                                  : (size_t)E * kTile * sizeof(TI);
  P.stg_bytes = (int)((rows + 1023) & ~(size_t)1023);
  if (P.halo_in && P.tma_kind) {  // both sides' halo values of a tile, by bulk copies into the same buffer
    P.halo_stg = P.stg_bytes;
    P.stg_bytes += 2 * kTile * P.halo_nd * 8;
    P.tma_bytes += 2 * kTile * P.halo_nd * 8;
  }
  const size_t out = (size_t)P.out_box_bytes * kXEpiWarps;
  P.nstg = fixed + out + 2 * (size_t)P.stg_bytes <= kSmemMax ? 2 : 1;
  return std::max(fixed + out + (size_t)P.nstg * P.stg_bytes, (size_t)116 * 1024);
}

template <typename TI, typename TO, int N, int AXIS, bool ITER, int MODE, int STG>
cfd_status launch_staged(DenseParams P, unsigned grid, cudaStream_t st) {
  const size_t smem = plan_smem<TI, N>(P);
  // The shared-memory opt-in is made once per device and instantiation, for the most any launch may
  // need, so later calls issue nothing but the launch (a stream under capture sees kernel nodes only).
  static std::atomic<bool> opted[64];
  int dev = 0;
  cfd_status s = cuda_fail(cudaGetDevice(&dev), "cudaGetDevice");
  if (s != CFD_OK) return s;
  auto fn = k_dense_exact<TI, TO, N, AXIS, ITER, MODE, STG>;
  if (dev < 0 || dev >= 64 || !opted[dev].load()) {
    s = cuda_fail(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax),
                  "cudaFuncSetAttribute");
    if (s != CFD_OK) return s;
    if (dev >= 0 && dev < 64) opted[dev].store(true);
  }
  if (smem > kSmemMax) { set_error("dense: shared memory plan too large"); return CFD_ERR_UNSUPPORTED; }
  constexpr int family = MODE == kHaloRows || MODE == kHaloDirect ? KF_HALO : KF_DENSE;
  launch_begin(family, st);
  launch_chained(fn, dim3(grid), kXThreads, smem, st, true, P);
  launch_end(family, st);
  return cuda_fail(cudaGetLastError(), "k_dense_exact launch");
}

template <typename TI, typename TO, int N, int AXIS, bool ITER, int MODE = kPlain>
cfd_status launch_one(const DenseParams &P, unsigned grid, cudaStream_t st) {
  if constexpr (AXIS != 2 || MODE == kDirect || MODE == kHaloDirect) {
    return launch_staged<TI, TO, N, AXIS, ITER, MODE, 0>(P, grid, st);
  } else {
    return P.tma_kind ? launch_staged<TI, TO, N, AXIS, ITER, MODE, 1>(P, grid, st)
                      : launch_staged<TI, TO, N, AXIS, ITER, MODE, 2>(P, grid, st);
  }
}

// Ghost width 4 has the axis compiled in; other widths share one instantiation per type.
template <typename TI, typename TO, int N, int MODE = kPlain>
cfd_status launch_exact_types(const DenseParams &P, unsigned grid, cudaStream_t st) {
  const bool it = P.halo_in != nullptr;
  if (P.g == 4) {
    if (P.axis == 2) return it ? launch_one<TI, TO, N, 2, true, MODE>(P, grid, st) : launch_one<TI, TO, N, 2, false, MODE>(P, grid, st);
    if (P.axis == 1) return it ? launch_one<TI, TO, N, 1, true, MODE>(P, grid, st) : launch_one<TI, TO, N, 1, false, MODE>(P, grid, st);
    return it ? launch_one<TI, TO, N, 0, true, MODE>(P, grid, st) : launch_one<TI, TO, N, 0, false, MODE>(P, grid, st);
  }
  return it ? launch_one<TI, TO, N, 3, true, MODE>(P, grid, st) : launch_one<TI, TO, N, 3, false, MODE>(P, grid, st);
}

// Halo passes: the first one (closed operator rows) has the axis compiled in for ghost width 4; the
// further iterates, which only n_iter > 1 needs, take the general form.
template <typename TI, int N>
cfd_status launch_exact_halo(const DenseParams &P, unsigned grid, cudaStream_t st) {
  if (P.halo_in) return launch_one<TI, double, N, 3, true, kHaloRows>(P, grid, st);
  if (P.g != 4) return launch_one<TI, double, N, 3, false, kHaloRows>(P, grid, st);
  if (P.axis == 2) return launch_one<TI, double, N, 2, false, kHaloRows>(P, grid, st);
  if (P.axis == 1) return launch_one<TI, double, N, 1, false, kHaloRows>(P, grid, st);
  return launch_one<TI, double, N, 0, false, kHaloRows>(P, grid, st);
}

template <int N>
cfd_status launch_exact(const DenseParams &P, bool f32_in, bool f32_out, unsigned grid, cudaStream_t st) {
  if (f32_in) return launch_exact_types<float, float, N>(P, grid, st);
  if (f32_out) return launch_exact_types<double, float, N>(P, grid, st);
  return launch_exact_types<double, double, N>(P, grid, st);
}

}  // namespace
}  // namespace cfd
