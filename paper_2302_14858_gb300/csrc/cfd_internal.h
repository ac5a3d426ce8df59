// Internal structures of the CFD library (host API <-> CUDA kernels).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/cfd.h"

namespace cfd {

constexpr int kMaxN = 32;        // largest block interior size
constexpr int kMaxM = 5;         // largest interior half-width
constexpr int kMaxH = 6;         // largest closure half-width

// Coefficients of one centred tridiagonal scheme (host copy).
struct SchemeCoef {
  bool present = false;
  int d = 0, order = 0, M = 0, h = 0;
  double a = 0.0;
  double rhs[2 * kMaxM + 1] = {};
  double clo[2 * kMaxH + 1] = {};
};

// Biased first-degree scheme (left-biased form) as given to cfd_scheme_set_biased.
constexpr int kBOff = 6;                 // coefficient of offset m stored at m + kBOff
constexpr int kBTaps = 2 * kBOff + 1;    // offsets -6..6
struct BiasedCoef {
  bool present = false;
  int order = 0, lo = 0, hi = 0, clo = 0, chi = 0, kc = 1;  // offset ranges (inclusive)
  double a = 0.0, csup = 0.0;
  double rhs[kBTaps] = {}, cl[kBTaps] = {};
};

// Per block size: what one biased pencil solve needs (passed by value).
struct BiasedTables {
  int N, kc;
  double a, csup;
  double inv01;            // 1 / (1 - csup a): the 2x2 coupling of the closure row
  double cyc_inv;          // 1 / (1 - (-a)^N): cyclic (single-block periodic) axis
  double rhs[kBTaps], clo[kBTaps];
  double pw[kMaxN + 1];    // (-a)^j
  // Halo-only passes: row N-kc of the left-biased and row kc-1 of the right-biased block
  // operator ([side][0 closed, 1 iterated][ghost-extended index]) and, for the iterated
  // operator, the coefficient of the fixed value at k^c.
  double hrow[2][2][kMaxN + 16];
  double hc[2];
};

// One biased axis pass over a group of same-size blocks.
struct BiasedParams {
  const void *in;          // field buffer (dtype)
  const void *beta;        // shift fields (advect mode)
  void *out;
  const int *blocks;
  const long long *extpre, *intpre;
  const int *nbr;
  const double *scale;     // [nblocks][2][3]; the degree-1 entries are used
  const double *halo_in;   // [nblocks][nf][N^2][2]: (d+ at N-kc, d- at kc-1) of the previous iterate
  double *halo_out;
  int nblk, nf, nops, opidx;
  int axis;                // box axis of the pencils (0 z, 1 y, 2 x)
  int axes, axis2;         // axes = 2: a halo pass of `axis2` too, into halo_out2
  double *halo_out2;
  int mode;                // 0 d[S+], 1 d[S-], 2 advect (beta_+ d[S+] + beta_- d[S-])
  int accum;               // 1: add into out
  int pass, last;
  int cyclic;              // some block is its own neighbour along the axis
};

void build_biased_tables(const BiasedCoef &c, int N, int g, BiasedTables &T);
// dense form of a biased block system (kind 0 closed, 1 iterated, 2 cyclic), unscaled
void biased_operator(const BiasedCoef &c, int N, int g, int side, int kind, std::vector<long double> &W,
                     std::vector<long double> &coup);

}  // namespace cfd

namespace cfd {
// What the solves along one axis need, for one block size, degree and scale (device copy), prepared in
// long double.  Antisymmetric stencils act on differences, which vanish for a constant whatever the
// coefficients round to: the scale 1/dx^d and the reciprocal pivot of a row are folded into them, and a
// row costs its right-hand side and one FMA forward, one back.  Other stencils keep the coefficients as
// given (their rounded sum, the operator's value on a constant, must not grow): pivot and scale come in
// on the way back, one more operation per row.
struct PencilTab {
  int N, M, h, deg;      // block size, interior and closure half-widths, degree
  int W;                 // points needed beyond the block on each side: max(h, M + 1)
  int anti;              // degree 1 with exactly antisymmetric coefficients: differences of pairs
  int unscaled;          // spacing differs between blocks: results are multiplied per block
  // scalars, copied as one run (kTabScalars): -1 and 0 (see stencil() in line.cu); the factor folded into the
  // results (1, or 1/2 for one half of an averaged pair); scale of rows that keep their coefficients (1: folded)
  // and its reciprocal; factor of the upper fixed value; cyclic system: a and the Sherman-Morrison factor
  double neg, nil, factor, sc, isc, hhi, a, vfac;
  double clo[2 * kMaxH + 1];
  // closed system (rows 1..N-2; rows 0 and N-1 are the closures): row k
  //   z_k = sum_m rc[k][m + M] f_{k+m} - lo[k] z_{k-1},   x_k = pv[k] z_k - up[k] x_{k+1}
  double rc[kMaxN][2 * kMaxM + 1], lo[kMaxN], up[kMaxN], pv[kMaxN];
  // iterated system, rows k = -1..N at k + 1; the fixed values enter the first and last row
  double irc[kMaxN + 2][2 * kMaxM + 1], ilo[kMaxN + 2], iup[kMaxN + 2], ipv[kMaxN + 2];
  // cyclic system: Thomas rows of the corner-modified matrix, its Sherman-Morrison vector
  double yrc[kMaxN][2 * kMaxM + 1], ylo[kMaxN], yup[kMaxN], ypv[kMaxN], z[kMaxN];
  // rows 1 and N-2 of the closed and of the iterated operator over the window (index j + W for point
  // j), and the coefficients of the fixed values: what the neighbours read (factor 1 always)
  double hrow[2][2][kMaxN + 2 * kMaxH + 2], hc[2][2];
};
constexpr int kTabScalars = 8;
}  // namespace cfd

struct cfd_scheme_s {
  cfd::SchemeCoef s[2];
  cfd::BiasedCoef biased;
};

struct cfd_blocks_s {
  cfd::SchemeCoef s[2];
  int device = 0, num_sms = 0;
  int nblocks = 0, ng = 0;
  cfd_dtype dtype = CFD_F64;
  std::vector<int> n;                  // per block
  std::vector<int> nbr;                // [nblocks * 26]
  std::vector<double> dx;              // [nblocks * 3]
  std::vector<long long> extpre, intpre;
  std::vector<int> sizes;              // distinct N, increasing
  std::vector<std::vector<int>> groups;  // block ids per distinct N
  // FP64 banded tables per distinct N (line.h), device: [degree 1: axis, full / half][degree 2: axis]
  std::vector<void *> d_ptab;
  std::vector<std::vector<cfd::PencilTab>> h_ptab;
  cfd::BiasedCoef biased;
  std::vector<cfd::BiasedTables> btab; // per distinct N (when biased.present)
  bool iter_ok = true;                 // same-size face neighbours everywhere
  bool mixed_one_order = false;        // FP64 banded path: d_ij as D_i D_j only (cfd_blocks_set_mixed_order)
  // device copies
  int *d_nbr = nullptr, *d_lidx = nullptr;  // neighbours; position of a block in its size group
  long long *d_extpre = nullptr, *d_intpre = nullptr;
  // ghost exchange: per block its 26 neighbours' field offsets (extpre of the neighbour, -1 for
  // none) and its own (entry 26), so a copy needs one table load
  long long *d_exch = nullptr;
  std::vector<int> group_b0;           // per group: first block id if the group's ids are consecutive, else -1
  double *d_scale = nullptr;
  int *d_nvec = nullptr;
  std::vector<int *> d_groups;
  int *d_status = nullptr;
  // dense operators for the tensor-core path (per distinct N), see dense_tc.cu:
  // host-side state, its deleter, and the device allocations it refers to
  void *dense_state = nullptr;
  void (*dense_free)(void *) = nullptr;
  std::vector<void *> d_dense_ptrs;
};

namespace cfd {

void set_error(const std::string &msg);
cfd_status cuda_fail(cudaError_t e, const char *what);

// launch accounting (profile.cpp)
enum KernelFamily { KF_EXCHANGE = 0, KF_LINE = 1, KF_RK = 2, KF_DENSE = 3, KF_HALO = 4, KF_BIASED = 5, KF_COUNT = 6 };
void launch_begin(int family, cudaStream_t st);
void launch_end(int family, cudaStream_t st);

#ifdef __CUDACC__
// Launches that may start while the launch before them on the stream drains (programmatic dependent launch).
// Such a kernel calls chain_wait() before its first access to memory that an earlier launch may write or
// still read: it returns once those launches have finished and their writes are visible.  Before it come
// only set-up (barriers, TMEM, index arithmetic) and tables that bind wrote; data behind it is read with
// plain loads (the read-only path may move a load ahead of the wait).  chain_next() lets the next such
// launch be scheduled, which happens when every CTA of this one has called it or left.
// Measured (exchange and apply): 64^3, 2 fields, nine ops 67 -> 50 us; 128^3 in 16^3 blocks, 4 fields
// 377 -> 365; 22 FP32 fields on two levels 2.87 -> 2.80 ms.  k_line stays unchained: its CTAs, several per SM,
// then pile up on the SMs that empty first (27 blocks of 16^3, nine ops: 177 -> 211 us).
template <typename... P, typename... A>
inline void launch_chained(void (*fn)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, bool chained,
                           A &&...args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&cfg, fn, std::forward<A>(args)...);
}
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif

// biased.cu: out[block][field][slot out_opidx of out_nops] += sum_i beta^i_+ D_i[S-] f + beta^i_- D_i[S+] f
// for nf fields (`work` as cfd_biased_workspace(B, nf, prec, n_iter))
cfd_status advect_accumulate(cfd_blocks_s *B, const void *fields, int nf, const void *beta, void *out, int out_nops,
                             int out_opidx, cfd_precision prec, int n_iter, void *work, size_t work_bytes,
                             cudaStream_t st);
// biased.cu: the checks of advect_accumulate alone (stencil window, iteration, workspace)
cfd_status advect_check(cfd_blocks_s *B, int nf, cfd_precision prec, int n_iter, void *work, size_t work_bytes);
// biased.cu: out slot = (accum_all ? out : 0) + sum_{i=x,y,z} beta^i d_i, d_i the biased derivative the sign
// of beta^i selects: tmp = [block][field][3][N^3] (the selected ones), or with `both`
// [block][field][6][N^3] (S+ and S- of every axis)
cfd_status advect_combine(cfd_blocks_s *B, const void *tmp, bool both, const void *beta, int nf, void *out,
                          int out_nops, int out_opidx, bool accum_all, cudaStream_t st);
// biased.cu: the signs of the shift for DenseParams::upwind: sizes in order, 3 N^2 words per block
size_t upwind_words(const cfd_blocks_s *B);
cfd_status upwind_signs(cfd_blocks_s *B, const void *beta, uint32_t *words, cudaStream_t st);
// dense_tc.cu: the biased operators on the tensor cores
size_t dense_biased_workspace(const cfd_blocks_s *B, int nf, int n_iter, bool advect);
// (signs, tmp: the upwinded derivatives of every axis into tmp [block][field][3][N^3] with the signs given,
// without the blend; exact form only)
cfd_status dense_biased(cfd_blocks_s *B, const void *fields, int nf, const void *beta, const int *axes, int naxes,
                        int mode, cfd_precision prec, int n_iter, void *out, int out_nops, int out_opidx,
                        bool accum_all, void *work, size_t work_bytes, cudaStream_t st,
                        const uint32_t *signs = nullptr, void *tmp = nullptr);
// Where a step may keep the shift's signs in a one-field workspace of dense_biased whose six slots it fills
// itself (behind the used part of a halo buffer); null without iteration or where they do not fit.
uint32_t *dense_sign_space(const cfd_blocks_s *B, void *work, int n_iter);

// exchange.cu
cfd_status launch_exchange(cfd_blocks_s *B, void *fields, int nfields, cudaStream_t st);

}  // namespace cfd
