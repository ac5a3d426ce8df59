// FP64 banded path: operator tables and launches of the per-pencil solves (line.cu).
#pragma once
#include "cfd_internal.h"

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
  double neg, nil;       // -1 and 0 (see stencil() in line.cu)
  double factor;         // folded into the results (1, or 1/2 for one half of an averaged pair)
  double clo[2 * kMaxH + 1];
  double sc, isc;        // scale of rows that keep their coefficients (1: folded), and its reciprocal
  // closed system (rows 1..N-2; rows 0 and N-1 are the closures): row k
  //   z_k = sum_m rc[k][m + M] f_{k+m} - lo[k] z_{k-1},   x_k = pv[k] z_k - up[k] x_{k+1}
  double rc[kMaxN][2 * kMaxM + 1], lo[kMaxN], up[kMaxN], pv[kMaxN];
  // iterated system, rows k = -1..N at k + 1; the fixed values enter the first and last row
  double irc[kMaxN + 2][2 * kMaxM + 1], ilo[kMaxN + 2], iup[kMaxN + 2], ipv[kMaxN + 2], hhi;
  // cyclic system: Thomas rows of the corner-modified matrix, its Sherman-Morrison vector
  double yrc[kMaxN][2 * kMaxM + 1], ylo[kMaxN], yup[kMaxN], ypv[kMaxN], z[kMaxN], a, vfac;
  // rows 1 and N-2 of the closed and of the iterated operator over the window (index j + W for point
  // j), and the coefficients of the fixed values: what the neighbours read (factor 1 always)
  double hrow[2][2][kMaxN + 2 * kMaxH + 2], hc[2][2];
};

void build_pencil_tab(const SchemeCoef &s, int N, long double scale, bool unscaled, double factor, PencilTab &T);

// One family of pencils of a launch.
struct PencilTask {
  const PencilTab *tab;
  int axis, t1, t2;      // pencil axis and transverse axes (0 z, 1 y, 2 x), t1 < t2
  int n1, n2;            // pencils along t1, t2
  int only;              // 0 every block, 1 the blocks that are cyclic along the axis, 2 the others
  // first transverse point relative to the block's own; strip = 1 (2): t1 (t2) runs over the ghost
  // points, the lower g then the upper g
  int strip;
  int gather;            // input: 0 the field, 1 own points of a derivative with its ghost strip
  int in_op;             // gather: slot of the output holding the derivative, -1: scratch at in_off
  long long in_off, strip_off;        // gather: elements per (block, field) stride and base in the region
  int out_op, accum;     // final output slot (-1: none); accum: add to it
  long long sc_off;      // scratch output base (-1: none): [block][field][N^3], or a strip (strip != 0)
  long long halo_in, halo_out;        // halo values: base in the halo region
};
constexpr int kMaxTasks = 6;
struct PencilArgs {
  const void *field;     // field dtype
  void *out;
  double *region;        // scratch
  double *halo;          // halo values [task base][block][field][pencil][2]
  const int *blocks, *lidx, *nbr;
  const long long *extpre, *intpre;
  const double *scale;
  int nblk, nf, nops, g, ntask, pass;  // pass: iterates done before this launch (0: closed)
  PencilTask task[kMaxTasks];
};

// halo: the values the neighbours read (rows 1 and N-2 of this pass's iterate); else the solve.  M: the
// interior half-width of every task of the launch, W: the widest window.
cfd_status launch_pencils(const PencilArgs &A, bool halo, bool f32, int N, int M, int W, cudaStream_t st);

}  // namespace cfd
