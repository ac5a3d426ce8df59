// FP64 banded path: operator tables and launches of the per-pencil solves (line.cu).
#pragma once
#include "cfd_internal.h"

namespace cfd {

void build_pencil_tab(const SchemeCoef &s, int N, long double scale, bool unscaled, double factor, PencilTab &T);

// One family of pencils of a launch.
struct PencilTask {
  const PencilTab *tab;
  int N, W, h, deg, anti, unscaled;   // the table's own (a launch need not wait for it to be read)
  int cyclic;            // the blocks concerned are cyclic along the axis (host: all or none, see `only`)
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
// interior half-width of every task of the launch.
cfd_status launch_pencils(const PencilArgs &A, bool halo, bool f32, int N, int M, cudaStream_t st);

}  // namespace cfd
