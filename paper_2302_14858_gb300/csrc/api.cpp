// Host side of the C ABI: scheme construction (closure by C_0 matching),
// MeshBlock binding (operator tables per block size) and launch planning.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "cfd_internal.h"
#include "dense.h"
#include "line.h"

namespace cfd {

static thread_local std::string g_err;

void set_error(const std::string &msg) { g_err = msg; }

cfd_status cuda_fail(cudaError_t e, const char *what) {
  if (e == cudaSuccess) return CFD_OK;
  set_error(std::string(what) + ": " + cudaGetErrorString(e));
  return CFD_ERR_CUDA;
}

namespace {

typedef long double ld;

ld fact(int n) {
  ld r = 1;
  for (int i = 2; i <= n; ++i) r *= i;
  return r;
}

// Power series helpers in u = eta^2 (centred schemes have even expansions).
std::vector<ld> series_div(const std::vector<ld> &a, const std::vector<ld> &b) {
  std::vector<ld> q(a.size(), 0);
  for (size_t k = 0; k < a.size(); ++k) {
    ld s = a[k];
    for (size_t i = 0; i < k; ++i) s -= q[i] * b[k - i];
    q[k] = s / b[0];
  }
  return q;
}

// Leading error constant C_0 of eps(eta) = eta~^d / eta^d - 1 ~ C_0 eta^order
// for a centred tridiagonal scheme (Eq. fdpwerrdef, Eq. errrelmodwavcent).
//   d = 1:  eta~ / eta = 2 sum_{m>0} a_m sin(m eta) / eta  /  (1 + 2 a cos eta)
//   d = 2:  eta~^2 / eta^2 = -(a_0 + 2 sum_{m>0} a_m cos(m eta)) / eta^2  /  (1 + 2 a cos eta)
ld interior_C0(const SchemeCoef &s) {
  const int K = s.order / 2 + 3;
  std::vector<ld> den(K, 0), num(K + 1, 0);
  for (int k = 0; k < K; ++k) den[k] = ((k % 2) ? -1 : 1) * 2.0L * (ld)s.a / fact(2 * k);
  den[0] += 1;
  const int M = s.M;
  if (s.d == 1) {
    for (int k = 0; k < K; ++k) {
      ld acc = 0;
      for (int m = 1; m <= M; ++m) acc += (ld)s.rhs[M + m] * powl((ld)m, 2 * k + 1);
      num[k] = ((k % 2) ? -1 : 1) * 2.0L * acc / fact(2 * k + 1);
    }
    num.resize(K);
  } else {
    for (int k = 0; k <= K; ++k) {
      ld acc = (k == 0) ? (ld)s.rhs[M] : 0;
      for (int m = 1; m <= M; ++m) acc += 2.0L * (ld)s.rhs[M + m] * powl((ld)m, 2 * k);
      num[k] = -((k % 2) ? -1 : 1) * acc / (k == 0 ? 1 : fact(2 * k));
    }
    // drop the eta^0 term (consistency makes it vanish) and divide by eta^2
    num.erase(num.begin());
  }
  std::vector<ld> r = series_div(num, den);
  return r[s.order / 2];  // coefficient of u^{order/2} = eta^{order}; eps = r - 1
}

bool solve_dense(std::vector<ld> A, std::vector<ld> b, int n, std::vector<ld> &x) {
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int r = c + 1; r < n; ++r)
      if (fabsl(A[r * n + c]) > fabsl(A[p * n + c])) p = r;
    if (A[p * n + c] == 0) return false;
    if (p != c) {
      for (int k = 0; k < n; ++k) std::swap(A[p * n + k], A[c * n + k]);
      std::swap(b[p], b[c]);
    }
    for (int r = c + 1; r < n; ++r) {
      const ld f = A[r * n + c] / A[c * n + c];
      for (int k = c; k < n; ++k) A[r * n + k] -= f * A[c * n + k];
      b[r] -= f * b[c];
    }
  }
  x.assign(n, 0);
  for (int r = n - 1; r >= 0; --r) {
    ld s = b[r];
    for (int k = r + 1; k < n; ++k) s -= A[r * n + k] * x[k];
    x[r] = s / A[r * n + r];
  }
  return true;
}

// Explicit centred closure of half-width h = order/2 + 1 (Sec. domdec_drp):
// formal order `order` plus the eta^order error constant equal to the
// interior's C_0.  Unknowns use the (anti)symmetry of centred stencils.
bool build_closure(SchemeCoef &s) {
  const ld C0 = interior_C0(s);
  const int h = s.order / 2 + 1;
  if (h > kMaxH) return false;
  std::vector<ld> A, b, x;
  if (s.d == 1) {
    // unknowns b_1..b_h; alpha-bar_{+-m} = +-b_m
    const int n = h;
    A.assign(n * n, 0);
    b.assign(n, 0);
    int row = 0;
    for (int q = 1; q < s.order; q += 2, ++row) {
      for (int m = 1; m <= h; ++m) A[row * n + (m - 1)] = 2.0L * powl((ld)m, q) / fact(q);
      b[row] = (q == 1) ? 1 : 0;
    }
    const int sg = ((s.order / 2) % 2) ? -1 : 1;
    for (int m = 1; m <= h; ++m) A[row * n + (m - 1)] = sg * 2.0L * powl((ld)m, s.order + 1) / fact(s.order + 1);
    b[row] = C0;
    if (!solve_dense(A, b, n, x)) return false;
    for (int i = 0; i < 2 * kMaxH + 1; ++i) s.clo[i] = 0;
    s.clo[h] = 0.0;
    for (int m = 1; m <= h; ++m) {
      s.clo[h + m] = (double)x[m - 1];
      s.clo[h - m] = -(double)x[m - 1];
    }
  } else {
    // unknowns b_0..b_h; alpha-bar_0 = b_0, alpha-bar_{+-m} = b_m
    const int n = h + 1;
    A.assign(n * n, 0);
    b.assign(n, 0);
    A[0] = 1;
    for (int m = 1; m <= h; ++m) A[m] = 2;
    int row = 1;
    for (int k = 1; k <= s.order / 2 + 1; ++k, ++row) {
      const int sg = (k % 2) ? -1 : 1;
      for (int m = 1; m <= h; ++m) A[row * n + m] = sg * 2.0L * powl((ld)m, 2 * k) / fact(2 * k);
      b[row] = (k == 1) ? -1.0L : (k == s.order / 2 + 1 ? -C0 : 0);
    }
    if (!solve_dense(A, b, n, x)) return false;
    for (int i = 0; i < 2 * kMaxH + 1; ++i) s.clo[i] = 0;
    s.clo[h] = (double)x[0];
    for (int m = 1; m <= h; ++m) s.clo[h + m] = s.clo[h - m] = (double)x[m];
  }
  s.h = h;
  return true;
}

cfd_status copy_desc(const cfd_scheme_desc *d, int deg, SchemeCoef &s) {
  if (!d) return CFD_OK;
  if (d->deriv != deg) { set_error("scheme degree does not match its slot"); return CFD_ERR_ARG; }
  if (d->M < 1 || d->M > kMaxM || !d->rhs) { set_error("interior half-width M out of range"); return CFD_ERR_ARG; }
  if (d->order < 2 || d->order % 2 || d->order > 10) { set_error("order must be even, 2..10"); return CFD_ERR_ARG; }
  if (!(fabs(d->lhs_offdiag) * 2 < 1)) { set_error("system not diagonally dominant (2|a| >= 1)"); return CFD_ERR_ARG; }
  s.present = true;
  s.d = deg;
  s.order = d->order;
  s.M = d->M;
  s.a = d->lhs_offdiag;
  double mx = 0;
  for (int i = 0; i < 2 * d->M + 1; ++i) {
    s.rhs[i] = d->rhs[i];
    mx = std::max(mx, fabs(d->rhs[i]));
  }
  for (int m = 1; m <= d->M; ++m) {
    const double lo = d->rhs[d->M - m], hi = d->rhs[d->M + m];
    const double bad = deg == 1 ? fabs(lo + hi) : fabs(lo - hi);
    if (bad > 1e-14 * mx) { set_error("interior stencil is not centred ((anti)symmetric)"); return CFD_ERR_ARG; }
  }
  if (d->closure) {
    if (d->closure_halfwidth < 1 || d->closure_halfwidth > kMaxH) {
      set_error("closure half-width out of range");
      return CFD_ERR_ARG;
    }
    s.h = d->closure_halfwidth;
    for (int i = 0; i < 2 * s.h + 1; ++i) s.clo[i] = d->closure[i];
  } else if (!build_closure(s)) {
    set_error("closure construction failed");
    return CFD_ERR_ARG;
  }
  return CFD_OK;
}

int dir_index(int dz, int dy, int dx) {
  int r = 9 * (dz + 1) + 3 * (dy + 1) + (dx + 1);
  return r > 13 ? r - 1 : r;
}

template <typename T>
cfd_status upload(T **dst, const T *src, size_t n) {
  cfd_status s = cuda_fail(cudaMalloc((void **)dst, n * sizeof(T) + 16), "cudaMalloc");
  if (s != CFD_OK) return s;
  return cuda_fail(cudaMemcpy(*dst, src, n * sizeof(T), cudaMemcpyHostToDevice), "cudaMemcpy");
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct OpList {
  int n = 0;
  int bit[9];
};

OpList ops_of(unsigned mask) {
  OpList o;
  for (int i = 0; i < 9; ++i)
    if (mask & (1u << i)) o.bit[o.n++] = i;
  return o;
}

// box axis index of a letter: x -> 2, y -> 1, z -> 0
const int kAxisOfOp1[3] = {2, 1, 0};                 // dx, dy, dz
const int kMixed[3][2] = {{2, 1}, {2, 0}, {1, 0}};   // (i, j): dxy, dxz, dyz

void banded_workspace_sizes(const cfd_blocks_s *B, int nf, unsigned mask, int n_iter, size_t *scratch,
                            size_t *halo) {
  size_t sc = 0, hp = 0;
  const bool mixed = (mask & (CFD_OP_DXY | CFD_OP_DXZ | CFD_OP_DYZ)) != 0;
  for (size_t gi = 0; gi < B->sizes.size(); ++gi) {
    const size_t N = B->sizes[gi], E = N + 2 * B->ng;
    if (mixed) sc = std::max(sc, B->groups[gi].size() * nf * E * N * N);
    hp = std::max(hp, E * N);
  }
  *scratch = sc;
  *halo = n_iter > 0 ? (size_t)B->nblocks * nf * hp * 2 : 0;
}

// table of (degree, box axis, half) among a size's tables
int ptab_index(int deg, int box, bool half) { return deg == 1 ? 2 * box + (half ? 1 : 0) : 6 + box; }

// FP64 banded apply.  `region`: the mixed ops' scratch (region_elems doubles), `halo`: the halo values of
// the iteration (halo_elems doubles); where both exist the halo space follows the scratch directly.
//
// Launches (all blocks, fields and axes of a size together): the single derivatives; then per inner axis
// j of the mixed ops the ghost strips of D_j (local evaluation on the ghost rows of the outer axes) and
// D_i on [strip | own points | strip].  Own points of D_j come from its output slot (FP64 fields with d_j
// requested) or from one scratch copy.  Each launch is preceded by n_iter halo passes.
cfd_status apply_banded(cfd_blocks_s *B, const void *fields, int nf, unsigned mask, int n_iter, void *out,
                        double *region, size_t region_elems, double *halo, size_t halo_elems, cudaStream_t st) {
  const OpList ol = ops_of(mask);
  auto slot = [&](int bit) {
    for (int i = 0; i < ol.n; ++i)
      if (ol.bit[i] == bit) return i;
    return -1;
  };
  if (((mask & 0x1C7) && !B->s[0].present) || ((mask & 0x38) && !B->s[1].present)) {
    set_error((mask & 0x1C0) && !B->s[0].present ? "mixed ops need the first-degree scheme"
                                                 : "op needs a scheme that was not given");
    return CFD_ERR_ARG;
  }
  for (int d = 0; d < 2; ++d) {
    const SchemeCoef &s = B->s[d];
    if (!(mask & (d ? 0x38 : 0x1C7))) continue;
    if (!((s.M == 3 && (s.h == 4 || s.h == 5)) || (s.M == 2 && s.h == 4) || (s.M == 1 && s.h == 3))) {
      set_error("banded path: unsupported stencil widths (M, closure half-width)");
      return CFD_ERR_UNSUPPORTED;
    }
  }
  const bool f32 = B->dtype == CFD_F32;
  const size_t all_elems = region_elems + halo_elems;
  double *all = region_elems ? region : halo;
  for (size_t gi = 0; gi < B->sizes.size(); ++gi) {
    const int N = B->sizes[gi], g = B->ng;
    const std::vector<int> &blocks = B->groups[gi];
    const long long per = (long long)blocks.size() * nf, n3 = (long long)N * N * N;
    const PencilTab *tabs = static_cast<const PencilTab *>(B->d_ptab[gi]);
    PencilArgs A;
    memset(&A, 0, sizeof(A));
    A.field = fields;
    A.out = out;
    A.region = region;
    A.blocks = B->d_groups[gi];
    A.lidx = B->d_lidx;
    A.nbr = B->d_nbr;
    A.extpre = B->d_extpre;
    A.intpre = B->d_intpre;
    A.scale = B->d_scale;
    A.nblk = (int)blocks.size();
    A.nf = nf;
    A.nops = ol.n;
    A.g = g;
    // blocks that are their own neighbour along an axis (no halo passes there): all, none or some
    bool cyc[3], some[3];
    for (int a = 0; a < 3; ++a) {
      size_t n = 0;
      for (int b : blocks)
        if (B->nbr[b * 26 + dir_index(-(a == 0), -(a == 1), -(a == 2))] == b &&
            B->nbr[b * 26 + dir_index(a == 0, a == 1, a == 2)] == b)
          ++n;
      cyc[a] = n == blocks.size();
      some[a] = n > 0 && !cyc[a];
    }
    auto half_width = [&](const PencilTask &t) { return B->s[t.tab - tabs >= 6 ? 1 : 0].M; };
    // tasks in as few launches as their number and the halo space allow
    auto run = [&](std::vector<PencilTask> ts, double *hbase, size_t hcap) -> cfd_status {
      const int bufs = n_iter > 1 ? 2 : 1;
      for (size_t k = 0, n = ts.size(); k < n; ++k)
        if (some[ts[k].axis]) {  // cyclic and other blocks in two tasks
          ts[k].only = 2;
          ts.push_back(ts[k]);
          ts.back().only = 1;
          ts.back().cyclic = 1;
        }
      for (size_t i = 0; i < ts.size();) {
        size_t used = 0, j = i;
        std::vector<long long> off;
        // (one launch has one interior half-width: degrees of different widths go apart)
        while (j < ts.size() && j - i < (size_t)kMaxTasks && half_width(ts[j]) == half_width(ts[i])) {
          const size_t need = n_iter && !cyc[ts[j].axis] && ts[j].only != 1 ? (size_t)ts[j].n1 * ts[j].n2 * per * 2 : 0;
          if (used + bufs * need > hcap && need) {
            if (j == i) { set_error("banded path: halo space too small"); return CFD_ERR_ARG; }
            break;
          }
          off.push_back((long long)used);
          used += bufs * need;
          ++j;
        }
        A.halo = hbase;
        for (int pass = 0; pass <= n_iter; ++pass) {
          const bool hp = pass < n_iter;
          A.pass = pass;
          A.ntask = 0;
          for (size_t k = i; k < j; ++k) {
            if (hp && (cyc[ts[k].axis] || ts[k].only == 1)) continue;
            PencilTask t = ts[k];
            const long long len = (long long)t.n1 * t.n2 * per * 2;
            t.halo_in = off[k - i] + (bufs == 2 ? ((pass - 1) & 1) * len : 0);
            t.halo_out = off[k - i] + (bufs == 2 ? (pass & 1) * len : 0);
            A.task[A.ntask++] = t;
          }
          cfd_status s = launch_pencils(A, hp, f32, N, half_width(ts[i]), st);
          if (s != CFD_OK) return s;
        }
        i = j;
      }
      return CFD_OK;
    };
    auto pencils = [&](int axis, int deg, bool half) {
      PencilTask t;
      memset(&t, 0, sizeof(t));
      t.tab = tabs + ptab_index(deg, axis, half);
      const PencilTab &T = B->h_ptab[gi][ptab_index(deg, axis, half)];
      t.N = T.N;
      t.W = T.W;
      t.h = T.h;
      t.deg = T.deg;
      t.anti = T.anti;
      t.unscaled = T.unscaled;
      t.cyclic = cyc[axis];
      t.axis = axis;
      t.t1 = axis == 0 ? 1 : 0;
      t.t2 = axis == 2 ? 1 : 2;
      t.n1 = t.n2 = N;
      t.out_op = -1;
      t.sc_off = -1;
      t.in_op = -1;
      return t;
    };
    // outer axes that follow each inner axis, and their ops
    std::vector<std::pair<int, int>> outer[3];  // [inner axis]: (outer axis, op slot)
    for (int mi = 0; mi < 3; ++mi) {
      const int o = slot(6 + mi);
      if (o < 0) continue;
      outer[kMixed[mi][1]].push_back({kMixed[mi][0], o});
      if (!B->mixed_one_order) outer[kMixed[mi][0]].push_back({kMixed[mi][1], o});
    }
    std::vector<PencilTask> ts;
    for (int bit = 0; bit < 6; ++bit) {
      const int o = slot(bit), a = kAxisOfOp1[bit % 3];
      if (o < 0 || (bit < 3 && f32 && !outer[a].empty())) continue;  // (computed with its FP64 copy below)
      PencilTask t = pencils(a, bit < 3 ? 1 : 2, false);
      t.out_op = o;
      ts.push_back(t);
    }
    cfd_status s = run(ts, all, all_elems);
    if (s != CFD_OK) return s;
    bool written[9] = {};
    for (int j = 0; j < 3; ++j) {
      const int oj = slot(2 - j);  // op bit of d_j: x (box axis 2) is bit 0
      const bool in_out = oj >= 0 && !f32;
      const long long strip = 2ll * g * N * N * per, base = in_out ? 0 : n3 * per;
      for (size_t k = 0; k < outer[j].size();) {
        size_t n = std::min(outer[j].size() - k, (size_t)((region_elems - base) / strip));
        if (n == 0) { set_error("banded path: scratch too small"); return CFD_ERR_ARG; }
        ts.clear();
        if (k == 0 && !in_out) {
          PencilTask t = pencils(j, 1, false);
          t.out_op = oj;
          t.sc_off = 0;
          ts.push_back(t);
        }
        for (size_t u = 0; u < n; ++u) {
          PencilTask t = pencils(j, 1, false);
          t.strip = outer[j][k + u].first == t.t1 ? 1 : 2;
          (t.strip == 1 ? t.n1 : t.n2) = 2 * g;
          t.sc_off = base + (long long)u * strip;
          ts.push_back(t);
        }
        if ((s = run(ts, halo, halo_elems)) != CFD_OK) return s;
        ts.clear();
        for (size_t u = 0; u < n; ++u) {
          const int op = outer[j][k + u].second;
          PencilTask t = pencils(outer[j][k + u].first, 1, !B->mixed_one_order);
          t.gather = 1;
          t.in_op = in_out ? oj : -1;
          t.strip_off = base + (long long)u * strip;
          t.out_op = op;
          t.accum = written[op];
          written[op] = true;
          ts.push_back(t);
        }
        if ((s = run(ts, halo, halo_elems)) != CFD_OK) return s;
        k += n;
      }
    }
  }
  return CFD_OK;
}

}  // namespace
}  // namespace cfd

using namespace cfd;

extern "C" {

const char *cfd_last_error(void) { return g_err.c_str(); }

cfd_status cfd_scheme_create(const cfd_scheme_desc *first, const cfd_scheme_desc *second, cfd_scheme_t *out) {
  if (!out || (!first && !second)) { set_error("cfd_scheme_create: null argument"); return CFD_ERR_ARG; }
  cfd_scheme_s *s = new (std::nothrow) cfd_scheme_s();
  if (!s) { set_error("out of host memory"); return CFD_ERR_ALLOC; }
  cfd_status st = copy_desc(first, 1, s->s[0]);
  if (st == CFD_OK) st = copy_desc(second, 2, s->s[1]);
  if (st != CFD_OK) { delete s; return st; }
  *out = s;
  return CFD_OK;
}

cfd_status cfd_scheme_closure(cfd_scheme_t scheme, int deriv, double *closure, int *halfwidth) {
  if (!scheme || (deriv != 1 && deriv != 2) || !closure || !halfwidth) {
    set_error("cfd_scheme_closure: bad argument");
    return CFD_ERR_ARG;
  }
  const SchemeCoef &s = scheme->s[deriv - 1];
  if (!s.present) { set_error("cfd_scheme_closure: degree not present"); return CFD_ERR_ARG; }
  *halfwidth = s.h;
  for (int i = 0; i < 2 * s.h + 1; ++i) closure[i] = s.clo[i];
  return CFD_OK;
}

void cfd_scheme_destroy(cfd_scheme_t scheme) { delete scheme; }

void cfd_blocks_destroy(cfd_blocks_t B) {
  if (!B) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(B->device);
  cudaFree(B->d_nbr);
  cudaFree(B->d_extpre);
  cudaFree(B->d_exch);
  cudaFree(B->d_intpre);
  cudaFree(B->d_scale);
  cudaFree(B->d_nvec);
  cudaFree(B->d_status);
  for (int *p : B->d_groups) cudaFree(p);
  for (void *p : B->d_ptab) cudaFree(p);
  cudaFree(B->d_lidx);
  for (void *p : B->d_dense_ptrs) cudaFree(p);
  if (B->dense_state && B->dense_free) B->dense_free(B->dense_state);
  cudaSetDevice(prev);
  delete B;
}

cfd_status cfd_blocks_bind(cfd_scheme_t scheme, int nblocks, const int *block_n, const double *dx,
                           const int *neighbors, int ng, cfd_dtype dtype, cfd_blocks_t *out) {
  if (!scheme || nblocks < 1 || !block_n || !dx || !neighbors || !out) {
    set_error("cfd_blocks_bind: null or empty argument");
    return CFD_ERR_ARG;
  }
  if (dtype != CFD_F64 && dtype != CFD_F32) { set_error("cfd_blocks_bind: dtype"); return CFD_ERR_ARG; }
  int need = 0;
  for (int d = 0; d < 2; ++d) {
    const SchemeCoef &s = scheme->s[d];
    if (s.present) need = std::max(need, std::max(s.h, s.M + 1));
  }
  if (ng < need || ng > 8) { set_error("cfd_blocks_bind: ghost width too small for the stencils (or > 8)"); return CFD_ERR_ARG; }
  cfd_blocks_s *B = new (std::nothrow) cfd_blocks_s();
  if (!B) { set_error("out of host memory"); return CFD_ERR_ALLOC; }
  B->s[0] = scheme->s[0];
  B->s[1] = scheme->s[1];
  B->biased = scheme->biased;
  cudaGetDevice(&B->device);
  if (cudaDeviceGetAttribute(&B->num_sms, cudaDevAttrMultiProcessorCount, B->device) != cudaSuccess) B->num_sms = 0;
  B->nblocks = nblocks;
  B->ng = ng;
  B->dtype = dtype;
  B->n.assign(block_n, block_n + nblocks);
  B->nbr.assign(neighbors, neighbors + (size_t)nblocks * 26);
  B->dx.assign(dx, dx + (size_t)nblocks * 3);
  auto fail = [&](cfd_status s, const char *msg) {
    if (msg) set_error(msg);
    cfd_blocks_destroy(B);
    return s;
  };
  for (int b = 0; b < nblocks; ++b) {
    const int N = B->n[b];
    if (N != 8 && N != 16 && N != 32) return fail(CFD_ERR_UNSUPPORTED, "cfd_blocks_bind: block size must be 8, 16 or 32");
    if (N < ng) return fail(CFD_ERR_ARG, "cfd_blocks_bind: N < ng");
    for (int a = 0; a < 3; ++a)
      if (!(B->dx[b * 3 + a] > 0)) return fail(CFD_ERR_ARG, "cfd_blocks_bind: dx must be positive");
    for (int r = 0; r < 26; ++r) {
      const int nb = B->nbr[b * 26 + r];
      if (nb < -1 || nb >= nblocks) return fail(CFD_ERR_ARG, "cfd_blocks_bind: neighbour index out of range");
      if (nb >= 0 && B->n[nb] != N) return fail(CFD_ERR_ARG, "cfd_blocks_bind: neighbour of another size (pass -1)");
    }
    // iteration needs face neighbours along every axis that is not cyclic
    for (int a = 0; a < 3; ++a) {
      const int dz = a == 0, dy = a == 1, dxx = a == 2;
      const int lo = B->nbr[b * 26 + dir_index(-dz, -dy, -dxx)], hi = B->nbr[b * 26 + dir_index(dz, dy, dxx)];
      if (lo == b && hi == b) continue;
      if (lo < 0 || hi < 0 || lo == b || hi == b) B->iter_ok = false;
    }
  }
  // prefix offsets
  B->extpre.resize(nblocks);
  B->intpre.resize(nblocks);
  long long e = 0, i = 0;
  for (int b = 0; b < nblocks; ++b) {
    B->extpre[b] = e;
    B->intpre[b] = i;
    const long long N = B->n[b], E = N + 2 * ng;
    e += E * E * E;
    i += N * N * N;
  }
  // groups by size
  std::map<int, std::vector<int>> gm;
  for (int b = 0; b < nblocks; ++b) gm[B->n[b]].push_back(b);
  for (auto &kv : gm) {
    B->sizes.push_back(kv.first);
    B->groups.push_back(kv.second);
    if (B->biased.present) {
      BiasedTables bt;
      build_biased_tables(B->biased, kv.first, ng, bt);
      B->btab.push_back(bt);
    }
  }
  // per-block scale 1/dx^d, [b][deg][axis x,y,z]
  std::vector<double> scale((size_t)nblocks * 6);
  for (int b = 0; b < nblocks; ++b)
    for (int a = 0; a < 3; ++a) {
      const double h = B->dx[b * 3 + a];
      scale[(b * 2 + 0) * 3 + a] = 1.0 / h;
      scale[(b * 2 + 1) * 3 + a] = 1.0 / (h * h);
    }
  cfd_status s;
  if ((s = upload(&B->d_nbr, B->nbr.data(), B->nbr.size())) != CFD_OK) return fail(s, nullptr);
  if ((s = upload(&B->d_extpre, B->extpre.data(), B->extpre.size())) != CFD_OK) return fail(s, nullptr);
  if ((s = upload(&B->d_intpre, B->intpre.data(), B->intpre.size())) != CFD_OK) return fail(s, nullptr);
  if ((s = upload(&B->d_scale, scale.data(), scale.size())) != CFD_OK) return fail(s, nullptr);
  if ((s = upload(&B->d_nvec, B->n.data(), B->n.size())) != CFD_OK) return fail(s, nullptr);
  for (auto &grp : B->groups) {
    int *p = nullptr;
    if ((s = upload(&p, grp.data(), grp.size())) != CFD_OK) return fail(s, nullptr);
    B->d_groups.push_back(p);
    bool consecutive = true;
    for (size_t k = 0; k < grp.size(); ++k)
      if (grp[k] != grp[0] + (int)k) consecutive = false;
    B->group_b0.push_back(consecutive ? grp[0] : -1);
  }
  // FP64 banded tables: spacing equal in a group is folded into them
  std::vector<int> lidx(nblocks);
  for (size_t gi = 0; gi < B->groups.size(); ++gi) {
    const std::vector<int> &grp = B->groups[gi];
    for (size_t k = 0; k < grp.size(); ++k) lidx[grp[k]] = (int)k;
    std::vector<PencilTab> tabs(9);
    for (int box = 0; box < 3; ++box) {
      const double h = B->dx[grp[0] * 3 + 2 - box];
      bool equal = true;
      for (int b : grp)
        if (B->dx[b * 3 + 2 - box] != h) equal = false;
      for (int d = 1; d <= 2; ++d) {
        if (!B->s[d - 1].present) continue;
        const ld scale = d == 1 ? 1.0L / h : 1.0L / ((ld)h * h);
        for (int half = 0; half < (d == 1 ? 2 : 1); ++half) {
          int same = -1;  // an axis with the same spacing has the same table
          for (int pb = 0; pb < box; ++pb)
            if (equal && B->dx[grp[0] * 3 + 2 - pb] == h && !tabs[ptab_index(d, pb, half != 0)].unscaled) same = pb;
          PencilTab &T = tabs[ptab_index(d, box, half != 0)];
          if (same >= 0) T = tabs[ptab_index(d, same, half != 0)];
          else build_pencil_tab(B->s[d - 1], grp.empty() ? 0 : B->n[grp[0]], scale, !equal, half ? 0.5 : 1.0, T);
        }
      }
    }
    PencilTab *p = nullptr;
    if ((s = upload(&p, tabs.data(), tabs.size())) != CFD_OK) return fail(s, nullptr);
    B->d_ptab.push_back(p);
    B->h_ptab.push_back(std::move(tabs));
  }
  if ((s = upload(&B->d_lidx, lidx.data(), lidx.size())) != CFD_OK) return fail(s, nullptr);
  {
    std::vector<long long> exch((size_t)nblocks * 27);
    for (int b = 0; b < nblocks; ++b) {
      for (int d = 0; d < 26; ++d) {
        const int nb = B->nbr[(size_t)b * 26 + d];
        exch[(size_t)b * 27 + d] = nb >= 0 ? B->extpre[nb] : -1;
      }
      exch[(size_t)b * 27 + 26] = B->extpre[b];
    }
    if ((s = upload(&B->d_exch, exch.data(), exch.size())) != CFD_OK) return fail(s, nullptr);
  }
  if ((s = cuda_fail(cudaMalloc((void **)&B->d_status, sizeof(int)), "cudaMalloc")) != CFD_OK) return fail(s, nullptr);
  if ((s = cuda_fail(cudaMemset(B->d_status, 0, sizeof(int)), "cudaMemset")) != CFD_OK) return fail(s, nullptr);
  if ((s = dense_bind(B)) != CFD_OK) return fail(s, nullptr);
  *out = B;
  return CFD_OK;
}

cfd_status cfd_exchange_ghosts(cfd_blocks_t B, void *fields, int nfields, void *stream) {
  if (!B || !fields || nfields < 1) { set_error("cfd_exchange_ghosts: bad argument"); return CFD_ERR_ARG; }
  return launch_exchange(B, fields, nfields, (cudaStream_t)stream);
}

cfd_status cfd_apply_workspace(cfd_blocks_t B, int nfields, unsigned op_mask, cfd_precision prec, int n_iter,
                               size_t *bytes) {
  if (!B || nfields < 1 || !bytes || (op_mask & ~CFD_OP_ALL) || !op_mask || n_iter < 0) {
    set_error("cfd_apply_workspace: bad argument");
    return CFD_ERR_ARG;
  }
  if (prec == CFD_FP64_BANDED) {
    size_t sc, ha;
    banded_workspace_sizes(B, nfields, op_mask, n_iter, &sc, &ha);
    *bytes = align256(sc * 8) + 2 * align256(ha * 8) + 256;
    return CFD_OK;
  }
  return dense_workspace(B, nfields, op_mask, prec, n_iter, bytes);
}

cfd_status cfd_apply(cfd_blocks_t B, const void *fields, int nfields, unsigned op_mask, cfd_precision prec,
                     int n_iter, void *out, void *work, size_t work_bytes, void *stream) {
  if (!B || !fields || !out || nfields < 1 || !op_mask || (op_mask & ~CFD_OP_ALL) || n_iter < 0 || n_iter > 64) {
    set_error("cfd_apply: bad argument");
    return CFD_ERR_ARG;
  }
  if (n_iter > 0 && !B->iter_ok) {
    set_error("cfd_apply: hybrid iteration needs same-size face neighbours on every decomposed axis");
    return CFD_ERR_UNSUPPORTED;
  }
  for (auto &grp : B->groups)
    if ((long long)grp.size() * nfields > 65535) {
      set_error("cfd_apply: blocks of one size x nfields exceeds 65535");
      return CFD_ERR_UNSUPPORTED;
    }
  size_t need = 0;
  cfd_status s = cfd_apply_workspace(B, nfields, op_mask, prec, n_iter, &need);
  if (s != CFD_OK) return s;
  if (need > 256 && (!work || work_bytes < need)) {
    set_error("cfd_apply: workspace too small (see cfd_apply_workspace)");
    return CFD_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (prec == CFD_FP64_BANDED) {
    size_t sc, ha;
    banded_workspace_sizes(B, nfields, op_mask, n_iter, &sc, &ha);
    double *scratch = (double *)(((uintptr_t)work + 255) & ~(uintptr_t)255);
    const size_t sc_elems = align256(sc * 8) / 8, ha_elems = 2 * align256(ha * 8) / 8;
    return apply_banded(B, fields, nfields, op_mask, n_iter, out, scratch, sc_elems, scratch + sc_elems, ha_elems, st);
  }
  return dense_apply(B, fields, nfields, op_mask, prec, n_iter, out, work, work_bytes, st);
}

cfd_status cfd_autotune(cfd_blocks_t B, const void *fields, int nfields, unsigned op_mask, cfd_precision prec,
                        int n_iter, void *out, void *work, size_t work_bytes, void *stream) {
  if (!B || prec == CFD_FP64_BANDED) {
    set_error("cfd_autotune: a blocks handle and a tensor-core precision are needed");
    return CFD_ERR_ARG;
  }
  dense_set_tuning(B, true);
  const cfd_status s = cfd_apply(B, fields, nfields, op_mask, prec, n_iter, out, work, work_bytes, stream);
  dense_set_tuning(B, false);
  return s;
}

cfd_status cfd_autotune_report(cfd_blocks_t B, char *buf, size_t len, size_t *needed) {
  if (!B || (!buf && len) || !needed) { set_error("cfd_autotune_report: bad argument"); return CFD_ERR_ARG; }
  const std::string r = dense_tuning_report(B);
  *needed = r.size() + 1;
  if (buf && len) {
    const size_t n = std::min(len - 1, r.size());
    memcpy(buf, r.data(), n);
    buf[n] = 0;
  }
  return CFD_OK;
}

cfd_status cfd_blocks_set_mixed_order(cfd_blocks_t B, int one_order) {
  if (!B || (one_order != 0 && one_order != 1)) {
    set_error("cfd_blocks_set_mixed_order: bad argument");
    return CFD_ERR_ARG;
  }
  if (one_order && !B->iter_ok) {
    set_error("cfd_blocks_set_mixed_order: one order needs same-size face neighbours on every decomposed axis");
    return CFD_ERR_UNSUPPORTED;
  }
  B->mixed_one_order = one_order != 0;
  return CFD_OK;
}

cfd_status cfd_sync_status(cfd_blocks_t B, void *stream) {
  if (!B) { set_error("cfd_sync_status: null handle"); return CFD_ERR_ARG; }
  cfd_status s = cuda_fail(cudaStreamSynchronize((cudaStream_t)stream), "cudaStreamSynchronize");
  if (s != CFD_OK) return s;
  int v = 0;
  s = cuda_fail(cudaMemcpy(&v, B->d_status, sizeof(int), cudaMemcpyDeviceToHost), "cudaMemcpy status");
  if (s != CFD_OK) return s;
  if (v == 0) return CFD_OK;
  cudaMemset(B->d_status, 0, sizeof(int));
  set_error(v == CFD_ERR_TIMEOUT ? "device: bounded wait ran out" : "device: self-check failed");
  return v == CFD_ERR_TIMEOUT ? CFD_ERR_TIMEOUT : CFD_ERR_DEVICE_ASSERT;
}

}  // extern "C"

// Internal hooks for the allocation-free entry point (static_scratch.cu):
// the FP64 banded apply with closures only, running on a caller-provided
// scratch region instead of the workspace argument.
namespace cfd {

size_t banded_closed_scratch_bytes(const cfd_blocks_s *B, int nf, unsigned mask) {
  size_t sc = 0, ha = 0;
  banded_workspace_sizes(B, nf, mask, 0, &sc, &ha);
  return sc * sizeof(double);
}

cfd_status apply_banded_closed(cfd_blocks_s *B, const void *fields, int nf, unsigned mask, void *out,
                               double *scratch, cudaStream_t st) {
  return apply_banded(B, fields, nf, mask, 0, out, scratch, banded_closed_scratch_bytes(B, nf, mask) / sizeof(double),
                      nullptr, 0, st);
}

}  // namespace cfd
