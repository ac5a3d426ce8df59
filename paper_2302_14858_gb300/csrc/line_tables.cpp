// Tables of the FP64 banded path (line.h), prepared in long double at bind time.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "line.h"

namespace cfd {

typedef long double ld;

void build_pencil_tab(const SchemeCoef &s, int N, ld scale, bool unscaled, double factor, PencilTab &T) {
  memset(&T, 0, sizeof(T));
  const int M = s.M, h = s.h;
  const ld a = s.a, sc = unscaled ? 1.0L : scale, f = factor;
  T.N = N;
  T.M = M;
  T.h = h;
  T.deg = s.d;
  T.W = std::max(h, M + 1);
  T.unscaled = unscaled;
  T.factor = factor;
  T.a = s.a;
  T.neg = -1.0;
  T.nil = 0.0;
  // antisymmetric to the last bit (the centre may hold the rounding of a zero)
  double mx = 0;
  for (int i = 0; i <= 2 * M; ++i) mx = std::max(mx, fabs(s.rhs[i]));
  T.anti = s.d == 1 && fabs(s.rhs[M]) <= 1e-25 * mx && fabs(s.clo[h]) <= 1e-25 * mx;
  for (int m = 1; m <= M; ++m)
    if (s.rhs[M - m] != -s.rhs[M + m]) T.anti = 0;
  for (int m = 1; m <= h; ++m)
    if (s.clo[h - m] != -s.clo[h + m]) T.anti = 0;
  // a row's coefficients with its factor v (antisymmetric) or as given (f is a power of two: exact)
  auto fold = [&](const double *src, int w, ld v, double *dst) {
    for (int i = 0; i <= 2 * w; ++i) dst[i] = T.anti ? (double)(src[i] * v) : src[i] * factor;
  };
  T.sc = T.anti ? 1.0 : (double)sc;
  T.isc = T.anti ? 1.0 : (double)(1.0L / sc);
  fold(s.clo, h, sc * f, T.clo);
  // LU of the rows in order: 1 / pivot inv, elimination factor a inv_{k-1} (folded rows: a inv_k)
  struct Row { ld inv, c; };
  auto row = [&](ld dd, ld lower, const Row &prev, double *rc, double &lo, double &up, double &pv, bool last) {
    Row r;
    r.inv = 1.0L / (dd - lower * prev.c);
    r.c = last ? 0.0L : a * r.inv;
    fold(s.rhs, M, sc * f * r.inv, rc);
    lo = (double)(T.anti ? lower * r.inv : lower * prev.inv);
    up = (double)r.c;
    pv = T.anti ? 1.0 : (double)(r.inv * sc);
    return r;
  };
  const Row unit = {1.0L, 0.0L};
  // closed
  Row p = unit;
  for (int k = 1; k < N - 1; ++k) p = row(1.0L, a, p, T.rc[k], T.lo[k], T.up[k], T.pv[k], false);
  // iterated: rows -1..N between the fixed values at -2 and N+1
  p = unit;
  for (int r = 0; r < N + 2; ++r) p = row(1.0L, a, p, T.irc[r], T.ilo[r], T.iup[r], T.ipv[r], false);
  T.hhi = (double)(p.c * f);
  // cyclic by Sherman-Morrison: A = T + u v^T with gamma = -1, T_00 = 2, T_{N-1,N-1} = 1 + a^2,
  // u = (-1, 0, .., a), v = (1, 0, .., -a)
  {
    std::vector<ld> y(N), cc(N);
    p = unit;
    for (int k = 0; k < N; ++k) {
      const ld dd = k == 0 ? 2.0L : (k == N - 1 ? 1.0L + a * a : 1.0L);
      p = row(dd, k ? a : 0.0L, p, T.yrc[k], T.ylo[k], T.yup[k], T.ypv[k], k == N - 1);
      cc[k] = p.c;
      const ld u = k == 0 ? -1.0L : (k == N - 1 ? a : 0.0L);
      y[k] = (u - (k ? a * y[k - 1] : 0.0L)) * p.inv;
    }
    for (int k = N - 2; k >= 0; --k) y[k] -= cc[k] * y[k + 1];
    for (int k = 0; k < N; ++k) T.z[k] = (double)y[k];
    T.vfac = (double)(1.0L / (1.0L + (y[0] - a * y[N - 1])));
  }
  // rows 1 and N-2 of the operators: solve the transposed systems A^T g = e_row, row = g^T B
  for (int it = 0; it < 2; ++it) {
    const int n = it ? N + 2 : N, k0 = it ? -1 : 0;  // rows k0 .. k0 + n - 1
    for (int w = 0; w < 2; ++w) {
      const int target = (w == 0 ? 1 : N - 2) - k0;
      auto off = [&](int r, int q) -> ld {  // A[r][q], tridiagonal; closed end rows are unit rows
        if (r == q) return 1.0L;
        if (!it && (r == 0 || r == n - 1)) return 0.0L;
        return a;
      };
      std::vector<ld> g(n, 0), cp(n, 0);
      ld den = 1.0L;  // Thomas on A^T: A^T[r][q] = A[q][r]
      for (int r = 0; r < n; ++r) {
        const ld l = r ? off(r - 1, r) : 0.0L, u = r < n - 1 ? off(r + 1, r) : 0.0L;
        den = 1.0L - l * (r ? cp[r - 1] : 0.0L);
        cp[r] = u / den;
        g[r] = ((r == target ? 1.0L : 0.0L) - (r ? l * g[r - 1] : 0.0L)) / den;
      }
      for (int r = n - 2; r >= 0; --r) g[r] -= cp[r] * g[r + 1];
      std::vector<ld> row(N + 2 * T.W, 0);
      for (int r = 0; r < n; ++r) {
        const int k = k0 + r;
        const bool end = !it && (k == 0 || k == N - 1);
        const int hw = end ? h : M;
        for (int m = -hw; m <= hw; ++m) row[k + m + T.W] += g[r] * (end ? s.clo[m + h] : s.rhs[m + M]) * sc;
      }
      for (size_t j = 0; j < row.size(); ++j) T.hrow[it][w][j] = (double)row[j];
      if (it) {  // the fixed values enter rows -1 and N as -a d
        T.hc[w][0] = (double)(-a * g[0]);
        T.hc[w][1] = (double)(-a * g[n - 1]);
      }
    }
  }
}

}  // namespace cfd
