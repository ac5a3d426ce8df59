// FP64 banded path: the per-pencil closed / iterated / cyclic tridiagonal solves (Eqs. sch_cent_om,
// iter_center_P), one thread per pencil.
//
// What bounds it: GB300's FP64 pipe, one warp instruction per 64 cycles and SM sub-partition.  Every
// other instruction hides behind that, so the kernel is written for few FP64 operations and enough
// warps, not for few instructions:
//   - the pencil sits in shared memory ([point][lane], 33 lanes wide: conflict-free along either
//     index), rows run in rolled loops with few registers, 20 to 36 warps per SM;
//   - a row is its stencil (three differences and three FMAs for an odd stencil with M = 3, seven FMAs
//     for an even one), one FMA forward and one back, and for an even stencil the pivot (line.h): 8 or
//     10 operations, 11 before;
//   - the passes of the hybrid iteration that only feed the neighbours compute the two values the
//     neighbours read, as two rows of the dense operator (~2 N FMAs per pencil instead of a solve);
//   - along x, pencils are rows: a warp loads and stores its 32 rows with consecutive lanes on
//     consecutive points and turns them in shared memory.
// Mixed derivatives take the inner derivative from the d_j output (or one FP64 copy of it) and only
// the ghost strips are solved again, where the version before solved the extended pencils for each of
// the six ordered pairs.  128^3 as 512 blocks of 16^3, 4 fields, nine ops, one iteration: 8.41 -> 3.65 ms
// (526 -> ~165 FP64 operations per point); 27 blocks of 16^3, one field: 447 -> 192 us in 15 launches
// instead of 37 (there latency counts: loads go out eight at a time, rows four at a time).
#include <algorithm>
#include <type_traits>

#include "line.h"

namespace cfd {

namespace {

// ---------------------------------------------------------------- kernels

__device__ __forceinline__ int dir_index(int dz, int dy, int dx) {
  int r = 9 * (dz + 1) + 3 * (dy + 1) + (dx + 1);
  return r > 13 ? r - 1 : r;
}

constexpr int kPitch = 33;   // lanes per point of a warp's tile, padded
constexpr int kLineWarps = 4;
constexpr int kTabDoubles = (kMaxN + 2) * (2 * 3 + 1) + 4 * (kMaxN + 2) + 2 * kMaxH + 1;  // M <= 3

// Every operation of the solves is an FMA of three register operands: on GB300 that form issues every
// 64 cycles per SM sub-partition, an add, a multiply or an FMA with a constant operand every 76
// (measured).  neg holds -1 and nil 0, loaded from memory so that they stay register operands.
//
// The stencils of R consecutive rows: r[u] = sum_m c[u][m] f_{k+u+m}, m = -M..M; p: the tile entry of
// point k of this lane, c: row k's coefficients, rows CW apart.  An antisymmetric stencil takes
// differences (its centre is zero: 2M operations instead of 2M + 1, and 13 % less rounding error
// measured); a symmetric one the plain chain, whose partial sums stay small (pair sums f_{k+m} + f_{k-m}
// cost as much and rounded 30 % worse).  R rows at a time are R independent chains: a row by row loop
// took 1.5 times as long where few warps share an SM.
template <int M, int R, bool anti>
__device__ __forceinline__ void stencils(double (&r)[R], const double *c, int cw, const double *p, double neg,
                                         double nil) {
  double f[R + 2 * M];
#pragma unroll
  for (int i = 0; i < R + 2 * M; ++i) f[i] = p[(i - M) * kPitch];
  if constexpr (anti) {
#pragma unroll
    for (int m = M; m >= 1; --m)
#pragma unroll
      for (int u = 0; u < R; ++u)
        r[u] = fma(c[u * cw + M + m], fma(f[u + M - m], neg, f[u + M + m]), m == M ? nil : r[u]);
  } else {
#pragma unroll
    for (int m = -M; m <= M; ++m)
#pragma unroll
      for (int u = 0; u < R; ++u) r[u] = fma(c[u * cw + M + m], f[u + M + m], m == -M ? nil : r[u]);
  }
}
// a closure row (half-width h <= kMaxH)
__device__ __forceinline__ double closure_row(const double *c, const double *p, int h, bool anti, double neg, double nil) {
  double s = nil;
  if (anti) {
    for (int m = h; m >= 1; --m) s = fma(c[h + m], fma(p[-m * kPitch], neg, p[m * kPitch]), s);
  } else {
    for (int m = -h; m <= h; ++m) s = fma(c[h + m], p[m * kPitch], s);
  }
  return s;
}

// Forward sweep over rows k0 .. k0 + n - 1 (n even): z_k = r_k - lo_k z_{k-1}, stored where point k - M
// was (the rows after k no longer read it).  c, lo: the first row's.
template <int M, bool anti>
__device__ __forceinline__ double forward(const double *c, const double *lo, double *f0, int k0, int n, double z,
                                          double neg, double nil) {
  constexpr int CW = 2 * M + 1;
  int i = 0;
  auto rows = [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    double r[R];
    stencils<M, R, anti>(r, c + i * CW, CW, f0 + (k0 + i) * kPitch, neg, nil);
#pragma unroll
    for (int u = 0; u < R; ++u) {
      z = fma(-lo[i + u], z, r[u]);
      f0[(k0 + i + u - M) * kPitch] = z;
    }
    i += R;
  };
  while (i + 4 <= n) rows(std::integral_constant<int, 4>());
  while (i < n) rows(std::integral_constant<int, 2>());
  return z;
}

// 32 rows (one per lane, pointer `mine`, n elements each) with consecutive lanes on consecutive elements,
// eight loads in flight: op(row, element, pointer of the row or null) returns what sink takes.
template <typename P, typename Load, typename Sink>
__device__ __forceinline__ void for_rows(P *mine, int n, Load load, Sink sink) {
  const int lane = threadIdx.x & 31;
  int r = 0, j = lane;
  for (int i = 0; i < n; i += 8) {
    double v[8];
    int rr[8], jj[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      while (j >= n) { j -= n; ++r; }
      rr[u] = r & 31;
      jj[u] = j;
      j += 32;
      P *row = reinterpret_cast<P *>(__shfl_sync(0xffffffffu, (long long)mine, rr[u]));
      v[u] = 0.0;
      if (i + u < n && row) v[u] = load(row, rr[u], jj[u]);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      P *row = reinterpret_cast<P *>(__shfl_sync(0xffffffffu, (long long)mine, rr[u]));
      if (i + u < n && row) sink(row, rr[u], jj[u], v[u]);
    }
  }
}

// T: field dtype.  M > 0: solve (interior half-width M); M = 0: a halo pass, which writes the two values
// the neighbours read.  The table's part that the CTA needs is copied to shared memory first (read row by
// row from memory it cost a miss per row: half the time of a small launch).
template <typename T, int M>
__global__ void __launch_bounds__(kLineWarps * 32) k_line(const __grid_constant__ PencilArgs A) {
  extern __shared__ double line_smem[];
  const PencilTask &K = A.task[blockIdx.y];
  const PencilTab &tab = *K.tab;
  const int N = K.N, W = K.W, L = N + 2 * W, g = A.g;
  const bool cyc = K.cyclic != 0, unscaled = K.unscaled != 0;
  const int lane = threadIdx.x & 31;
  constexpr bool HALO = M == 0;
  constexpr int CW = 2 * M + 1;
  // shared: closed or iterated rows [N + 2][CW], lo, up [N + 2] each, closure; cyclic rows, lo, up, z
  // (halo passes: the two operator rows); then a tile per warp
  double *s_rc = line_smem, *s_lo = s_rc + (kMaxN + 2) * CW, *s_up = s_lo + kMaxN + 2, *s_clo = s_up + kMaxN + 2,
         *s_z = s_clo + 2 * kMaxH + 1, *s_pv = s_z + kMaxN + 2;
  double *tile = line_smem + kTabDoubles + (threadIdx.x >> 5) * (L * kPitch);
  const int np = K.n1 * K.n2;
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if ((long long)blockIdx.x * blockDim.x >= (long long)np * A.nblk * A.nf) return;  // (whole CTAs)
  bool valid = id < (long long)np * A.nblk * A.nf;
  const int job = valid ? (int)(id / np) : 0, p = valid ? (int)(id - (long long)job * np) : 0;
  const int lb = job / A.nf, q = job - lb * A.nf, b = A.blocks[lb];
  const int i1 = p / K.n2, i2 = p - i1 * K.n2;
  // transverse point relative to the block's own points
  const int c1 = K.strip == 1 ? (i1 < g ? i1 - g : N + i1 - g) : i1;
  const int c2 = K.strip == 2 ? (i2 < g ? i2 - g : N + i2 - g) : i2;
  const int ax = K.axis, E = N + 2 * g;
  const long long n3 = (long long)N * N * N;
  auto stride = [](int axis, int n) { return axis == 0 ? n * n : (axis == 1 ? n : 1); };

  // the face neighbours (a block that is its own on both sides is a whole periodic line)
  const bool look = K.only || (!cyc && A.pass > 0);
  const int blo = look ? A.nbr[b * 26 + dir_index(-(ax == 0), -(ax == 1), -(ax == 2))] : 0;
  const int bhi = look ? A.nbr[b * 26 + dir_index(ax == 0, ax == 1, ax == 2)] : 0;
  if (K.only) valid = valid && (blo == b && bhi == b) == (K.only == 1);
  // (copied while the pencils are fetched; one barrier for both)
  if (HALO) {
    const double *h = &tab.hrow[A.pass > 0][0][0];
    constexpr int HW = sizeof(tab.hrow[0][0]) / sizeof(double);
    for (int i = threadIdx.x; i < 2 * HW; i += blockDim.x) s_rc[i] = __ldg(h + i);
  } else {
    const double(*rc)[2 * kMaxM + 1] = cyc ? tab.yrc : (A.pass > 0 ? tab.irc : tab.rc);
    const double *lo = cyc ? tab.ylo : (A.pass > 0 ? tab.ilo : tab.lo);
    const double *up = cyc ? tab.yup : (A.pass > 0 ? tab.iup : tab.up);
    const double *pv = cyc ? tab.ypv : (A.pass > 0 ? tab.ipv : tab.pv);
    const int rows = !cyc && A.pass > 0 ? N + 2 : N;
    for (int i = threadIdx.x; i < rows * CW; i += blockDim.x) s_rc[i] = __ldg(&rc[i / CW][i % CW]);
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
      s_lo[i] = __ldg(lo + i);
      s_up[i] = __ldg(up + i);
      s_pv[i] = __ldg(pv + i);
      if (cyc) s_z[i] = __ldg(&tab.z[i]);
    }
    if (threadIdx.x <= 2 * kMaxH) s_clo[threadIdx.x] = __ldg(&tab.clo[threadIdx.x]);
  }

  // ---- the pencil: points -W .. N+W-1 at tile entries 0 .. L-1
  if (!K.gather) {
    const T *src = static_cast<const T *>(A.field) + (long long)A.nf * A.extpre[b] + (long long)q * E * E * E +
                   (c1 + g) * stride(K.t1, E) + (c2 + g) * stride(K.t2, E) + (long long)(g - W) * stride(ax, E);
    if (ax == 2) {
      for_rows(valid ? src : nullptr, L, [](const T *row, int, int k) { return (double)__ldg(row + k); },
               [&](const T *, int r, int k, double v) { tile[k * kPitch + r] = v; });
    } else if (valid) {
      const int s = stride(ax, E);
#pragma unroll 8
      for (int j = 0; j < L; ++j) tile[j * kPitch + lane] = (double)__ldg(src + (long long)j * s);
    }
  } else {
    // own points of the inner derivative (FP64: an output slot, or the scratch copy), ghosts from its strip
    const double *own = K.in_op >= 0 ? static_cast<const double *>(A.out) + (long long)A.nf * A.nops * A.intpre[b] +
                                           ((long long)q * A.nops + K.in_op) * n3
                                     : A.region + K.in_off + (long long)job * n3;
    own += c1 * stride(K.t1, N) + c2 * stride(K.t2, N);
    // (plain loads: the derivative was written by an earlier launch on the stream, but `out` is written here)
    if (ax == 2) {
      for_rows(valid ? own : nullptr, N, [](const double *row, int, int k) { return row[k]; },
               [&](const double *, int r, int k, double v) { tile[(W + k) * kPitch + r] = v; });
    } else if (valid) {
      const int s = stride(ax, N);
#pragma unroll 8
      for (int j = 0; j < N; ++j) tile[(W + j) * kPitch + lane] = own[(long long)j * s];
    }
    if (valid) {  // strip layout: [2g ghost points along the axis][N][N] (t1, t2)
      const double *st = A.region + K.strip_off + (long long)job * (2 * g * N * N) + c1 * N + c2;
#pragma unroll 4
      for (int j = 0; j < W; ++j) {
        tile[j * kPitch + lane] = st[(long long)(g - W + j) * N * N];
        tile[(W + N + j) * kPitch + lane] = st[(long long)(g + j) * N * N];
      }
    }
  }
  __syncthreads();
  double *f0 = tile + W * kPitch + lane;  // point 0 of this lane's pencil
  const double scale = unscaled ? A.scale[(b * 2 + (K.deg - 1)) * 3 + (2 - ax)] : 1.0;
  // the neighbours' previous iterate at k^c = -2 and N+1 (their rows N-2 and 1)
  double dlo = 0.0, dhi = 0.0;
  if (valid && !cyc && A.pass > 0) {
    const int nlo = A.lidx[blo], nhi = A.lidx[bhi];
    const double *h = A.halo + K.halo_in;
    dlo = h[(((long long)nlo * A.nf + q) * np + p) * 2 + 1];
    dhi = h[(((long long)nhi * A.nf + q) * np + p) * 2 + 0];
    if (unscaled) {
      dlo /= scale;
      dhi /= scale;
    }
  }

  if constexpr (HALO) {
    if (!valid || cyc) return;
    const int it = A.pass > 0 ? 1 : 0;
    double *h = A.halo + K.halo_out + ((long long)job * np + p) * 2;
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      int j = 0;
      constexpr int HW = sizeof(tab.hrow[0][0]) / sizeof(double);
      const double *c = s_rc + w * HW, *f = tile + lane;
      double s0 = it ? fma(tab.hc[w][0], dlo, tab.hc[w][1] * dhi) : 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      for (; j + 4 <= L; j += 4) {
        s0 = fma(c[j], f[j * kPitch], s0);
        s1 = fma(c[j + 1], f[(j + 1) * kPitch], s1);
        s2 = fma(c[j + 2], f[(j + 2) * kPitch], s2);
        s3 = fma(c[j + 3], f[(j + 3) * kPitch], s3);
      }
      for (; j < L; ++j) s0 = fma(c[j], f[j * kPitch], s0);
      s0 = (s0 + s1) + (s2 + s3);
      h[w] = unscaled ? s0 * scale : s0;
    }
    return;
  } else {
    // (the stencil's kind and the output's are compile-time inside: left to run time, the compiler executes
    // both sides of a choice between operations and selects, two more per output)
    auto solve = [&](auto anti_c, auto add_c, auto unscaled_c) {
    constexpr bool anti = decltype(anti_c)::value, ADD = decltype(add_c)::value, UNSCALED = decltype(unscaled_c)::value;
    // ---- solve
    const double neg = __ldg(&tab.neg), nil = __ldg(&tab.nil), one = -neg;
    double *zrow = f0 - M * kPitch;
    const bool closed = !cyc && A.pass == 0;
    double x = 0.0, z = 0.0, x0 = 0.0;
    int top;                 // rows top .. 0 come back from z
    const double *up, *pv;   // x_k = pv[k] z_k - up[k] x_{k+1} (pv: rows that keep their coefficients)
    auto scaled = [&](double v, double p) { return anti ? v : fma(v, p, nil); };
    if (cyc) {
      z = forward<M, anti>(s_rc, s_lo, f0, 0, N, 0.0, neg, nil);
      x = scaled(z, s_pv[N - 1]);
      zrow[(N - 1) * kPitch] = x;
      const double xn = x;
      for (int k = N - 2; k >= 0; --k) {
        x = fma(-s_up[k], x, scaled(zrow[k * kPitch], s_pv[k]));
        zrow[k * kPitch] = x;
      }
      const double s = fma(-tab.a, xn, x) * tab.vfac;   // (x_0 - a x_{N-1}) vfac
      for (int k = 0; k < N; ++k) zrow[k * kPitch] = fma(-s, s_z[k], zrow[k * kPitch]);
      top = -1;
      up = pv = nullptr;
    } else if (closed) {
      x0 = closure_row(s_clo, f0, K.h, anti, neg, nil);
      x = closure_row(s_clo, f0 + (N - 1) * kPitch, K.h, anti, neg, nil);
      // (the closure rows take a zero times their neighbour, so a NaN or an infinity reaches the whole pencil)
      x = fma(nil, forward<M, anti>(s_rc + CW, s_lo + 1, f0, 1, N - 2, x0, neg, nil), scaled(x, tab.sc));
      x0 = scaled(x0, tab.sc);
      top = N - 2;
      up = s_up;
      pv = s_pv;
    } else {
      // row -1 starts from the fixed value: z_{-2} enters as hlo / lo times it
      z = forward<M, anti>(s_rc, s_lo, f0, -1, N + 2, scaled(tab.factor * dlo, tab.isc), neg, nil);
      x = fma(-tab.hhi, dhi, scaled(z, s_pv[N + 1]));  // row N
      top = N - 1;
      up = s_up + 1;
      pv = s_pv + 1;
    }
    // ---- outputs
    T *out = nullptr;
    double *sc = nullptr;
    long long sstr = 1;
    if (valid && K.out_op >= 0)
      out = static_cast<T *>(A.out) + (long long)A.nf * A.nops * A.intpre[b] + ((long long)q * A.nops + K.out_op) * n3 +
            c1 * stride(K.t1, N) + c2 * stride(K.t2, N);
    if (valid && K.sc_off >= 0) {
      if (!K.strip) {
        sc = A.region + K.sc_off + (long long)job * n3 + c1 * stride(K.t1, N) + c2 * stride(K.t2, N);
        sstr = stride(ax, N);
      } else {
        // strip of axis i (the strip's transverse axis): [2g][N][N] over the other two axes in order
        const int o = K.strip == 1 ? K.t2 : K.t1;        // the remaining transverse axis
        const int gi = K.strip == 1 ? i1 : i2, co = K.strip == 1 ? i2 : i1;
        sc = A.region + K.sc_off + (long long)job * (2 * g * N * N) + (long long)gi * N * N + co * (o < ax ? N : 1);
        sstr = ax < o ? N : 1;
      }
    }
    const long long ostr = stride(ax, N);
    const bool rows = ax == 2 && !K.strip;  // x pencils leave through the tile, row by row
    auto emit = [&](int k, double v, double old) {
      if constexpr (UNSCALED) v = fma(v, scale, nil);
      if (rows) {
        zrow[k * kPitch] = v;
        return;
      }
      if (sc) sc[k * sstr] = v;
      if (out) out[k * ostr] = (T)(ADD ? fma(old, one, v) : v);
    };
    auto before = [&](int k) { return ADD && out && !rows ? (double)out[k * ostr] : 0.0; };
    if (top < 0) {
      if (!rows || UNSCALED)
        for (int k = 0; k < N; ++k) emit(k, zrow[k * kPitch], before(k));
    } else {
      if (closed) {
        const double a = before(N - 1);
        emit(N - 1, x, a);
      }
      // four rows' loads at a time
      const int last = closed ? 1 : 0;
      int k = top;
      for (; k - 3 >= last; k -= 4) {
        double zz[4], uu[4], old[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { zz[u] = scaled(zrow[(k - u) * kPitch], pv[k - u]); uu[u] = up[k - u]; old[u] = before(k - u); }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          x = fma(-uu[u], x, zz[u]);
          emit(k - u, x, old[u]);
        }
      }
      for (; k >= last; --k) {
        const double old = before(k);
        x = fma(-up[k], x, scaled(zrow[k * kPitch], pv[k]));
        emit(k, x, old);
      }
      if (closed) emit(0, fma(nil, x, x0), before(0));
    }
    if (rows) {
      __syncwarp();
      const double *row0 = tile + (W - M) * kPitch;
      if (K.sc_off >= 0)
        for_rows(sc, N, [&](double *, int r, int k) { return row0[k * kPitch + r]; },
                 [](double *row, int, int k, double v) { row[k] = v; });
      if (K.out_op >= 0) {
        for_rows(out, N,
                 [&](T *row, int r, int k) { 
                   double v = row0[k * kPitch + r];
                   if constexpr (ADD) v = fma((double)row[k], one, v);
                   return v;
                 },
                 [](T *row, int, int k, double v) { row[k] = (T)v; });
      }
    }
    };
    using std::false_type;
    using std::true_type;
    if (unscaled) {
      if (K.anti) K.accum ? solve(true_type(), true_type(), true_type()) : solve(true_type(), false_type(), true_type());
      else K.accum ? solve(false_type(), true_type(), true_type()) : solve(false_type(), false_type(), true_type());
    } else if (K.anti) {
      K.accum ? solve(true_type(), true_type(), false_type()) : solve(true_type(), false_type(), false_type());
    } else {
      K.accum ? solve(false_type(), true_type(), false_type()) : solve(false_type(), false_type(), false_type());
    }
  }
}

}  // namespace

cfd_status launch_pencils(const PencilArgs &A, bool halo, bool f32, int N, int M, cudaStream_t st) {
  // Windows of the launch's own tasks: W <= 5 (the widths apply_banded admits) keeps N = 32 within the 48 KB
  // that need no opt-in; a scheme's other degree may be wider.
  long long most = 0;
  int W = 0;
  for (int t = 0; t < A.ntask; ++t) {
    most = std::max(most, (long long)A.task[t].n1 * A.task[t].n2 * A.nblk * A.nf);
    W = std::max(W, A.task[t].W);
  }
  if (most == 0 || A.ntask == 0) return CFD_OK;
  const dim3 grid((unsigned)((most + kLineWarps * 32 - 1) / (kLineWarps * 32)), (unsigned)A.ntask);
  const size_t smem = ((size_t)kLineWarps * (N + 2 * W) * kPitch + kTabDoubles) * sizeof(double);
  static_assert(((size_t)kLineWarps * (kMaxN + 2 * 5) * kPitch + kTabDoubles) * sizeof(double) <= 48 * 1024, "no opt-in");
  void (*fn)(const __grid_constant__ PencilArgs) = nullptr;
  switch (halo ? 0 : M) {
    case 0: fn = f32 ? k_line<float, 0> : k_line<double, 0>; break;
    case 1: fn = f32 ? k_line<float, 1> : k_line<double, 1>; break;
    case 2: fn = f32 ? k_line<float, 2> : k_line<double, 2>; break;
    case 3: fn = f32 ? k_line<float, 3> : k_line<double, 3>; break;
    default: set_error("banded path: interior half-width above 3"); return CFD_ERR_UNSUPPORTED;
  }
  launch_begin(KF_LINE, st);
  fn<<<grid, kLineWarps * 32, smem, st>>>(A);
  launch_end(KF_LINE, st);
  return cuda_fail(cudaGetLastError(), "k_line launch");
}

}  // namespace cfd
