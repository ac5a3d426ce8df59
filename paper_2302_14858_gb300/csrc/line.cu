// FP64 banded path: the per-pencil closed / iterated / cyclic tridiagonal solves (Eqs. sch_cent_om,
// iter_center_P), one thread per pencil.
//
// What bounds it: GB300's FP64 pipe, one warp instruction per 64 cycles and SM sub-partition.  Every
// other instruction hides behind that, so the kernel is written for few FP64 operations and enough
// warps, not for few instructions:
//   - the pencil sits in shared memory ([point][lane], 33 lanes wide: conflict-free along either
//     index), rows run in rolled loops with few registers, 16 to 24 warps per SM;
//   - a row is its stencil (three differences and three FMAs for an odd stencil with M = 3, seven FMAs
//     for an even one), one FMA forward and one back, and for an even stencil the pivot (line.h): 8 or
//     10 operations, 11 before;
//   - the passes of the hybrid iteration that only feed the neighbours compute the two values the
//     neighbours read, as two rows of the dense operator (~2 N FMAs per pencil instead of a solve);
//   - along x, pencils are rows: a warp loads and stores its 32 rows with consecutive lanes on
//     consecutive points and turns them in shared memory;
//   - pencils and tables arrive by asynchronous copies, all in flight at once.
// Mixed derivatives take the inner derivative from the d_j output (or one FP64 copy of it) and only
// the ghost strips are solved again, where the version before solved the extended pencils for each of
// the six ordered pairs.  128^3 as 512 blocks of 16^3, 4 fields, nine ops, one iteration: 8.41 -> 3.03 ms
// (526 -> ~150 FP64 operations per point); 27 blocks of 16^3, one field: 447 -> 156 us in 15 launches
// instead of 37.  Small launches are a chain of latencies: d_x and d_xx of 2^3 blocks of 8^3 take 6.0 and 7.1 us
// (8.4 and 9.1 with loads eight at a time and the table through registers), of 16^3 8.4 and 10.0 (11.7, 13.1).
#include <stddef.h>

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
constexpr int kTabDoubles = (kMaxN + 2) * (2 * 3 + 1) + 4 * (kMaxN + 2) + 2 * kMaxH + 1 + kTabScalars;  // M <= 3

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
// The two closure rows (half-width h), at points p and q: two chains side by side.
template <bool anti>
__device__ __forceinline__ void closure_rows(double &s, double &t, const double *c, const double *p, const double *q,
                                             int h, double neg, double nil) {
  s = t = nil;
  if constexpr (anti) {
#pragma unroll
    for (int m = 5; m >= 1; --m) {
      if (m > h) continue;
      s = fma(c[h + m], fma(p[-m * kPitch], neg, p[m * kPitch]), s);
      t = fma(c[h + m], fma(q[-m * kPitch], neg, q[m * kPitch]), t);
    }
  } else {
#pragma unroll
    for (int m = -5; m <= 5; ++m) {
      if (m < -h || m > h) continue;
      s = fma(c[h + m], p[m * kPitch], s);
      t = fma(c[h + m], q[m * kPitch], t);
    }
  }
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

// 32 rows (one per lane, pointer `mine`, n elements each) with consecutive lanes on consecutive elements:
// f(pointer of the row, row, element) for the rows that are not null, U of them side by side.
template <int U, typename P, typename F>
__device__ __forceinline__ void for_rows(P *mine, int n, F f) {
  const int dr = 32 / n, dj = 32 - dr * n, lane = threadIdx.x & 31;
  int r = lane / n, j = lane - r * n;
  for (int i = 0; i < n; i += U) {
    P *row[U];
    int rr[U], jj[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      rr[u] = r & 31;
      jj[u] = j;
      row[u] = reinterpret_cast<P *>(__shfl_sync(0xffffffffu, (long long)mine, rr[u]));
      if (i + u >= n) row[u] = nullptr;
      r += dr;
      j += dj;
      if (j >= n) {
        j -= n;
        ++r;
      }
    }
    f(row, rr, jj);
  }
}

// Copies that need no register until the wait: a launch of few warps has a whole pencil and its table in
// flight at once (eight loads at a time took a memory latency per batch).
__device__ __forceinline__ void copy_async(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async(double *dst, const float *src) {  // (into the low half: widened later)
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// (double)f by integer instructions for zeros and normal values (a conversion holds the FP64 pipe for 64 cycles).
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), e = u & 0x7F800000u;
  if ((e == 0 && (u << 1) != 0) || e == 0x7F800000u) return (double)f;
  const unsigned hi = (u & 0x80000000u) | (e ? ((u & 0x7FFFFFFFu) >> 3) + (896u << 20) : 0u);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// T: field dtype.  M > 0: solve (interior half-width M); M = 0: a halo pass, which writes the two values
// the neighbours read.  The table's part that the CTA needs is copied to shared memory first (read row by
// row from memory it cost a miss per row: half the time of a small launch).  Registers: with 80 allowed
// (6 CTAs per SM) the 128^3 case takes 3.03 ms; left to itself the compiler takes 64 and spills, 3.21.
template <typename T, int M>
__global__ void __launch_bounds__(kLineWarps * 32, 6) k_line(const __grid_constant__ PencilArgs A) {
  extern __shared__ double line_smem[];
  const PencilTask &K = A.task[blockIdx.y];
  const PencilTab &tab = *K.tab;
  const int N = K.N, W = K.W, L = N + 2 * W, g = A.g;
  const bool cyc = K.cyclic != 0, unscaled = K.unscaled != 0;
  const int lane = threadIdx.x & 31;
  constexpr bool HALO = M == 0;
  constexpr int CW = 2 * M + 1;
  // shared: closed or iterated rows [N + 2][CW], lo, up [N + 2] each, closure; cyclic rows, lo, up, z
  // (halo passes: the two operator rows), the scalars; then a tile per warp
  double *s_rc = line_smem, *s_lo = s_rc + (kMaxN + 2) * CW, *s_up = s_lo + kMaxN + 2, *s_clo = s_up + kMaxN + 2,
         *s_z = s_clo + 2 * kMaxH + 1, *s_pv = s_z + kMaxN + 2, *s_k = s_pv + kMaxN + 2;
  double *tile = line_smem + kTabDoubles + (threadIdx.x >> 5) * (L * kPitch);
  const int np = K.n1 * K.n2;
  // (the entry points admit 65535 blocks x fields of a size: fewer than 2^27 pencils)
  const int id = (int)(blockIdx.x * blockDim.x + threadIdx.x), npen = np * A.nblk * A.nf;
  if ((int)(blockIdx.x * blockDim.x) >= npen) return;  // (whole CTAs)
  bool valid = id < npen;
  const int job = valid ? id / np : 0, p = valid ? id - job * np : 0;
  // the table's part, in flight while the pencils are fetched; one barrier for both
  {
    const int t = threadIdx.x;
    if (HALO) {
      constexpr int HW = sizeof(tab.hrow[0][0]) / sizeof(double);
      const double *h = &tab.hrow[A.pass > 0][0][0];
      for (int i = t; i < 2 * HW; i += blockDim.x) copy_async(s_rc + i, h + i);
      if (t < 4) copy_async(s_k + t, &tab.hc[0][0] + t);
    } else {
      const bool iter = !cyc && A.pass > 0;
      const double(*rc)[2 * kMaxM + 1] = cyc ? tab.yrc : (iter ? tab.irc : tab.rc);
      const double *lo = cyc ? tab.ylo : (iter ? tab.ilo : tab.lo);
      const double *up = cyc ? tab.yup : (iter ? tab.iup : tab.up);
      const double *pv = cyc ? tab.ypv : (iter ? tab.ipv : tab.pv);
      const int rows = iter ? N + 2 : N;
      for (int i = t; i < rows * CW; i += blockDim.x) copy_async(s_rc + i, &rc[i / CW][i % CW]);
      if (t < rows) {
        copy_async(s_lo + t, lo + t);
        copy_async(s_up + t, up + t);
        copy_async(s_pv + t, pv + t);
        if (cyc) copy_async(s_z + t, &tab.z[t]);
      } else if (t >= 64 && t <= 64 + 2 * kMaxH) {
        copy_async(s_clo + t - 64, &tab.clo[t - 64]);
      } else if (t >= 96 && t < 96 + kTabScalars) {
        static_assert(offsetof(PencilTab, vfac) == offsetof(PencilTab, neg) + (kTabScalars - 1) * sizeof(double), "one run");
        copy_async(s_k + t - 96, &tab.neg + (t - 96));
      }
    }
  }
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
  // ---- the pencil: points -W .. N+W-1 at tile entries 0 .. L-1
  if (!K.gather) {
    const T *src = static_cast<const T *>(A.field) + (long long)A.nf * A.extpre[b] + (long long)q * E * E * E +
                   (c1 + g) * stride(K.t1, E) + (c2 + g) * stride(K.t2, E) + (long long)(g - W) * stride(ax, E);
    if (ax == 2) {
      for_rows<4>(valid ? src : nullptr, L, [&](const T *const(&row)[4], const int(&r)[4], const int(&k)[4]) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (row[u]) copy_async(tile + k[u] * kPitch + r[u], row[u] + k[u]);
      });
    } else if (valid) {
      const int s = stride(ax, E);
#pragma unroll 8
      for (int j = 0; j < L; ++j) copy_async(tile + j * kPitch + lane, src + (long long)j * s);
    }
  } else {
    // own points of the inner derivative (FP64: an output slot, or the scratch copy), ghosts from its strip
    const double *own = K.in_op >= 0 ? static_cast<const double *>(A.out) + (long long)A.nf * A.nops * A.intpre[b] +
                                           ((long long)q * A.nops + K.in_op) * n3
                                     : A.region + K.in_off + (long long)job * n3;
    own += c1 * stride(K.t1, N) + c2 * stride(K.t2, N);
    if (ax == 2) {
      for_rows<4>(valid ? own : nullptr, N, [&](const double *const(&row)[4], const int(&r)[4], const int(&k)[4]) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (row[u]) copy_async(tile + (W + k[u]) * kPitch + r[u], row[u] + k[u]);
      });
    } else if (valid) {
      const int s = stride(ax, N);
#pragma unroll 8
      for (int j = 0; j < N; ++j) copy_async(tile + (W + j) * kPitch + lane, own + (long long)j * s);
    }
    if (valid) {  // strip layout: [2g ghost points along the axis][N][N] (t1, t2)
      const double *st = A.region + K.strip_off + (long long)job * (2 * g * N * N) + c1 * N + c2;
#pragma unroll 4
      for (int j = 0; j < W; ++j) {
        copy_async(tile + j * kPitch + lane, st + (long long)(g - W + j) * N * N);
        copy_async(tile + (W + N + j) * kPitch + lane, st + (long long)(g + j) * N * N);
      }
    }
  }
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
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (sizeof(T) == 4 && !K.gather) {
#pragma unroll 8
    for (int j = 0; j < L; ++j) {
      double *e = tile + j * kPitch + lane;
      *e = widen(*reinterpret_cast<const float *>(e));
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
      double s0 = it ? fma(s_k[2 * w], dlo, s_k[2 * w + 1] * dhi) : 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
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
    const double neg = s_k[0], nil = s_k[1], factor = s_k[2], sc_k = s_k[3], isc = s_k[4], hhi = s_k[5], one = -neg;
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
      const double s = fma(-s_k[6], xn, x) * s_k[7];   // (x_0 - a x_{N-1}) vfac
      for (int k = 0; k < N; ++k) zrow[k * kPitch] = fma(-s, s_z[k], zrow[k * kPitch]);
      top = -1;
      up = pv = nullptr;
    } else if (closed) {
      closure_rows<anti>(x0, x, s_clo, f0, f0 + (N - 1) * kPitch, K.h, neg, nil);
      // (the closure rows take a zero times their neighbour, so a NaN or an infinity reaches the whole pencil)
      x = fma(nil, forward<M, anti>(s_rc + CW, s_lo + 1, f0, 1, N - 2, x0, neg, nil), scaled(x, sc_k));
      x0 = scaled(x0, sc_k);
      top = N - 2;
      up = s_up;
      pv = s_pv;
    } else {
      // row -1 starts from the fixed value: z_{-2} enters as hlo / lo times it
      z = forward<M, anti>(s_rc, s_lo, f0, -1, N + 2, scaled(factor * dlo, isc), neg, nil);
      x = fma(-hhi, dhi, scaled(z, s_pv[N + 1]));  // row N
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
        for_rows<4>(sc, N, [&](double *const(&row)[4], const int(&r)[4], const int(&k)[4]) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (row[u]) row[u][k[u]] = row0[k[u] * kPitch + r[u]];
        });
      if (K.out_op >= 0)
        for_rows<8>(out, N, [&](T *const(&row)[8], const int(&r)[8], const int(&k)[8]) {
          T old[8];
          if constexpr (ADD) {
#pragma unroll
            for (int u = 0; u < 8; ++u) old[u] = row[u] ? row[u][k[u]] : T(0);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (!row[u]) continue;
            double v = row0[k[u] * kPitch + r[u]];
            if constexpr (ADD) v = fma((double)old[u], one, v);
            row[u][k[u]] = (T)v;
          }
        });
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
