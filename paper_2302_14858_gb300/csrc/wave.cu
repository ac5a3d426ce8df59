// Classical RK4 (ERK4) driver for the linear wave system
//   d/dt Phi = K,  d/dt K = sum_i D2_i Phi   (Eq. toyShiftWaveEqnSys, zero shift)
// on MeshBlocks, and the 2S low-storage driver with Kreiss-Oliger dissipation and shift terms.  Each
// stage: ghost exchange, the three second derivatives through cfd_apply, elementwise kernels.
//
// The elementwise kernels are bound by GB300's FP64 pipe as much as by memory (one warp operation per 64
// cycles and SM sub-partition: ten per point are 0.29 ms at 256^3, as long as 1.9 GB of traffic), so both
// are counted.  Adds are FMAs with a register operand 1, which issue every 64 cycles instead of 76.
#include <string.h>

#include <type_traits>

#include "cfd_internal.h"

namespace cfd {
namespace {

// V consecutive doubles (16-byte accesses for V = 2)
template <int V>
struct alignas(8 * V) Pack { double v[V]; };
template <int V>
__device__ __forceinline__ Pack<V> ld(const double *p) { return *reinterpret_cast<const Pack<V> *>(p); }
template <int V>
__device__ __forceinline__ void st(double *p, const Pack<V> &x) { *reinterpret_cast<Pack<V> *>(p) = x; }

// The constants of a kernel in shared memory: loaded from there they are register operands (an FMA with
// a constant-bank operand takes 76 cycles of the FP64 pipe instead of 64).
template <int C>
__device__ __forceinline__ void stage_constants(double (&s)[C], const double (&c)[C]) {
  if (threadIdx.x < C) s[threadIdx.x] = c[threadIdx.x];
  __syncthreads();
}

struct StageArgs {
  double *phi;          // field layout (ghosts) : the state Phi
  double *K;            // field layout          : the state K
  double *phis;         // field layout          : stage Phi (input of the next Laplacian)
  const double *lap;    // interior, 3 ops       : d_xx, d_yy, d_zz of the stage Phi
  double *a, *b;        // interior              : Laplacians kept between stages, see k_rk_combine
  const long long *extpre, *intpre;
  const int *blocks;
  int N, g;
  double c[4];          // 1, and the stage's factors
};

// ERK4 for Phi_t = K, K_t = l(Phi): every stage Phi is Phi + c dt K plus one earlier Laplacian, so the
// stage K and the accumulators of Phi need not be kept.  With l_s the Laplacian of stage s:
//   1: phis = Phi + dt/2 K                        a = l_1
//   2: phis = Phi + dt/2 K + dt^2/4 l_1           b = l_2
//   3: phis = Phi + dt K + dt^2/2 l_2             a = l_1 + l_2 + l_3,  b = a + (l_2 + l_3)
//   4: Phi += dt K + dt^2/6 a                     K += dt/6 (b + l_4)
// 34 values moved and 20 FP64 operations per point and step (43 and 34 with stage K and two
// accumulators); 256^3: 1.24 -> 0.70 ms per step.
// NC: the block size as a compile-time constant (0: taken from A.N at run time).
template <int NC, int V, int STAGE>
__global__ void __launch_bounds__(256) k_rk_combine(const StageArgs A) {
  __shared__ double sc[4];
  stage_constants(sc, A.c);
  const int N = NC ? NC : A.N, E = N + 2 * A.g;
  const int n3 = N * N * N;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  if (i >= n3) return;
  const int blk = A.blocks[blockIdx.y];
  const int x = i % N, y = (i / N) % N, z = i / (N * N);
  const long long e = A.extpre[blk] + ((z + A.g) * E + (y + A.g)) * E + (x + A.g);
  const long long in = A.intpre[blk] + i;
  const double *L = A.lap + 3 * A.intpre[blk] + i;
  const double one = sc[0], c1 = sc[1], c2 = sc[2], c3 = sc[3];
  const Pack<V> lx = ld<V>(L), ly = ld<V>(L + n3), lz = ld<V>(L + 2 * n3), p = ld<V>(A.phi + e), k = ld<V>(A.K + e);
  Pack<V> a, b;
  if constexpr (STAGE > 1) a = ld<V>(A.a + in);
  if constexpr (STAGE > 2) b = ld<V>(A.b + in);
  Pack<V> po, ko, ao, bo;
#pragma unroll
  for (int u = 0; u < V; ++u) {
    const double lap = fma(fma(lx.v[u], one, ly.v[u]), one, lz.v[u]);
    po.v[u] = fma(c1, k.v[u], p.v[u]);
    if constexpr (STAGE == 1) {
      ao.v[u] = lap;
    } else if constexpr (STAGE == 2) {
      po.v[u] = fma(c2, a.v[u], po.v[u]);
      bo.v[u] = lap;
    } else if constexpr (STAGE == 3) {
      po.v[u] = fma(c2, b.v[u], po.v[u]);
      const double t = fma(b.v[u], one, lap);
      ao.v[u] = fma(a.v[u], one, t);
      bo.v[u] = fma(ao.v[u], one, t);
    } else {
      po.v[u] = fma(c2, a.v[u], po.v[u]);
      ko.v[u] = fma(c3, fma(b.v[u], one, lap), k.v[u]);
    }
  }
  if constexpr (STAGE < 4) {
    st<V>(A.phis + e, po);
    if constexpr (STAGE != 2) st<V>(A.a + in, ao);
    if constexpr (STAGE != 1) st<V>(A.b + in, bo);
  } else {
    st<V>(A.phi + e, po);
    st<V>(A.K + e, ko);
  }
}

// ---------------------------------------------------------------- 2S low-storage RK + KO dissipation

struct RhsArgs {
  const double *phi, *K;     // field layout, ghosts exchanged (K's only when ko_on)
  double *lap;               // interior, 3 ops: d_xx, d_yy, d_zz in; F_K, F_Phi out (slots 0, 1)
  const long long *extpre, *intpre;
  const int *blocks;
  const double *scale;       // [b][degree][axis x, y, z] = 1/dx^d
  int N, g, r, ko_on;
  double ko;                 // -((-1)^r / 2^{2r}) sigma
  double one;                // 1
  int c[13];                 // (D_+)^r (D_-)^r stencil (2r)E_r, m = -r..r
};

// Right-hand side of the wave system with Kreiss-Oliger terms (Eq. dissdef) at every
// interior point: F_K = (d_xx + d_yy) + d_zz + sum_i Q_i[K], F_Phi = K + sum_i Q_i[Phi].
// TK is the precision of the dissipation stencil sums.
template <int NC, typename TK>
__global__ void k_wave_rhs(const RhsArgs A) {
  const int N = NC ? NC : A.N, g = A.g, E = N + 2 * g;
  const int n3 = N * N * N;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n3) return;
  const int b = A.blocks[blockIdx.y];
  const int x = i % N, y = (i / N) % N, z = i / (N * N);
  const long long e = A.extpre[b] + ((z + g) * E + (y + g)) * E + (x + g);
  double *L = A.lap + 3 * A.intpre[b];
  double fk = __dadd_rn(__dadd_rn(L[i], L[n3 + i]), L[2 * n3 + i]);
  double fp = A.K[e];
  if (A.ko_on) {
    const long long stride[3] = {1, E, (long long)E * E};   // x, y, z
    for (int a = 0; a < 3; ++a) {
      const double w = __dmul_rn(A.ko, A.scale[(b * 2 + 0) * 3 + a]);
      TK sp = 0, sk = 0;
      for (int m = -A.r; m <= A.r; ++m) {
        const long long o = e + m * stride[a];
        sp += (TK)A.c[m + A.r] * (TK)A.phi[o];
        sk += (TK)A.c[m + A.r] * (TK)A.K[o];
      }
      fp = __dadd_rn(fp, __dmul_rn(w, (double)sp));
      fk = __dadd_rn(fk, __dmul_rn(w, (double)sk));
    }
  }
  L[i] = fk;
  L[n3 + i] = fp;
}

// The same right-hand side in FP64 for N in {16, 32} and r = RR, tiled: a CTA of N x TY threads owns TY rows of
// one block and marches along z.  The x and y stencil taps come from the current z plane staged in shared
// memory (with an RR-wide halo), the z taps from a queue of 2RR+1 values per thread in registers, so every
// field value is read from global memory about once per plane instead of 2r+1 times per direction.  The
// arithmetic and its order are those of k_wave_rhs (taps m = -r..r summed per axis, axes x, y, z added in that
// order).
template <int N, int RR>
__global__ void __launch_bounds__(256) k_wave_rhs_tiled(const RhsArgs A) {
  constexpr int TY = 256 / N, W = N + 2 * RR, H = TY + 2 * RR, Q = 2 * RR + 1;
  __shared__ double sp_[H][W], sk_[H][W];
  const int g = A.g, E = N + 2 * g;
  const long long E2 = (long long)E * E;
  const int tx = threadIdx.x, ty = threadIdx.y, t = ty * N + tx;
  const int y0 = blockIdx.x * TY;
  const int b = A.blocks[blockIdx.y];
  const int n3 = N * N * N;
  const double *phi = A.phi + A.extpre[b], *K = A.K + A.extpre[b];
  double *L = A.lap + 3 * A.intpre[b];
  const double wx = __dmul_rn(A.ko, A.scale[(b * 2 + 0) * 3 + 0]);
  const double wy = __dmul_rn(A.ko, A.scale[(b * 2 + 0) * 3 + 1]);
  const double wz = __dmul_rn(A.ko, A.scale[(b * 2 + 0) * 3 + 2]);
  double c[Q];
#pragma unroll
  for (int m = 0; m < Q; ++m) c[m] = (double)A.c[m];
  // this thread's column (x, y) in the ghost-extended block
  const long long col = (long long)(y0 + ty + g) * E + (tx + g);
  double qp[Q], qk[Q];
#pragma unroll
  for (int m = 0; m < Q - 1; ++m) {  // z = -RR .. RR-1 (ghost planes exist: RR <= g)
    qp[m + 1] = phi[(long long)(g + m - RR) * E2 + col];
    qk[m + 1] = K[(long long)(g + m - RR) * E2 + col];
  }
  for (int z = 0; z < N; ++z) {
    // shift the z queue and load plane z + RR
#pragma unroll
    for (int m = 0; m < Q - 1; ++m) { qp[m] = qp[m + 1]; qk[m] = qk[m + 1]; }
    qp[Q - 1] = phi[(long long)(g + z + RR) * E2 + col];
    qk[Q - 1] = K[(long long)(g + z + RR) * E2 + col];
    __syncthreads();  // the previous plane's taps are read
    const long long plane = (long long)(g + z) * E2;
    for (int i = t; i < H * W; i += 256) {
      const int r = i / W, xx = i - r * W;
      const long long o = plane + (long long)(y0 + r - RR + g) * E + (xx - RR + g);
      sp_[r][xx] = phi[o];
      sk_[r][xx] = K[o];
    }
    __syncthreads();
    const int i = (z * N + (y0 + ty)) * N + tx;
    double fk = __dadd_rn(__dadd_rn(L[i], L[n3 + i]), L[2 * n3 + i]);
    double fp = K[plane + col];
    double px = 0, kx = 0, py = 0, ky = 0, pz = 0, kz = 0;
#pragma unroll
    for (int m = 0; m < Q; ++m) {
      px += c[m] * sp_[ty + RR][tx + m];
      kx += c[m] * sk_[ty + RR][tx + m];
      py += c[m] * sp_[ty + m][tx + RR];
      ky += c[m] * sk_[ty + m][tx + RR];
      pz += c[m] * qp[m];
      kz += c[m] * qk[m];
    }
    fp = __dadd_rn(fp, __dmul_rn(wx, px));
    fk = __dadd_rn(fk, __dmul_rn(wx, kx));
    fp = __dadd_rn(fp, __dmul_rn(wy, py));
    fk = __dadd_rn(fk, __dmul_rn(wy, ky));
    fp = __dadd_rn(fp, __dmul_rn(wz, pz));
    fk = __dadd_rn(fk, __dmul_rn(wz, kz));
    L[i] = fk;
    L[n3 + i] = fp;
  }
}

// A double as a float, rounded to nearest, with integer instructions (a conversion holds the FP64 pipe for
// 64 cycles per warp, these ten take ~20 of the integer pipe): the exponent rebias flips one bit, the
// rounding bit is added with its carry (ties up).  Values outside the normal floats take the conversion.
__device__ __forceinline__ float to_float(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v), a = hi & 0x7FFFFFFFu;
  if (a - 0x38100000u < 0x47E00000u - 0x38100000u)
    return __uint_as_float((((__funnelshift_l(lo, hi, 3) & 0x7FFFFFFFu) ^ 0x40000000u) + ((lo >> 28) & 1u)) |
                           (hi & 0x80000000u));
  return a == 0 ? 0.0f : (float)v;
}
// A float as a double, exactly, with integer instructions: subnormals are scaled up by 2^32 first.  (With a
// conversion for them the compiler executes it always, and the step without shift at 128^3 took 629 us, not 600.)
__device__ __forceinline__ double to_double(float f) {
  const bool small = (__float_as_uint(f) & 0x7F800000u) == 0;
  const unsigned u = __float_as_uint(small ? f * 0x1p32f : f), e = (u >> 23) & 0xFFu;
  if (e == 0xFFu) return (double)f;
  return e == 0 ? 0.0
                : __hiloint2double((int)((u & 0x80000000u) | ((e + (small ? 864u : 896u)) << 20) | ((u >> 3) & 0xFFFFFu)),
                                   (int)(u << 29));
}

// The right-hand side with FP32 stencil sums for N in {16, 32} and r = 4, the tensor-core steps' form.  A
// CTA of N x 16 threads marches along z through the planes of its 16 rows.  Each plane (with its 4-wide
// halo) is converted to FP32 once, when it enters a ring of planes four steps ahead; the z taps come from a
// register queue fed by the ring.  What bounds it: the FP64 pipe had 13 operations per point (seven of them
// conversions), 0.52 ms a stage at 256^3; with four it is memory latency: 0.43 ms with five planes in the
// ring, two barriers per plane and the Laplacian's loads behind the first; 0.37 with a sixth plane, so that
// the slot written is none of those that warps behind the single barrier still read, and those loads ahead
// of it.  (Two points per thread, 24 warps per SM instead of 32: 0.52.)
template <int N>
__global__ void __launch_bounds__(N * 16) k_wave_rhs_ring(const RhsArgs A) {
  constexpr int RR = 4, TY = 16, NT = N * TY, W = N + 2 * RR, H = TY + 2 * RR, Q = 2 * RR + 1, HW = H * W, SLOTS = RR + 2;
  constexpr int PER = (HW + NT - 1) / NT;  // values of a plane and field per thread
  __shared__ float ring[SLOTS][2][HW];
  __shared__ double s_one;
  const int g = A.g, E = N + 2 * g;
  const long long E2 = (long long)E * E;
  const int t = threadIdx.x, tx = t % N, ty = t / N;
  const int y0 = blockIdx.x * TY;
  const int b = A.blocks[blockIdx.y];
  const int n3 = N * N * N;
  const double *f[2] = {A.phi + A.extpre[b], A.K + A.extpre[b]};
  double *L = A.lap + 3 * A.intpre[b];
  if (t == 0) s_one = A.one;
  const double *sc = A.scale + (b * 2 + 0) * 3;
  const float wx = (float)(A.ko * sc[0]), wy = (float)(A.ko * sc[1]), wz = (float)(A.ko * sc[2]);
  float c[Q];
#pragma unroll
  for (int m = 0; m < Q; ++m) c[m] = (float)A.c[m];
  int off[PER];            // this thread's places in a plane
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int i = min(t + u * NT, HW - 1), r = i / W, xx = i - r * W;
    off[u] = (y0 + r - RR + g) * E + (xx - RR + g);
  }
  double raw[2][PER];
  auto fetch = [&](int z) {  // z in -4 .. N + 3
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int u = 0; u < PER; ++u) raw[q][u] = __ldg(f[q] + (long long)(z + g) * E2 + off[u]);
  };
  auto put = [&](int slot) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int u = 0; u < PER; ++u)
        if (t + u * NT < HW) ring[slot][q][t + u * NT] = to_float(raw[q][u]);
  };
  const int own = (ty + RR) * W + tx + RR;
  const long long col = (long long)(y0 + ty + g) * E + (tx + g);
  float qz[2][Q];
  for (int z = 0; z < RR; ++z) {
    fetch(z);
    put(z);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int m = 0; m < RR; ++m) qz[q][m + 1] = to_float(__ldg(f[q] + (long long)(g + m - RR) * E2 + col));
  __syncthreads();
  const double one = s_one;
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int m = 0; m < RR; ++m) qz[q][RR + 1 + m] = ring[m][q][own];
  fetch(RR);
  int cur = 0, in = RR;      // ring slots of plane z and of plane z + 4
  for (int z = 0; z < N; ++z) {
    const int i = (z * N + (y0 + ty)) * N + tx;
    const double l0 = L[i], l1 = L[n3 + i], l2 = L[2 * n3 + i], kk = __ldg(f[1] + (long long)(g + z) * E2 + col);
    put(in);
    __syncthreads();
    if (z + 1 < N) fetch(z + 1 + RR);
    float sum[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
      for (int m = 0; m < Q - 1; ++m) qz[q][m] = qz[q][m + 1];
      qz[q][Q - 1] = ring[in][q][own];
      const float *pl = ring[cur][q] + own;
      float px = 0, py = 0, pz = 0;
#pragma unroll
      for (int m = 0; m < Q; ++m) {
        px += c[m] * pl[m - RR];
        py += c[m] * pl[(m - RR) * W];
        pz += c[m] * qz[q][m];
      }
      sum[q] = wx * px + wy * py + wz * pz;
    }
    L[i] = fma(fma(fma(l0, one, l1), one, l2), one, to_double(sum[1]));
    L[n3 + i] = fma(kk, one, to_double(sum[0]));
    cur = cur == SLOTS - 1 ? 0 : cur + 1;
    in = in == SLOTS - 1 ? 0 : in + 1;
  }
}

struct UpdArgs {
  double *phi, *K;           // field layout: S1, updated in place (interior)
  double *s2p, *s2k;         // interior: S2
  const double *lap;         // F_K, F_Phi (slots 0, 1)
  const double *adv_p, *adv_k, *beta;  // shift terms: the selected derivatives of Phi and K, [block][3][N^3], and the shift
  const long long *extpre, *intpre;
  const int *blocks;
  int N, g, first;
  double c[5];               // 1, gamma1, gamma2, beta dt, delta
};

// S2 <- S2 + delta S1;  S1 <- gamma1 S1 + gamma2 S2 + (beta dt) F, per field; ADV: F gets the upwinded shift
// terms beta^i d_i here (blending them into F first moved 18 more values per point and step stage;
// 256^3: 0.45 + 2 x 0.28 -> 0.43 ms).
template <int NC, int V, bool ADV>
__global__ void __launch_bounds__(256) k_lsrk_update(const UpdArgs A) {
  __shared__ double sc[5];
  stage_constants(sc, A.c);
  const int N = NC ? NC : A.N, g = A.g, E = N + 2 * g;
  const int n3 = N * N * N;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  if (i >= n3) return;
  const int b = A.blocks[blockIdx.y];
  const int x = i % N, y = (i / N) % N, z = i / (N * N);
  const long long ofs = ((z + g) * E + (y + g)) * E + (x + g), e = A.extpre[b] + ofs;
  const long long in = A.intpre[b] + i;
  const double *L = A.lap + 3 * A.intpre[b] + i;
  const double g1 = sc[1], g2 = sc[2], bdt = sc[3], de = sc[4];
  Pack<V> S[2] = {ld<V>(A.phi + e), ld<V>(A.K + e)}, F[2] = {ld<V>(L + n3), ld<V>(L)}, T[2], dv[2][3], bv[3];
  if (!A.first) {
    T[0] = ld<V>(A.s2p + in);
    T[1] = ld<V>(A.s2k + in);
  }
  if constexpr (ADV) {
    const long long E3 = (long long)E * E * E;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      bv[c] = ld<V>(A.beta + 3 * A.extpre[b] + c * E3 + ofs);
      dv[0][c] = ld<V>(A.adv_p + 3 * A.intpre[b] + i + c * n3);
      dv[1][c] = ld<V>(A.adv_k + 3 * A.intpre[b] + i + c * n3);
    }
  }
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int u = 0; u < V; ++u) {
      double f = F[q].v[u];
      if constexpr (ADV) {
#pragma unroll
        for (int c = 0; c < 3; ++c) f = fma(bv[c].v[u], dv[q][c].v[u], f);
      }
      const double s = S[q].v[u], s2 = A.first ? de * s : fma(de, s, T[q].v[u]);
      T[q].v[u] = s2;
      S[q].v[u] = fma(g1, s, fma(g2, s2, bdt * f));
    }
  st<V>(A.s2p + in, T[0]);
  st<V>(A.s2k + in, T[1]);
  st<V>(A.phi + e, S[0]);
  st<V>(A.K + e, S[1]);
}

// go(block size as a constant or 0, vector width 2 or 1)
template <typename F>
void by_size(int N, bool vec, F go) {
  using std::integral_constant;
  auto by_v = [&](auto nc) {
    if (vec) go(nc, integral_constant<int, 2>());
    else go(nc, integral_constant<int, 1>());
  };
  if (N == 32) by_v(integral_constant<int, 32>());
  else if (N == 16) by_v(integral_constant<int, 16>());
  else by_v(integral_constant<int, 0>());
}

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

struct WaveLayout {
  size_t ext = 0, in = 0, apply = 0;
  size_t total() const { return al(ext * 8) + al(in * 8) * 2 + al(3 * in * 8) + apply + 256; }
};

cfd_status wave_layout(cfd_blocks_s *B, cfd_precision prec, int n_iter, WaveLayout &L) {
  for (int b = 0; b < B->nblocks; ++b) {
    const size_t N = B->n[b], E = N + 2 * B->ng;
    L.ext += E * E * E;
    L.in += N * N * N;
  }
  return cfd_apply_workspace(B, 1, CFD_OP_DXX | CFD_OP_DYY | CFD_OP_DZZ, prec, n_iter, &L.apply);
}

}  // namespace
}  // namespace cfd

using namespace cfd;

extern "C" cfd_status cfd_wave_workspace(cfd_blocks_t B, cfd_precision prec, int n_iter, size_t *bytes) {
  if (!B || !bytes) { set_error("cfd_wave_workspace: bad argument"); return CFD_ERR_ARG; }
  WaveLayout L;
  cfd_status s = wave_layout(B, prec, n_iter, L);
  if (s != CFD_OK) return s;
  *bytes = L.total();
  return CFD_OK;
}

extern "C" cfd_status cfd_wave_rk_step(cfd_blocks_t B, void *phi, void *K, double dt, cfd_precision prec, int n_iter,
                                       void *work, size_t work_bytes, void *stream) {
  if (!B || !phi || !K || !work) { set_error("cfd_wave_rk_step: bad argument"); return CFD_ERR_ARG; }
  if (B->dtype != CFD_F64) { set_error("cfd_wave_rk_step: FP64 fields only"); return CFD_ERR_UNSUPPORTED; }
  if (!B->s[1].present) { set_error("cfd_wave_rk_step: needs the second-degree scheme"); return CFD_ERR_ARG; }
  for (int v : B->nbr)
    if (v < 0) { set_error("cfd_wave_rk_step: every ghost region needs a neighbour"); return CFD_ERR_UNSUPPORTED; }
  WaveLayout L;
  cfd_status s = wave_layout(B, prec, n_iter, L);
  if (s != CFD_OK) return s;
  if (work_bytes < L.total()) { set_error("cfd_wave_rk_step: workspace too small"); return CFD_ERR_ARG; }
  cudaStream_t st = (cudaStream_t)stream;
  char *base = (char *)(((uintptr_t)work + 255) & ~(uintptr_t)255);
  double *phis = (double *)base;  base += al(L.ext * 8);
  double *la = (double *)base;    base += al(L.in * 8);
  double *lb = (double *)base;    base += al(L.in * 8);
  double *lap = (double *)base;   base += al(3 * L.in * 8);
  void *aw = base;
  const unsigned ops = CFD_OP_DXX | CFD_OP_DYY | CFD_OP_DZZ;
  const double cs[4][4] = {{1, 0.5 * dt, 0, 0}, {1, 0.5 * dt, 0.25 * dt * dt, 0}, {1, dt, 0.5 * dt * dt, 0},
                           {1, dt, dt * dt / 6.0, dt / 6.0}};
  const bool vec = B->ng % 2 == 0 && !(((uintptr_t)phi | (uintptr_t)K) & 15);
  for (int stage = 1; stage <= 4; ++stage) {
    double *src = stage == 1 ? (double *)phi : phis;
    if ((s = cfd_exchange_ghosts(B, src, 1, stream)) != CFD_OK) return s;
    if ((s = cfd_apply(B, src, 1, ops, prec, n_iter, lap, aw, L.apply, stream)) != CFD_OK) return s;
    for (size_t gi = 0; gi < B->sizes.size(); ++gi) {
      StageArgs A;
      A.phi = (double *)phi;
      A.K = (double *)K;
      A.phis = phis;
      A.lap = lap;
      A.a = la;
      A.b = lb;
      A.extpre = B->d_extpre;
      A.intpre = B->d_intpre;
      A.blocks = B->d_groups[gi];
      A.N = B->sizes[gi];
      A.g = B->ng;
      memcpy(A.c, cs[stage - 1], sizeof(A.c));
      auto go = [&](auto nc, auto vc) {
        constexpr int NC = decltype(nc)::value, V = decltype(vc)::value;
        const int n3 = A.N * A.N * A.N;
        const dim3 grid((unsigned)((n3 / V + 255) / 256), (unsigned)B->groups[gi].size());
        if (stage == 1) k_rk_combine<NC, V, 1><<<grid, 256, 0, st>>>(A);
        else if (stage == 2) k_rk_combine<NC, V, 2><<<grid, 256, 0, st>>>(A);
        else if (stage == 3) k_rk_combine<NC, V, 3><<<grid, 256, 0, st>>>(A);
        else k_rk_combine<NC, V, 4><<<grid, 256, 0, st>>>(A);
      };
      launch_begin(KF_RK, st);
      by_size(A.N, vec, go);
      launch_end(KF_RK, st);
      if ((s = cuda_fail(cudaGetLastError(), "k_rk_combine launch")) != CFD_OK) return s;
    }
  }
  return CFD_OK;
}

extern "C" cfd_status cfd_wave_lsrk_workspace(cfd_blocks_t B, cfd_precision prec, int n_iter, size_t *bytes) {
  if (!B || !bytes) { set_error("cfd_wave_lsrk_workspace: bad argument"); return CFD_ERR_ARG; }
  WaveLayout L;
  cfd_status s = wave_layout(B, prec, n_iter, L);
  if (s != CFD_OK) return s;
  *bytes = al(L.in * 8) * 2 + al(3 * L.in * 8) + al(L.apply) + 256;
  return CFD_OK;
}

namespace cfd {
namespace {

// One 2S step of the wave system with Kreiss-Oliger terms; with `beta` the shifted system of
// Eq. toyShiftWaveEqnSys (flat gamma): the upwinded advective terms beta^i d_i Phi and
// beta^i d_i K are added to F_Phi and F_K.
cfd_status lsrk_impl(const char *who, cfd_blocks_s *B, void *phi, void *K, const void *beta, double dt,
                     const cfd_lsrk_desc *rk, double sigma, int ko_r, cfd_precision prec, int n_iter, void *work,
                     size_t work_bytes, cudaStream_t st) {
  auto fail = [&](cfd_status code, const char *msg) {
    set_error(std::string(who) + ": " + msg);
    return code;
  };
  if (!B || !phi || !K || !work || !rk) return fail(CFD_ERR_ARG, "bad argument");
  if (rk->stages < 1 || rk->stages > 8 || !rk->gamma1 || !rk->gamma2 || !rk->beta || !rk->delta)
    return fail(CFD_ERR_ARG, "1..8 stages with all four coefficient arrays");
  if (!(sigma >= 0) || (sigma > 0 && (ko_r < 1 || ko_r > B->ng || ko_r > 6)))
    return fail(CFD_ERR_ARG, "sigma >= 0 and 1 <= ko_r <= min(ng, 6)");
  if (B->dtype != CFD_F64) return fail(CFD_ERR_UNSUPPORTED, "FP64 fields only");
  if (!B->s[1].present) return fail(CFD_ERR_ARG, "needs the second-degree scheme");
  if (beta && !B->biased.present) return fail(CFD_ERR_ARG, "the shift terms need a biased scheme (cfd_scheme_set_biased)");
  for (int v : B->nbr)
    if (v < 0) return fail(CFD_ERR_UNSUPPORTED, "every ghost region needs a neighbour");
  WaveLayout L;
  cfd_status s = wave_layout(B, prec, n_iter, L);
  if (s != CFD_OK) return s;
  size_t bws = 0;
  if (beta && (s = cfd_biased_workspace(B, 1, prec, n_iter, &bws)) != CFD_OK) return s;
  const size_t need = al(L.in * 8) * 2 + al(3 * L.in * 8) + al(L.apply) + bws + 256;
  if (work_bytes < need) return fail(CFD_ERR_ARG, "workspace too small");
  char *base = (char *)(((uintptr_t)work + 255) & ~(uintptr_t)255);
  double *s2p = (double *)base;  base += al(L.in * 8);
  double *s2k = (double *)base;  base += al(L.in * 8);
  double *lap = (double *)base;  base += al(3 * L.in * 8);
  void *aw = base;               base += al(L.apply);
  void *bw = bws ? (void *)base : nullptr;
  const unsigned ops = CFD_OP_DXX | CFD_OP_DYY | CFD_OP_DZZ;
  const bool ko_on = sigma > 0;
  RhsArgs R;
  memset(&R, 0, sizeof(R));
  R.phi = (const double *)phi;
  R.K = (const double *)K;
  R.lap = lap;
  R.extpre = B->d_extpre;
  R.intpre = B->d_intpre;
  R.scale = B->d_scale;
  R.g = B->ng;
  R.ko_on = ko_on ? 1 : 0;
  R.one = 1.0;
  if (ko_on) {
    // (D_+)^r (D_-)^r: (-1)^(r+m) C(2r, r+m); prefactor -((-1)^r / 2^{2r}) sigma
    const int r = ko_r;
    R.r = r;
    long long binom = 1;
    for (int j = 0; j <= 2 * r; ++j) {
      R.c[j] = (int)((j % 2 == 0 ? 1 : -1) * binom);  // m = j - r: (-1)^(r+m) C(2r, r+m) = (-1)^j C(2r, j)
      binom = binom * (2 * r - j) / (j + 1);
    }
    R.ko = -((r % 2 == 0) ? 1.0 : -1.0) / (double)(1ll << (2 * r)) * sigma;
  }
  const bool vec = B->ng % 2 == 0 && !(((uintptr_t)phi | (uintptr_t)K | (uintptr_t)beta) & 15);
  // Exact tensor-core shift terms: both fields' selected derivatives fill the six slots of the advection's
  // workspace and the update blends them; the signs of the shift, constant during the step, are made once.
  uint32_t *signs = beta && prec == CFD_TC_BF16_EXACT ? dense_sign_space(B, bw, n_iter) : nullptr;
  const bool fused = signs != nullptr;
  double *tmp = fused ? (double *)(((uintptr_t)bw + 255) & ~(uintptr_t)255) : nullptr;
  if (fused && (s = advect_check(B, 1, prec, n_iter, bw, bws)) != CFD_OK) return s;
  if (fused && (s = upwind_signs(B, beta, signs, st)) != CFD_OK) return s;
  auto launch1 = [&](auto nc, const RhsArgs &A, dim3 grid) {
    if (prec == CFD_FP64_BANDED) k_wave_rhs<decltype(nc)::value, double><<<grid, 256, 0, st>>>(A);
    else k_wave_rhs<decltype(nc)::value, float><<<grid, 256, 0, st>>>(A);
  };
  for (int stage = 0; stage < rk->stages; ++stage) {
    if ((s = cfd_exchange_ghosts(B, phi, 1, st)) != CFD_OK) return s;
    if ((ko_on || beta) && (s = cfd_exchange_ghosts(B, K, 1, st)) != CFD_OK) return s;
    if ((s = cfd_apply(B, phi, 1, ops, prec, n_iter, lap, aw, L.apply, st)) != CFD_OK) return s;
    for (size_t gi = 0; gi < B->sizes.size(); ++gi) {
      const int N = B->sizes[gi];
      const long long n3 = (long long)N * N * N;
      dim3 grid((unsigned)((n3 + 255) / 256), (unsigned)B->groups[gi].size());
      RhsArgs A = R;
      A.blocks = B->d_groups[gi];
      A.N = N;
      launch_begin(KF_RK, st);
      if (ko_on && ko_r == 4 && (N == 32 || N == 16)) {
        const dim3 tg((unsigned)(N / (256 / N)), (unsigned)B->groups[gi].size());
        const dim3 tb((unsigned)N, (unsigned)(256 / N)), rg((unsigned)(N / 16), (unsigned)B->groups[gi].size());
        if (prec != CFD_FP64_BANDED) {
          if (N == 32) k_wave_rhs_ring<32><<<rg, 512, 0, st>>>(A);
          else k_wave_rhs_ring<16><<<rg, 256, 0, st>>>(A);
        } else if (N == 32) {
          k_wave_rhs_tiled<32, 4><<<tg, tb, 0, st>>>(A);
        } else {
          k_wave_rhs_tiled<16, 4><<<tg, tb, 0, st>>>(A);
        }
      } else if (N == 32) launch1(std::integral_constant<int, 32>(), A, grid);
      else if (N == 16) launch1(std::integral_constant<int, 16>(), A, grid);
      else launch1(std::integral_constant<int, 0>(), A, grid);
      launch_end(KF_RK, st);
      if ((s = cuda_fail(cudaGetLastError(), "k_wave_rhs launch")) != CFD_OK) return s;
    }
    if (beta && fused) {
      // the upwinded derivatives of Phi and K, blended by the update below
      const int axes[3] = {2, 1, 0};
      if ((s = dense_biased(B, phi, 1, beta, axes, 3, 2, prec, n_iter, nullptr, 1, 0, false, bw, bws, st, signs, tmp)) != CFD_OK)
        return s;
      if ((s = dense_biased(B, K, 1, beta, axes, 3, 2, prec, n_iter, nullptr, 1, 0, false, bw, bws, st, signs,
                            tmp + 3 * L.in)) != CFD_OK)
        return s;
    } else if (beta) {
      // F_Phi (slot 1) += beta . grad Phi, F_K (slot 0) += beta . grad K, upwinded
      if ((s = advect_accumulate(B, phi, 1, beta, lap, 3, 1, prec, n_iter, bw, bws, st)) != CFD_OK) return s;
      if ((s = advect_accumulate(B, K, 1, beta, lap, 3, 0, prec, n_iter, bw, bws, st)) != CFD_OK) return s;
    }
    for (size_t gi = 0; gi < B->sizes.size(); ++gi) {
      UpdArgs U;
      memset(&U, 0, sizeof(U));
      U.phi = (double *)phi;
      U.K = (double *)K;
      U.s2p = s2p;
      U.s2k = s2k;
      U.lap = lap;
      U.adv_p = tmp;
      U.adv_k = tmp ? tmp + 3 * L.in : nullptr;
      U.beta = (const double *)beta;
      U.extpre = B->d_extpre;
      U.intpre = B->d_intpre;
      U.blocks = B->d_groups[gi];
      U.N = B->sizes[gi];
      U.g = B->ng;
      U.first = stage == 0;
      const double cs[5] = {1.0, rk->gamma1[stage], rk->gamma2[stage], rk->beta[stage] * dt, rk->delta[stage]};
      memcpy(U.c, cs, sizeof(U.c));
      auto go = [&](auto nc, auto vc) {
        constexpr int NC = decltype(nc)::value, V = decltype(vc)::value;
        const int n3 = U.N * U.N * U.N;
        const dim3 grid((unsigned)((n3 / V + 255) / 256), (unsigned)B->groups[gi].size());
        if (fused) k_lsrk_update<NC, V, true><<<grid, 256, 0, st>>>(U);
        else k_lsrk_update<NC, V, false><<<grid, 256, 0, st>>>(U);
      };
      launch_begin(KF_RK, st);
      by_size(U.N, vec, go);
      launch_end(KF_RK, st);
      if ((s = cuda_fail(cudaGetLastError(), "k_lsrk_update launch")) != CFD_OK) return s;
    }
  }
  return CFD_OK;
}

}  // namespace
}  // namespace cfd

extern "C" cfd_status cfd_wave_lsrk_step(cfd_blocks_t B, void *phi, void *K, double dt, const cfd_lsrk_desc *rk,
                                         double sigma, int ko_r, cfd_precision prec, int n_iter, void *work,
                                         size_t work_bytes, void *stream) {
  return lsrk_impl("cfd_wave_lsrk_step", B, phi, K, nullptr, dt, rk, sigma, ko_r, prec, n_iter, work, work_bytes,
                   (cudaStream_t)stream);
}

extern "C" cfd_status cfd_shifted_wave_workspace(cfd_blocks_t B, cfd_precision prec, int n_iter, size_t *bytes) {
  if (!B || !bytes) { set_error("cfd_shifted_wave_workspace: bad argument"); return CFD_ERR_ARG; }
  WaveLayout L;
  cfd_status s = wave_layout(B, prec, n_iter, L);
  if (s != CFD_OK) return s;
  size_t bws = 0;
  if ((s = cfd_biased_workspace(B, 1, prec, n_iter, &bws)) != CFD_OK) return s;
  *bytes = al(L.in * 8) * 2 + al(3 * L.in * 8) + al(L.apply) + bws + 256;
  return CFD_OK;
}

extern "C" cfd_status cfd_shifted_wave_lsrk_step(cfd_blocks_t B, void *phi, void *K, const void *beta, double dt,
                                                 const cfd_lsrk_desc *rk, double sigma, int ko_r, cfd_precision prec,
                                                 int n_iter, void *work, size_t work_bytes, void *stream) {
  if (!beta) { set_error("cfd_shifted_wave_lsrk_step: beta is null (use cfd_wave_lsrk_step)"); return CFD_ERR_ARG; }
  return lsrk_impl("cfd_shifted_wave_lsrk_step", B, phi, K, beta, dt, rk, sigma, ko_r, prec, n_iter, work,
                   work_bytes, (cudaStream_t)stream);
}
