// Ghost exchange between blocks (matrix G, Eq. example_G).
#include <type_traits>

#include "cfd_internal.h"

namespace cfd {

namespace {

__device__ __forceinline__ int dir_index(int dz, int dy, int dx) {
  int r = 9 * (dz + 1) + 3 * (dy + 1) + (dx + 1);
  return r > 13 ? r - 1 : r;
}

// ---------------------------------------------------------------- ghost exchange

template <typename T, int V> struct VecOf { using type = T; };
template <> struct VecOf<double, 2> { using type = double2; };
template <> struct VecOf<float, 4> { using type = float4; };

// One thread per kVPT groups of V consecutive ghost cells along x (V values = 16 bytes where
// the ghost width, N and the rows keep 16-byte alignment; V = 1 otherwise), enumerated without
// idle threads: part A covers the rows (fixed z, y) that lie in the ghost shell along y or z
// (all of x), part B the x ghosts of the N^2 interior rows.  Consecutive threads take
// consecutive x, so destination rows and source segments are contiguous.  The field offsets
// of the block and its 26 neighbours come from one table (one load each, independent of the
// data), and each thread issues its kVPT copies together, so the copies, not a chain of
// dependent table loads, set the pace.  The common (N, g) pairs are compiled with constant
// sizes (divisions become multiply-shifts); NC = 0 takes them at run time.
constexpr int kVPT = 4;

template <typename T, int NC, int GC, int V>
__global__ void __launch_bounds__(256) k_exchange(T *f, int nf, const int *__restrict__ blocks, int b0, int N_,
                                                  int g_, const long long *__restrict__ tab) {
  using VT = typename VecOf<T, V>::type;
  const int N = NC ? NC : N_, g = NC ? GC : g_;
  const int E = N + 2 * g, Ev = E / V, gv = g / V, Nv = N / V, G2v = 2 * gv;
  const int nA = (E * E - N * N) * Ev, nB = N * N * G2v;
  const int job = blockIdx.y;
  const int lb = job / nf, q = job - lb * nf;
  const int b = b0 >= 0 ? b0 + lb : blocks[lb];
  const long long *tb = tab + (long long)b * 27;
  const long long cells = (long long)E * E * E;
  T *base = f + nf * tb[26] + q * cells;
  int dst[kVPT], src[kVPT];
  long long nbo[kVPT];
#pragma unroll
  for (int u = 0; u < kVPT; ++u) {
    const int idx = (blockIdx.x * kVPT + u) * blockDim.x + threadIdx.x;
    nbo[u] = -1;
    dst[u] = src[u] = 0;
    if (idx >= nA + nB) continue;
    int x, y, z;
    if (idx < nA) {
      const int r = idx / Ev;
      x = (idx - r * Ev) * V;
      const int G2 = 2 * g;
      if (r < G2 * E) {              // z in the ghost shell: whole planes
        const int zz = r / E;
        y = r - zz * E;
        z = zz < g ? zz : zz + N;
      } else {                       // z interior, y in the ghost shell
        const int r2 = r - G2 * E, zz = r2 / G2, yy = r2 - zz * G2;
        z = g + zz;
        y = yy < g ? yy : yy + N;
      }
    } else {                         // interior row, x ghosts
      const int r = idx - nA, row = r / G2v, xx = r - row * G2v, zz = row / N;
      x = (xx < gv ? xx : xx + Nv) * V;
      y = g + row - zz * N;
      z = g + zz;
    }
    const int dx = x < g ? -1 : (x >= N + g ? 1 : 0);
    const int dy = y < g ? -1 : (y >= N + g ? 1 : 0);
    const int dz = z < g ? -1 : (z >= N + g ? 1 : 0);
    nbo[u] = __ldg(tb + dir_index(dz, dy, dx));
    dst[u] = (z * E + y) * E + x;
    src[u] = dst[u] - ((dz * E + dy) * E + dx) * N;
  }
  chain_next();
  chain_wait();
  VT v[kVPT];
#pragma unroll
  for (int u = 0; u < kVPT; ++u)
    if (nbo[u] >= 0) v[u] = *reinterpret_cast<const VT *>(f + nf * nbo[u] + q * cells + src[u]);
#pragma unroll
  for (int u = 0; u < kVPT; ++u)
    if (nbo[u] >= 0) *reinterpret_cast<VT *>(base + dst[u]) = v[u];
}

}  // namespace

cfd_status launch_exchange(cfd_blocks_s *B, void *fields, int nf, cudaStream_t st) {
  for (auto &grp : B->groups)
    if ((long long)grp.size() * nf > 65535) {  // (block, field) pairs of one size go in gridDim.y
      set_error("ghost exchange: blocks of one size x nfields exceeds 65535");
      return CFD_ERR_UNSUPPORTED;
    }
  for (size_t gi = 0; gi < B->sizes.size(); ++gi) {
    const int N = B->sizes[gi];
    const int nblk = (int)B->groups[gi].size();
    const long long E = N + 2 * B->ng;
    const long long ghosts = E * E * E - (long long)N * N * N;
    const int g = B->ng;
    launch_begin(KF_EXCHANGE, st);
    auto go = [&](auto tag, auto nc, auto gc, auto vc) {
      using T = decltype(tag);
      constexpr int V = decltype(vc)::value;
      dim3 grid((unsigned)((ghosts / V + 256 * kVPT - 1) / (256 * kVPT)), nblk * nf);
      // Chained where the grid is about one wave (8 CTAs on each SM), where launch latency counts: an
      // exchange and d_x of one 32^3 block 10.2 -> 8.4 us.  Larger ones lose by starting in the tail of the
      // launch before (256^3, 4 fields, exchange and nine ops: 2.14 ms chained, 2.03 not).
      const bool chained = (long long)grid.x * grid.y <= 8ll * (B->num_sms > 0 ? B->num_sms : 148);
      launch_chained(k_exchange<T, decltype(nc)::value, decltype(gc)::value, V>, grid, 256, 0, st, chained,
                     static_cast<T *>(fields), nf, B->d_groups[gi], B->group_b0[gi], N, g, B->d_exch);
    };
    auto by_size = [&](auto tag, auto vc) {
      using I = std::integral_constant<int, 0>;
      if (g == 4 && N == 16) go(tag, std::integral_constant<int, 16>(), std::integral_constant<int, 4>(), vc);
      else if (g == 4 && N == 32) go(tag, std::integral_constant<int, 32>(), std::integral_constant<int, 4>(), vc);
      else if (g == 4 && N == 8) go(tag, std::integral_constant<int, 8>(), std::integral_constant<int, 4>(), vc);
      else go(tag, I(), I(), vc);
    };
    // 16-byte copies need g, N (hence E) multiples of the vector width and an aligned buffer
    const bool al16 = ((uintptr_t)fields & 15) == 0;
    if (B->dtype == CFD_F64) {
      if (al16 && g % 2 == 0) by_size(double(), std::integral_constant<int, 2>());
      else by_size(double(), std::integral_constant<int, 1>());
    } else {
      if (al16 && g % 4 == 0 && N % 4 == 0) by_size(float(), std::integral_constant<int, 4>());
      else by_size(float(), std::integral_constant<int, 1>());
    }
    launch_end(KF_EXCHANGE, st);
    cfd_status s = cuda_fail(cudaGetLastError(), "k_exchange launch");
    if (s != CFD_OK) return s;
  }
  return CFD_OK;
}

}  // namespace cfd
