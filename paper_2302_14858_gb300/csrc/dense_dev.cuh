// Device helpers shared by the tensor-core kernels (dense_tc.cu, dense_exact.cuh): shared-memory
// descriptors, tcgen05.mma, mbarriers with bounded waits, cp.async, tile arithmetic.
#pragma once
#include "dense.h"

namespace cfd {
namespace {

constexpr int kTile = 128;         // pencils per tile (MMA M)
constexpr int kTmemCols = 512;
constexpr long long kWaitLimit = 4000000000LL;  // clock cycles (~2 s) before giving up
constexpr int kBadTau = 1 << 20;  // pencil scale of a pencil holding a NaN or an infinity

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// BF16 or FP16 operands (the instruction descriptor says which)
__device__ __forceinline__ void mma_16bit(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

// The commit's mbarrier is arrived on when every MMA this thread has issued so far has completed.
__device__ __forceinline__ void mma_commit(uint32_t mbar_addr) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar_addr));
}

__device__ __forceinline__ int biased_exp(double v) {
  return (int)((((unsigned long long)__double_as_longlong(v)) >> 52) & 0x7FF);
}
__device__ __forceinline__ int biased_exp(float v) { return (int)((__float_as_uint(v) >> 23) & 0xFF); }
__device__ __forceinline__ int tau_exp(int emax, double) { return emax - 1022; }
__device__ __forceinline__ int tau_exp(int emax, float) { return emax - 126; }
__device__ __forceinline__ int nonfinite_exp(double) { return 0x7FF; }
__device__ __forceinline__ int nonfinite_exp(float) { return 0xFF; }

// Wait for the phase `parity` of an mbarrier for at most `limit` clock cycles.  The main loops
// use the launch's limit (DenseParams::wait_limit); the exit path, which drains the CTA's own
// copies and MMAs before it frees TMEM, always uses kWaitLimit.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar_addr, uint32_t parity, long long limit = kWaitLimit) {
  const long long t0 = clock64();
  uint32_t done = 0;
  while (!done) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar_addr), "r"(parity)
        : "memory");
    if (!done && clock64() - t0 > limit) return false;
  }
  return true;
}
__device__ __forceinline__ void mbar_init(uint32_t addr, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t addr) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}

__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src));
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src));
}

__device__ __forceinline__ long long stride_of(int axis, long long s0, long long s1) {
  return axis == 0 ? s0 : (axis == 1 ? s1 : 1ll);
}

// Y * 2^E as an IEEE double (d = Y, |Y| < 2^55): the power-of-two scale is an add to the exponent
// field.  `checked`: results below the normal range flush to a signed zero, results above it
// become infinities, and `bad` gives a NaN; without it the caller has established that the
// exponent stays in range for every Y.
template <bool checked>
__device__ __forceinline__ double scaled_double(double d, int E, bool bad) {
  const int hi = __double2hiint(d), lo = __double2loint(d);
  if (!checked) return d == 0.0 ? 0.0 : __hiloint2double(hi + (E << 20), lo);
  const int fe = (hi >> 20) & 0x7FF;  // 0 only for d = 0 here (d is an integer or an FP32 value)
  if (bad) return __longlong_as_double(0x7FF8000000000000ll);
  if (fe == 0 || fe + E <= 0) return __hiloint2double(hi & (int)0x80000000, 0);
  if (fe + E >= 2047) return __hiloint2double((hi & (int)0x80000000) | 0x7FF00000, 0);
  return __hiloint2double(hi + (E << 20), lo);
}

// y * 2^E in FP32 for |E| <= 300: two exact power-of-two factors (each a normal float),
// so the only rounding is that of the final product (under- and overflow as IEEE).
__device__ __forceinline__ float scale_pow2(float y, int E) {
  E = max(-300, min(300, E));
  const int e1 = E / 2, e2 = E - e1;
  return y * __int_as_float((e1 + 127) << 23) * __int_as_float((e2 + 127) << 23);
}

struct TileCoord {
  int lb, q, b, t1, t2;
  bool valid;
};

// The tiles of this CTA: interleaved (tile = CTA + k * grid) or a contiguous run of
// tiles_per_cta (tile_order 1; neighbouring tiles share input rows in L2).
struct TileRange {
  int first, end, step;
};
__device__ __forceinline__ TileRange tile_range(const DenseParams &P) {
  TileRange r;
  if (P.tile_order) {
    r.first = blockIdx.x * P.tiles_per_cta;
    r.end = min(P.ntiles, r.first + P.tiles_per_cta);
    r.step = 1;
  } else {
    r.first = blockIdx.x;
    r.end = P.ntiles;
    r.step = gridDim.x;
  }
  return r;
}

__device__ __forceinline__ int dir_index_dev(int dz, int dy, int dx) {
  const int r = 9 * (dz + 1) + 3 * (dy + 1) + (dx + 1);
  return r > 13 ? r - 1 : r;
}

// n / d for 0 <= n < 2^22 with inv = 1/d rounded to FP32: (n + 1/2) / d stays at least 1/(2d)
// away from an integer, more than the two roundings can move it
__device__ __forceinline__ int fdiv(int n, float inv) { return __float2int_rz(((float)n + 0.5f) * inv); }

// pencil index p (within the block and field) of pencil `pencil` of a tile
__device__ __forceinline__ int tile_pencil(const DenseParams &P, int tile, int pencil) {
  const int job = fdiv(tile, P.inv_tpj), tj = tile - job * P.tiles_per_job;
  return tj * kTile + pencil;
}

__device__ __forceinline__ TileCoord tile_coord(const DenseParams &P, int tile, int pencil) {
  TileCoord c;
  const int job = fdiv(tile, P.inv_tpj), tj = tile - job * P.tiles_per_job;
  c.lb = fdiv(job, P.inv_nf);
  c.q = job - c.lb * P.nf;
  c.b = P.contig ? P.b0 + c.lb : P.blocks[c.lb];
  const int p = tj * kTile + pencil;
  c.valid = p < P.n1 * P.n2;
  c.t1 = c.valid ? fdiv(p, P.inv_n2) : 0;
  c.t2 = c.valid ? p - c.t1 * P.n2 : 0;
  return c;
}

}  // namespace
}  // namespace cfd
