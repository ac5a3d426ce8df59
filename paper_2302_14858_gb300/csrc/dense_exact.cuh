// The exact tensor-core form (CFD_TC_BF16_EXACT) of the dense block operators: FP16 digit slices.
//
// out[p, i] = sum_j f[p, j] D[i, j] for 128-pencil tiles, with FP64-level results from FP16 products.
// D row i is scaled by a power of two sigma_i and every pencil p by tau_p; both factors become 40-bit
// fixed point in four balanced base-1024 digits,
//     D_ij / sigma_i = sum_t b_t 2^{-9-10t},   f_pj / tau_p = sum_s a_s 2^{-9-10s},  |a_s|, |b_t| <= 512,
// each an integer that FP16 holds exactly.  A product of digits is below 2^18; the pairs of one level
// k = s + t accumulate in the same FP32 TMEM columns, and levels k <= 3 (10 pairs) are kept.  A level
// sum is bounded by 512 sum_j (|b_0| + .. + |b_k|), whatever the pencil: below 2^24 it is an exact integer.
// Over every row of the Q13, P12 and X_2 operators (closed, iterated, cyclic; N = 16 and 32; up to eight spacings) the
// largest bounds are 0.32, 0.65 and 0.92 of 2^24 for levels 1, 2 and 3; an operator whose digits are all near
// 512 may exceed it and then rounds in units of 2 of that level (2^-37 and 2^-47 for levels 2 and 3).  The
// dropped pairs (three of level 4) and the 2^-40 roundings leave ~4 x 2^-40 sigma_i tau_p rms per output over K = 40
// columns; five base-256 digits with levels 0-4, the form before, left 4.5 x 2^-40 with 15 pairs.
//
// Measured (256^3 as 512 blocks of 32^3, 4 FP64 fields, nine ops: six launches, event times): five
// BF16 digits with 15 pairs, 8 + 8 warps, one staging buffer 2.87 ms in all; this form with 8 epilogue
// warps 2.69; with 16 epilogue warps and TMA stores of the x outputs 2.03 (S_x 0.37, S_y 0.45, S_z 0.48,
// T_x 0.25, T_y 0.24 ms); direct outer stages, the operator's load behind the first tiles and a quarter of
// the outputs converted by integers 1.79 (S 0.36 to 0.37, T 0.24 to 0.25); x stages compiled for one staging
// and levels 0 and 3 made integers by an FP32 add 1.73 (S 0.34 to 0.35, T 0.23 to 0.24).  A producer's value
// costs ~20 instructions against ~45 before, an output ~14 against ~28.  What bounds it now: T stages DRAM; S
// stages DRAM (0.25 ms at the copy rate) and the FP64 pipe (48 conversions of 64 cycles per SM sub-partition
// and tile, 0.17 ms) beside the integer work, no one of them alone.
//
// Roles (28 warps, one persistent CTA per SM):
//   warps 0-7    producers: wait for a staged tile, split it into 4 digit rows of A[buf];
//   warps 8-23   epilogue: read the TMEM levels, rebuild and store the outputs, in units of 8 operator
//                rows x 32 pencils (four warps share a lane quadrant: a conversion to FP64 holds the
//                FP64 pipe for 64 cycles per warp, and four warps keep it fed through each other's
//                TMEM reads, integer work and stores);
//   warp 24      issues every tcgen05.mma;   warp 25  issues the TMA copies;   26, 27 idle.
// Registers: 72 per thread at launch (7 warpgroups, 504 in all per lane); the producers take 96, the
// epilogue keeps 72, the last warpgroup gives back all but 24 (2 x 96 + 4 x 72 + 24 = 504).
// A producer warp owns 16 pencils, two lanes each (lanes l and l + 16), so the pencil's largest
// exponent is one shuffle away and no barrier spans the producers: they meet the other roles only
// through mbarriers with one arrival per warp.  Staging is double buffered where it fits, so a tile's
// copy has a whole tile time to land.  Both operators of a stage (degrees 1 and 2) share one MMA
// chain (64 rows x 4 levels = 256 TMEM columns, two buffers).
#pragma once
#include <cuda_fp16.h>

#include "dense_dev.cuh"

namespace cfd {
namespace {

constexpr int kSl = 4;                   // digits per factor, and levels kept
constexpr int kXProdWarps = 8, kXEpiWarps = 16;
constexpr int kXProd = kXProdWarps * 32;
constexpr int kXThreads = kXProd + kXEpiWarps * 32 + 128;
constexpr int kXUnit = 8;                // operator rows of an epilogue unit
constexpr int kXRowBytes = 64;           // inner bytes of a staged box of x rows
constexpr int kXEtau = 8;                // pencil-scale ring (tiles)
constexpr int16_t kBadTau16 = 32767;     // kBadTau in the ring (scales are -1022 .. 1024)

// ---------------------------------------------------------------- digits

// 4 x (the 40-bit magnitude |v| / tau 2^39, rounded) + the digit offsets, as 64 bits: after the add
// the balanced digits sit at bits 2, 12, 22 (each + 512) and the top digit, as the FP16 pattern of
// 1024 + (d_0 + 512), in the high word.  C = emax + 12 (double) or emax (float); elements below
// 2^-41 tau shift out to zero, subnormal elements too (emax >= 64 here).
constexpr uint32_t kOffLo = 0x80000000u + 0x200000u + 0x800u + 2u, kOffHi = 0x6600u;

__device__ __forceinline__ uint64_t shr_clamped(uint64_t m, int sh) {  // sh >= 0; >= 64 gives 0
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(sh));
  return r;
}
__device__ __forceinline__ uint64_t fixed4(double v, int C) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | 0x100000u) << 32) | lo;
  return shr_clamped(m, C - (int)((hi >> 20) & 0x7FFu)) + (((uint64_t)kOffHi << 32) | kOffLo);
}
__device__ __forceinline__ uint64_t fixed4(float v, int C) {
  const uint32_t u = __float_as_uint(v);
  const uint64_t m = (uint64_t)((u & 0x7FFFFFu) | 0x800000u) << 17;
  return shr_clamped(m, C - (int)((u >> 23) & 0xFFu)) + (((uint64_t)kOffHi << 32) | kOffLo);
}
__device__ __forceinline__ uint32_t sign_word(double v) { return (uint32_t)__double2hiint(v); }
__device__ __forceinline__ uint32_t sign_word(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t abs_word(double v) { return (uint32_t)__double2hiint(v) & 0x7FFFFFFFu; }
__device__ __forceinline__ uint32_t abs_word(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }
constexpr int exp_shift(double) { return 20; }
constexpr int exp_shift(float) { return 23; }
__device__ __forceinline__ int split_base(int emax, double) { return emax + 12; }
__device__ __forceinline__ int split_base(int emax, float) { return emax; }

// Digits of two elements as FP16 pairs, most significant first.  A field becomes 1024 + (d + 512)
// by placing it in the mantissa of an FP16 1024; one HFMA2 removes 1536 and applies the signs.
__device__ __forceinline__ void digits_pair(uint64_t P, uint64_t Q, uint32_t sp, uint32_t sq, uint32_t (&w)[kSl]) {
  const uint32_t pl = (uint32_t)P, ph = (uint32_t)(P >> 32), ql = (uint32_t)Q, qh = (uint32_t)(Q >> 32);
  const uint32_t sg = __byte_perm(sp, sq, 0x7632) & 0x80008000u;
  const uint32_t one = sg | 0x3C003C00u, off = sg ^ 0xE600E600u;  // +-1, -+1536
  uint32_t f[kSl];
  f[0] = __byte_perm(ph, qh, 0x5410);
  f[1] = ((__byte_perm(pl, ql, 0x7632) >> 6) & 0x03FF03FFu) | 0x64006400u;
  f[2] = ((__byte_perm(pl, ql, 0x6521) >> 4) & 0x03FF03FFu) | 0x64006400u;
  f[3] = ((__byte_perm(pl, ql, 0x5410) >> 2) & 0x03FF03FFu) | 0x64006400u;
#pragma unroll
  for (int s = 0; s < kSl; ++s) asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(w[s]) : "r"(f[s]), "r"(one), "r"(off));
}

// M elements (2, 4 or 8) into the digit rows: dst is slice 0's address, slices `slice` bytes apart.
template <typename TI, int M>
__device__ __forceinline__ void split_store(const TI *v, int C, unsigned char *dst, int slice) {
  uint32_t w[kSl][M / 2];
#pragma unroll
  for (int k = 0; k < M; k += 2) {
    uint32_t d[kSl];
    digits_pair(fixed4(v[k], C), fixed4(v[k + 1], C), sign_word(v[k]), sign_word(v[k + 1]), d);
#pragma unroll
    for (int s = 0; s < kSl; ++s) w[s][k / 2] = d[s];
  }
#pragma unroll
  for (int s = 0; s < kSl; ++s) {
    if constexpr (M == 8) *reinterpret_cast<uint4 *>(dst + s * slice) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    else if constexpr (M == 4) *reinterpret_cast<uint2 *>(dst + s * slice) = make_uint2(w[s][0], w[s][1]);
    else *reinterpret_cast<uint32_t *>(dst + s * slice) = w[s][0];
  }
}

// A pencil whose largest exponent is below 64 (nearly all of it zeros or close to the bottom of the
// range): zeros and subnormals become exact zeros and the other exponents move up by 64.
__device__ __forceinline__ double lift64(double v) {
  const int hi = __double2hiint(v);
  return (hi & 0x7FF00000) ? __hiloint2double(hi + (64 << 20), __double2loint(v)) : 0.0;
}
__device__ __forceinline__ float lift64(float v) {
  const uint32_t u = __float_as_uint(v);
  return (u & 0x7F800000u) ? __uint_as_float(u + (64u << 23)) : 0.0f;
}

// ---------------------------------------------------------------- epilogue

__device__ __forceinline__ void load_levels(uint32_t (&acc)[kSl][8], uint32_t taddr, uint32_t lev) {
#pragma unroll
  for (int k = 0; k < kSl; ++k)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(acc[k][0]), "=r"(acc[k][1]), "=r"(acc[k][2]), "=r"(acc[k][3]), "=r"(acc[k][4]),
                   "=r"(acc[k][5]), "=r"(acc[k][6]), "=r"(acc[k][7])
                 : "r"(taddr + (uint32_t)k * lev));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// after the last group of a tile: one arrival per warp frees the TMEM buffer
__device__ __forceinline__ void release_levels(uint32_t t_empty) {
  if (!t_empty) return;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(t_empty);
}

// The levels of one output as a 64-bit integer in units of 2^-43 sigma tau, joined as integers: t1 = x0 2^10 + x1
// (|x0| < 2^21 - 2^14, see the row scale in exact_image) and t2 = x2 2^5 + round(x3 2^-5), |t2| < 2^31 - 2^28.
// The only rounding is the last level's, 2^-44 at most (the two low levels joined in FP32 rounded at 2^-24 of
// their sum).  x0 and x3 2^-5 are below 2^22: adding 1.5 2^23 leaves their integer in the mantissa, at the cost of
// an FP32 operation where a conversion takes eight.
template <int C>
__device__ __forceinline__ long long exact_y(const uint32_t (&acc)[kSl][C], int c) {
  constexpr float kBias = 12582912.0f;
  constexpr uint32_t kBiasBits = 0x4B400000u;
  const uint32_t x0 = __float_as_uint(__uint_as_float(acc[0][c]) + kBias);
  const uint32_t x3 = __float_as_uint(fmaf(__uint_as_float(acc[3][c]), 0.03125f, kBias));
  const int t1 = (int)(x0 * 1024u + (uint32_t)__float2int_rn(__uint_as_float(acc[1][c])) - kBiasBits * 1024u);
  const int t2 = (int)((uint32_t)__float2int_rn(__uint_as_float(acc[2][c])) * 32u + x3 - kBiasBits);
  return ((long long)t1 << 15) + (long long)t2;
}
constexpr int kYUnit = 43, kFUnit = 48;  // result exponents: 2^(rowexp + etau - unit)
// FP32 outputs: the levels in FP32, in units of 2^-48 sigma tau, the low ones first, so that only the last sum
// rounds near an output's last place (by Horner's rule from the top the errors against 64 bits were ~6 % larger)
template <int C>
__device__ __forceinline__ float exact_f(const uint32_t (&acc)[kSl][C], int c) {
  static_assert(kSl == 4, "four levels");
  float y = fmaf(__uint_as_float(acc[2][c]), 0x1p10f, __uint_as_float(acc[3][c]));
  y = fmaf(__uint_as_float(acc[1][c]), 0x1p20f, y);
  return fmaf(__uint_as_float(acc[0][c]), 0x1p30f, y);
}

// y 2^E for |y| < 2^53 and a result in the normal range (0 for y = 0): exact either way, by the FP64 pipe's
// conversion (64 cycles per warp) or by integer instructions (some 30 more than the other way's few).  The
// FP64 pipe is the busier: 0.23 of a 256^3 two-degree stage's 0.35 ms if it converted every output (0.17 with
// three in four).
template <bool INT>
__device__ __forceinline__ double scaled_y(long long y, int E) {
  if constexpr (INT) {
    const unsigned s = (unsigned)(y >> 32) & 0x80000000u;
    const unsigned long long a = y < 0 ? 0ull - (unsigned long long)y : (unsigned long long)y;
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
    const int n = (ah ? 0 : 32) + __clz(ah ? ah : al);   // leading zeros, 64 for y = 0
    const unsigned long long m = a << (n - 11);          // the leading one at bit 52
    const unsigned hi = ((unsigned)(m >> 32) + ((unsigned)(E + 1023 + 62 - n) << 20)) | s;
    return a ? __hiloint2double((int)hi, (int)(unsigned)m) : 0.0;
  } else {
    const double d = __ll2double_rn(y);
    const int hi = __double2hiint(d), lo = __double2loint(d);
    return __hiloint2double(hi ? hi + (E << 20) : 0, lo);
  }
}
// kIntOuts outputs of every group of four by integer instructions.  Nine ops at 256^3, 4 fields: none 2.08,
// one 2.03, two 2.05 ms; 64^3, 2 fields: 73.4, 68.9, 67.6 us; 22 FP32 fields on two levels: 2.89, 2.87, 2.91.
constexpr int kIntOuts = 1;
constexpr bool int_out(int u) { return u >= 4 - kIntOuts; }

// 8 rows of a pencil whose outputs all stay in the normal range.  FIN: final outputs, SC: the FP64
// intermediate (with the face neighbours' ghost copies where gx / gy are set).  ROW: the output axis is
// x, where a lane holds 8 consecutive values of its own row: written straight to memory every store
// instruction would touch 32 lines with 16 bytes each, so they go through `box` (this warp's
// [32 pencils][8] slot, swizzled as the output tensor map says) and one TMA store.
template <typename TO, bool ROW, bool FIN, bool SC>
__device__ __forceinline__ void rows_fast(uint32_t taddr, uint32_t lev, int etau, const int *rowexp, TO *fin,
                                          long long fin_stride, double *sc, long long sc_stride, long long gx,
                                          long long gy, uint32_t t_empty, unsigned char *box) {
  uint32_t acc[kSl][8];
  load_levels(acc, taddr, lev);
  release_levels(t_empty);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c0 = 0; c0 < 8; c0 += 4) {
    const int4 ra = *reinterpret_cast<const int4 *>(rowexp + c0);
    const int rx[4] = {ra.x, ra.y, ra.z, ra.w};
    TO o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = c0 + u;
      double dv = 0.0;
      if (sizeof(TO) == 8 || SC) {
        dv = int_out(u) ? scaled_y<true>(exact_y(acc, c), rx[u] + etau - kYUnit)
                        : scaled_y<false>(exact_y(acc, c), rx[u] + etau - kYUnit);
      }
      if constexpr (sizeof(TO) == 8) o[u] = dv;
      else o[u] = FIN ? exact_f(acc, c) * __int_as_float((rx[u] + etau - kFUnit + 127) << 23) : 0.f;
      if constexpr (SC) {
        double *s = sc + c * sc_stride;
        *s = dv;
        if (gx) s[gx] = dv;  // the face neighbours' ghost column and row
        if (gy) s[gy] = dv;
      }
      if constexpr (FIN && !ROW) fin[c * fin_stride] = o[u];
    }
    if constexpr (FIN && ROW) {
      if constexpr (sizeof(TO) == 8) {  // 64-byte rows: chunk ^ (row / 2) % 4
        const int sw = (lane >> 1) & 3;
        *reinterpret_cast<double2 *>(box + lane * 64 + (((c0 / 2) ^ sw) << 4)) = make_double2(o[0], o[1]);
        *reinterpret_cast<double2 *>(box + lane * 64 + (((c0 / 2 + 1) ^ sw) << 4)) = make_double2(o[2], o[3]);
      } else {                          // 32-byte rows: chunk ^ (row / 4) % 2
        *reinterpret_cast<float4 *>(box + lane * 32 + (((c0 / 4) ^ ((lane >> 2) & 1)) << 4)) =
            make_float4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// 8 rows of any pencil: per-thread outputs, non-finite pencils, exponents at the ends of the range.
template <typename TO>
__device__ __noinline__ void rows_any(uint32_t taddr, uint32_t lev, int etau, const int *rowexp, TO *fin,
                                      long long fin_stride, double *sc, long long sc_stride, long long gx,
                                      long long gy, bool wf, bool ws, uint32_t t_empty) {
  uint32_t acc[kSl][8];
  load_levels(acc, taddr, lev);
  release_levels(t_empty);
  const bool bad = etau == kBadTau;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int ex = rowexp[c] + etau;
    const double dv = (sizeof(TO) == 8 || ws) ? scaled_double<true>(__ll2double_rn(exact_y(acc, c)), ex - kYUnit, bad) : 0.0;
    if (wf) {
      if constexpr (sizeof(TO) == 8) fin[c * fin_stride] = dv;
      else fin[c * fin_stride] = bad ? __int_as_float(0x7FC00000) : scale_pow2(exact_f(acc, c), ex - kFUnit);
    }
    if (ws) {
      double *s = sc + c * sc_stride;
      *s = dv;
      if (gx) s[gx] = dv;
      if (gy) s[gy] = dv;
    }
  }
}

// 8 rows of an upwinded stage: of the two biased derivatives of a point only the one the shift selects
// (bit of `word`: the right-biased one, the second segment, `seg1` TMEM columns on) is rebuilt and stored.
// The choice is made on the accumulators, before the conversion to FP64: half the conversions and half
// the stores of writing both (256^3, 4 fields: a stage 0.36 -> 0.27 to 0.30 ms).  SAFE: as rows_fast.
template <typename TO, bool ROW, bool SAFE>
__device__ __forceinline__ void rows_upwind(uint32_t taddr, uint32_t lev, uint32_t seg1, int etau, const int *rowexp,
                                            int rstep, TO *fin, long long fin_stride, bool wf, uint32_t word,
                                            uint32_t t_empty, unsigned char *box) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int c0 = 0; c0 < 8; c0 += 4) {
    uint32_t a[kSl][4], b[kSl][4];
#pragma unroll
    for (int k = 0; k < kSl; ++k) {
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(a[k][0]), "=r"(a[k][1]), "=r"(a[k][2]), "=r"(a[k][3])
                   : "r"(taddr + (uint32_t)k * lev + (uint32_t)c0));
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(b[k][0]), "=r"(b[k][1]), "=r"(b[k][2]), "=r"(b[k][3])
                   : "r"(taddr + (uint32_t)k * lev + seg1 + (uint32_t)c0));
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (c0 == 4) release_levels(t_empty);
    const int4 r0 = *reinterpret_cast<const int4 *>(rowexp + c0), r1 = *reinterpret_cast<const int4 *>(rowexp + rstep + c0);
    const int x0[4] = {r0.x, r0.y, r0.z, r0.w}, x1[4] = {r1.x, r1.y, r1.z, r1.w};
    TO o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool right = (word >> (c0 + u)) & 1u;
#pragma unroll
      for (int k = 0; k < kSl; ++k) a[k][u] = right ? b[k][u] : a[k][u];
      const int ex = (right ? x1[u] : x0[u]) + etau;
      if constexpr (SAFE) {
        if constexpr (sizeof(TO) == 8) {
          o[u] = int_out(u) ? scaled_y<true>(exact_y(a, u), ex - kYUnit) : scaled_y<false>(exact_y(a, u), ex - kYUnit);
        } else {
          o[u] = exact_f(a, u) * __int_as_float((ex - kFUnit + 127) << 23);
        }
      } else {
        const bool bad = etau == kBadTau;
        if constexpr (sizeof(TO) == 8) o[u] = scaled_double<true>(__ll2double_rn(exact_y(a, u)), ex - kYUnit, bad);
        else o[u] = bad ? __int_as_float(0x7FC00000) : scale_pow2(exact_f(a, u), ex - kFUnit);
      }
      if constexpr (!ROW) {
        if (wf) fin[(c0 + u) * fin_stride] = o[u];
      }
    }
    if constexpr (ROW) {
      if constexpr (sizeof(TO) == 8) {
        const int sw = (lane >> 1) & 3;
        *reinterpret_cast<double2 *>(box + lane * 64 + (((c0 / 2) ^ sw) << 4)) = make_double2(o[0], o[1]);
        *reinterpret_cast<double2 *>(box + lane * 64 + (((c0 / 2 + 1) ^ sw) << 4)) = make_double2(o[2], o[3]);
      } else {
        *reinterpret_cast<float4 *>(box + lane * 32 + (((c0 / 4) ^ ((lane >> 2) & 1)) << 4)) =
            make_float4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// ---------------------------------------------------------------- the kernel

// N: block size (16, 32).  AXIS 0, 1, 2: pencils along z, y, x with ghost width 4 (every stride and
// the split of a pencil's columns are constants); AXIS 3: any axis and ghost width.  ITER: a pass of
// an iterated stage that takes the neighbours' previous iterate as four more columns per pencil.
// HALO: a halo pass of the hybrid iteration (Eq. iter_center_P): four operator rows (16 with their
// zero padding), whose outputs are the values the neighbours read at their k^c nodes.  It costs the
// producers' share of a stage, against ~11 FP32 operations per coefficient and row in compensated
// FP32 on the CUDA cores (256^3, 4 fields: see halo_pass in dense_tc.cu).
// UPWIND: the two biased operators of an axis, one output (rows_upwind).  (An instantiation of its own:
// as a branch of the plain epilogue it cost that one 4 %.)
// DIRECT: an outer stage of a mixed derivative that takes the inner one from its output slot, own points
// from the block's, ghost columns from the face neighbours' (g = 4, FP64; the columns are in the order
// [own | lower | upper], and so are the operator's).  No intermediate is written or read: at 256^3, 4
// fields, the y and z stages drop from 0.45 and 0.49 to 0.38 ms.
enum ExactMode { kPlain = 0, kHaloRows = 1, kUpwind = 2, kDirect = 3, kHaloDirect = 4 };
// STG: the staging of the input, 0: P.tma_kind decides, 1: TMA, 2: copies.  x stages have it compiled in: with both
// in one kernel the copy loop cost the TMA stages up to a tenth (T_x of 16^3 blocks, 22 FP32 fields: 0.172 against
// 0.150 ms), and without it they are 2 to 5 % faster than before it (256^3, one iteration: 3.12 -> 3.00 ms).
template <typename TI, typename TO, int N, int AXIS, bool ITER, int MODE, int STG>
__global__ void __launch_bounds__(kXThreads, 1) k_dense_exact(const __grid_constant__ DenseParams P) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr bool GEN = AXIS == 3, HALO = MODE == kHaloRows || MODE == kHaloDirect, UPWIND = MODE == kUpwind,
                 DIRECT = MODE == kDirect || MODE == kHaloDirect;
  static_assert(!DIRECT || (AXIS == 1 || AXIS == 2), "outer stages run along y and x");
  constexpr int KP = N == 32 ? 48 : 32, NCH = KP / 8;
  constexpr int ES = sizeof(TI);
  constexpr int SLICE = kTile * KP * 2, A_BYTES = kSl * SLICE;
  const int axis = GEN ? P.axis : AXIS;
  const int g = GEN ? P.g : 4;
  const int E = N + 2 * g;
  const int R = P.rows;
  constexpr int SR = HALO ? 16 : N;  // operator rows of a segment
  const int B_BYTES = kSl * R * KP * 2;
  // (direct stages have no other staging than TMA)
  const int kind = STG == 2 ? 0 : (DIRECT || STG == 1 ? 1 : P.tma_kind), nstg = P.nstg, stg_bytes = P.stg_bytes;
  const int nbuf = R > 32 ? 2 : 4, buf_cols = kTmemCols / nbuf;

  unsigned char *sA = smem, *sB = smem + 2 * A_BYTES;
  const int stg_off = (2 * A_BYTES + B_BYTES + 1023) & ~1023;
  unsigned char *stg0 = smem + stg_off;
  unsigned char *s_out = stg0 + nstg * stg_bytes;  // x stages: one output box per epilogue warp
  int *s_rowexp = reinterpret_cast<int *>(s_out + P.out_box_bytes * kXEpiWarps);
  int16_t *s_etau = reinterpret_cast<int16_t *>(s_rowexp + 64);
  uint64_t *bars = reinterpret_cast<uint64_t *>(s_etau + kXEtau * kTile);
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 28);
  const uint32_t bar0 = smem_u32(bars);
  auto a_full = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  auto a_empty = [&](int i) { return bar0 + 8u * (uint32_t)(2 + i); };
  auto s_full = [&](int i) { return bar0 + 8u * (uint32_t)(4 + i); };
  auto s_empty = [&](int i) { return bar0 + 8u * (uint32_t)(6 + i); };
  auto t_full = [&](int i) { return bar0 + 8u * (uint32_t)(8 + i); };
  auto t_empty = [&](int i) { return bar0 + 8u * (uint32_t)(12 + i); };
  auto meta_full = [&](int i) { return bar0 + 8u * (uint32_t)(16 + i); };
  const uint32_t drain = bar0 + 8u * 24u, b_full = bar0 + 8u * 25u;
  const long long WL = P.wait_limit;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == kXProdWarps + kXEpiWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(a_full(i), kXProdWarps);
      mbar_init(a_empty(i), 1);
      mbar_init(s_full(i), kind ? 1 : kXProd);
      mbar_init(s_empty(i), kXProdWarps);
    }
    // warps that read a TMEM buffer: all, where a tile has two units of 8 rows (N = 16 with one operator
    // or upwinded) half of them in turn, in a halo pass one per lane quadrant in turn
    const int readers = HALO ? kXEpiWarps / 4 : kXEpiWarps / 4 * min(4, (UPWIND ? 1 : P.nseg[0]) * (N / kXUnit));
    for (int i = 0; i < 4; ++i) { mbar_init(t_full(i), 1); mbar_init(t_empty(i), readers); }
    for (int i = 0; i < kXEtau; ++i) mbar_init(meta_full(i), kXProdWarps);
    mbar_init(drain, 1);
    mbar_init(b_full, kXEpiWarps);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  bool failed = false;
  chain_next();
  const TileRange tr = tile_range(P);
  // a whole warp waits together: its lanes leave a loop on the same outcome
  auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, WL));
  };

  if (warp < kXProdWarps) {
    // ================================================================ producers
    asm volatile("setmaxnreg.inc.sync.aligned.u32 96;");
    if constexpr (!GEN) {
      // the columns behind the pencil (K padding; halo columns are rewritten per tile) stay zero: each lane
      // clears its pencil's rows of one buffer
      const int zp = warp * 16 + (lane & 15);
      unsigned char *z = sA + (lane >> 4) * A_BYTES + (zp >> 3) * (NCH * 128) + (zp & 7) * 16;
#pragma unroll
      for (int sl = 0; sl < kSl; ++sl)
#pragma unroll
        for (int ch = (N + 8) / 8; ch < NCH; ++ch)
          *reinterpret_cast<uint4 *>(z + sl * SLICE + ch * 128) = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
    }
    chain_wait();
    const int pl = warp * 16 + (lane & 15), half = lane >> 4;
    // staged element j of this lane's pencil: x rows in boxes of 64 bytes, 16-byte chunks swizzled by
    // the row (chunk ^ (row / 2) % 4: eight rows' chunks cover all banks); columns [t1][j][N] along y,
    // [j][128] along z
    const int col_base = axis == 1 ? (pl / N) * (DIRECT ? N : E) * N + pl % N : pl, col_step = axis == 1 ? N : kTile;
    auto stg_byte = [&](int pp, int j) -> int {  // for the cp.async path and single elements
      if (axis == 2) {
        const int c = j * ES / 16;
        return (c >> 2) * (kTile * kXRowBytes) + pp * kXRowBytes + (((c & 3) ^ ((pp >> 1) & 3)) << 4) + (j * ES) % 16;
      }
      return ((axis == 1 ? (pp / N) * E * N + pp % N : pp) + j * col_step) * ES;
    };
    auto load = [&](const unsigned char *st, int j0, int n, TI *v) {  // n elements from j0 (multiples of 4)
      if (axis == 2) {
        constexpr int VE = 16 / ES;
#pragma unroll
        for (int k = 0; k < 8; k += VE) {
          if (k >= n) break;
          const int c = (j0 + k) * ES / 16;
          const uint4 u = *reinterpret_cast<const uint4 *>(st + (c >> 2) * (kTile * kXRowBytes) + pl * kXRowBytes +
                                                           (((c & 3) ^ ((pl >> 1) & 3)) << 4));
          if constexpr (ES == 8) {
            v[k] = __hiloint2double((int)u.y, (int)u.x);
            v[k + 1] = __hiloint2double((int)u.w, (int)u.z);
          } else {
            v[k] = __uint_as_float(u.x);
            v[k + 1] = __uint_as_float(u.y);
            v[k + 2] = __uint_as_float(u.z);
            v[k + 3] = __uint_as_float(u.w);
          }
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (k < n) v[k] = reinterpret_cast<const TI *>(st)[col_base + (j0 + k) * col_step];
      }
    };
    // cp.async staging (tiles that are not a box of the input): all producers, element or 16-byte copies
    const long long is0 = (long long)P.in_dims[1] * P.in_dims[2], is1 = P.in_dims[2];
    const long long s_t1 = stride_of(P.t1, is0, is1), s_t2 = stride_of(P.t2, is0, is1),
                    s_ax = stride_of(axis, is0, is1);
    const int in_s1 = P.t1 == 0 ? P.in_start[0] : (P.t1 == 1 ? P.in_start[1] : P.in_start[2]);
    const int in_s2 = P.t2 == 0 ? P.in_start[0] : (P.t2 == 1 ? P.in_start[1] : P.in_start[2]);
    const long long E3 = (long long)E * E * E;
    // 16-byte rows along x: consecutive threads on consecutive pieces.  A thread per row touches 32 rows per warp
    // instruction (256^3, 4 fields, S_x staged this way: 0.93 -> 0.46 ms together with the row boxes on the way
    // out, see plan_out_tma).  Rows that are not aligned stay with a thread per row, element by element: the
    // spread-out form was up to 1.37 times slower there (16^3 blocks, FP32).
    auto copy_rows = [&](unsigned char *st, int tile) {
      constexpr int VE = 16 / ES;
      const int job = fdiv(tile, P.inv_tpj), p0 = (tile - job * P.tiles_per_job) * kTile, np = P.n1 * P.n2;
      const int lb = fdiv(job, P.inv_nf), q = job - lb * P.nf;
      const TI *in = static_cast<const TI *>(P.in) +
                     (!P.in_field ? (long long)job * (long long)P.in_box
                      : P.contig  ? (long long)P.nf * P.ext0 + (long long)job * E3
                                  : (long long)P.nf * P.extpre[P.blocks[lb]] + (long long)q * E3);
      const int per = E / VE;            // pieces of a row
      const int dp = kXProd / per, dr = kXProd - dp * per;
      int pp = tid / per, r = tid - pp * per;
      while (pp < kTile) {
        const int p = p0 + pp;
        if (p < np) {
          const int t1 = fdiv(p, P.inv_n2), t2 = p - t1 * P.n2;
          cp_async16(st + stg_byte(pp, r * VE), in + (long long)(in_s1 + t1) * s_t1 + (long long)(in_s2 + t2) * s_t2 + r * VE);
        }
        pp += dp;
        r += dr;
        if (r >= per) {
          r -= per;
          ++pp;
        }
      }
    };
    auto prefetch = [&](int tile, int sb) {
      unsigned char *st = stg0 + sb * stg_bytes;
      if (axis == 2 && P.xrow) {
        copy_rows(st, tile);
      } else {
        const int pp = tid & (kTile - 1), jq = tid >> 7;
        const TileCoord c = tile_coord(P, tile, pp);
        if (c.valid) {
          const long long job = (long long)c.lb * P.nf + c.q;
          const long long ib = (!P.in_field ? job * (long long)P.in_box
                                : P.contig  ? (long long)P.nf * P.ext0 + job * E3
                                            : (long long)P.nf * P.extpre[c.b] + (long long)c.q * E3) +
                               (long long)(in_s1 + c.t1) * s_t1 + (long long)(in_s2 + c.t2) * s_t2;
          const TI *src = static_cast<const TI *>(P.in) + ib;
          for (int j = jq; j < E; j += 2) {
            if constexpr (ES == 8) cp_async8(st + stg_byte(pp, j), src + (long long)j * s_ax);
            else cp_async4(st + stg_byte(pp, j), src + (long long)j * s_ax);
          }
        }
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(s_full(sb)) : "memory");
    };
    // The neighbours' previous iterate at k^c, as columns E + m of the pencil: m = 2d from the lower
    // neighbour's row N-2 (side 1), m = 2d + 1 from the upper neighbour's row 1 (side 0), degree slot d.
    // Layout [block][field][side][pencil][halo_nd]: a stage of one degree holds (and moves) only its own.
    // With TMA the copies of a tile bring its two runs of 128 pencils behind the staged pencils; loaded by
    // the producers themselves, a tile ahead, they cost the T stages at 256^3 a quarter (0.31 against
    // 0.28 ms: the index arithmetic sat on the producers' critical path).
    const int np = P.n1 * P.n2;
    auto halo = [&](const unsigned char *st, int tile, int m) -> TI {
      const int d = m >> 1, up = m & 1, dd = P.halo_nd == 2 ? d : 0;
      if (!((P.halo_deg_mask >> d) & 1)) return TI(0);
      if (kind) return TI(reinterpret_cast<const double *>(st + P.halo_stg)[(up * kTile + pl) * P.halo_nd + dd]);
      const TileCoord c = tile_coord(P, tile, pl);
      if (!c.valid) return TI(0);
      const int sg = up ? 1 : -1;
      const int nb = P.nbr[c.b * 26 + dir_index_dev(axis == 0 ? sg : 0, axis == 1 ? sg : 0, axis == 2 ? sg : 0)];
      const long long hp = (((long long)nb * P.nf + c.q) * 2 + (up ? 0 : 1)) * np + tile_pencil(P, tile, pl);
      return TI(P.halo_in[hp * P.halo_nd + dd]);
    };
    constexpr int NFULL = GEN ? (NCH + 1) / 2 : N / 16;          // whole chunks of this lane
    constexpr int NV = NFULL * 8 + (GEN ? 0 : 4 + (ITER ? 2 : 0));  // values of this lane
    if (!kind)
      for (int k = 0, t = tr.first; k < nstg && t < tr.end; ++k, t += tr.step) prefetch(t, k);
    int it = 0;
    for (int tile = tr.first; tile < tr.end; tile += tr.step, ++it) {
      const int buf = it & 1, sb = nstg == 2 ? it & 1 : 0, su = nstg == 2 ? it >> 1 : it;
      if (!wait(s_full(sb), (uint32_t)(su & 1))) { failed = true; break; }
      const unsigned char *st = stg0 + sb * stg_bytes;
      TI v[NV];
      if constexpr (GEN) {
        const bool valid = kind || tile_coord(P, tile, pl).valid;
#pragma unroll
        for (int h = 0; h < NFULL; ++h)
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int j = (half + 2 * h) * 8 + k;
            TI x = TI(0);
            if (valid && j < E) x = *reinterpret_cast<const TI *>(st + stg_byte(pl, j));
            else if (ITER && valid && j < E + 4) x = halo(st, tile, j - E);
            v[h * 8 + k] = x;
          }
      } else {
#pragma unroll
        for (int h = 0; h < NFULL; ++h) load(st, (half + 2 * h) * 8, 8, v + h * 8);
        if constexpr (DIRECT) {
          // the lower (upper) neighbour's four columns: [128 rows][4] in 32-byte rows, chunk ^ (row / 4) % 2,
          // or [t1][4][N]
          const unsigned char *gs = st + kTile * N * ES + half * (kTile * 4 * ES);
          if (axis == 2) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const double2 u = *reinterpret_cast<const double2 *>(gs + pl * 32 + ((k ^ ((pl >> 2) & 1)) << 4));
              v[NFULL * 8 + 2 * k] = u.x;
              v[NFULL * 8 + 2 * k + 1] = u.y;
            }
          } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              v[NFULL * 8 + k] = reinterpret_cast<const TI *>(gs)[(pl / N) * 4 * N + pl % N + k * N];
          }
        } else {
          load(st, N + 4 * half, 4, v + NFULL * 8);
        }
        if constexpr (ITER) {  // the two lanes of a pencil take one degree slot each
          v[NFULL * 8 + 4] = halo(st, tile, 2 * half);
          v[NFULL * 8 + 5] = halo(st, tile, 2 * half + 1);
        }
        if (!kind && !tile_coord(P, tile, pl).valid) {
#pragma unroll
          for (int k = 0; k < NV; ++k) v[k] = TI(0);
        }
      }
      uint32_t am = 0;
#pragma unroll
      for (int k = 0; k < NV; ++k) am = max(am, abs_word(v[k]));
      am = max(am, __shfl_xor_sync(0xffffffffu, am, 16));  // also: every lane has read its staged values
      if (lane == 0) mbar_arrive(s_empty(sb));
      if (!kind && tile + nstg * tr.step < tr.end) {
        if (!wait(s_empty(sb), (uint32_t)(su & 1))) { failed = true; break; }
        prefetch(tile + nstg * tr.step, sb);
      }
      int emax = (int)(am >> exp_shift(TI(0)));
      // a NaN or an infinity anywhere in the pencil: every output of the pencil is NaN (the epilogue
      // sees kBadTau); its digits are written as zeros
      const bool bad = emax >= nonfinite_exp(TI(0));
      const int etau = bad ? kBadTau16 : tau_exp(emax, TI(0));
      if (emax < 64) {
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = lift64(v[k]);
        emax += 64;
      }
      if (bad) emax += 128;  // every shift runs past the significand
      const int C = split_base(emax, TI(0));
      // A[buf] must be free: the MMAs of its previous use have completed
      if (it >= 2 && !wait(a_empty(buf), (uint32_t)(((it >> 1) - 1) & 1))) { failed = true; break; }
      if (half == 0) s_etau[(it & (kXEtau - 1)) * kTile + pl] = (int16_t)etau;
      // canonical K-major rows, no swizzle: [row / 8][chunk][row % 8][8]
      unsigned char *row = sA + buf * A_BYTES + (pl >> 3) * (NCH * 128) + (pl & 7) * 16;
#pragma unroll
      for (int h = 0; h < NFULL; ++h) {
        if (GEN && half + 2 * h >= NCH) break;
        split_store<TI, 8>(v + h * 8, C, row + (half + 2 * h) * 128, SLICE);
      }
      if constexpr (!GEN) {
        split_store<TI, 4>(v + NFULL * 8, C, row + (N / 8) * 128 + 8 * half, SLICE);
        if constexpr (ITER) split_store<TI, 2>(v + NFULL * 8 + 4, C, row + (N / 8 + 1) * 128 + 4 * half, SLICE);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(meta_full(it & (kXEtau - 1)));
        mbar_arrive(a_full(buf));
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp < kXProdWarps + kXEpiWarps) {
    // ================================================================ epilogue
    // First the operator digits, while the first tiles are copied and split: slices stacked along the MMA's
    // N rows, [t][segment][N].  (With the whole CTA loading them before it starts, a launch of one tile per
    // CTA took 0.3 us longer, 256^3 with nine ops 20 us.)
    {
      const int et = tid - kXProd;
      constexpr int ET = kXEpiWarps * 32, U = SR * KP * 2 / 16;
      for (int sg = 0; sg < P.nseg[0]; ++sg) {
        const uint4 *src = reinterpret_cast<const uint4 *>(P.seg_img[0][sg]);
        for (int i = et; i < kSl * U; i += ET) {
          const int t = i / U, r = i - t * U;
          reinterpret_cast<uint4 *>(sB + (t * R + sg * SR) * KP * 2)[r] = __ldg(src + i);
        }
        for (int i = et; i < SR; i += ET) s_rowexp[sg * SR + i] = P.seg_exp[0][sg][i];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(b_full);
      asm volatile("bar.sync 1, %0;" ::"n"(ET) : "memory");  // the row exponents
      chain_wait();
    }
    const int quad = warp & 3, ew = (warp - kXProdWarps) >> 2;
    const int pl = quad * 32 + lane;
    constexpr int UPS = N / kXUnit;  // units per segment
    constexpr long long n3 = (long long)N * N * N;
    const long long f_t1 = axis == 0 ? N : N * N, f_t2 = axis == 2 ? N : 1,
                    f_ax = axis == 2 ? 1 : (axis == 1 ? N : N * N);
    const long long ss0 = (long long)P.sc_dims[1] * P.sc_dims[2], ss1 = P.sc_dims[2];
    const long long c_t1 = stride_of(P.t1, ss0, ss1), c_t2 = stride_of(P.t2, ss0, ss1);
    // the intermediate's boxes: [N][N][E] after the y stage, [N][E][E] after the z stage
    const long long c_ax = GEN ? stride_of(axis, ss0, ss1) : (AXIS == 1 ? E : E * E);
    const int sc_s1 = P.t1 == 0 ? P.sc_start[0] : (P.t1 == 1 ? P.sc_start[1] : P.sc_start[2]);
    const int sc_s2 = P.t2 == 0 ? P.sc_start[0] : (P.t2 == 1 ? P.sc_start[1] : P.sc_start[2]);
    // range of the row exponents: with the pencil scale it decides whether every output of a thread
    // stays in the normal range
    int rlo = s_rowexp[0], rhi = rlo;
    for (int i = 1; i < R; ++i) {
      rlo = min(rlo, s_rowexp[i]);
      rhi = max(rhi, s_rowexp[i]);
    }
    // |Y| < 2^47: Y 2^E is normal; FP32: the scale itself is a normal float
    constexpr int kLo = sizeof(TO) == 8 ? -1022 + kYUnit : -126 + kFUnit;
    constexpr int kHi = sizeof(TO) == 8 ? 976 + kYUnit : 127 + kFUnit;
    if constexpr (HALO) {
      // rows 0..3: row 1 and row N-2 of degree slot 0, then of slot 1 (biased schemes: rows 1 and 2);
      // the tiles go round the four warps of a lane quadrant
      const int np = P.n1 * P.n2;
      int it = 0;
      for (int tile = tr.first; tile < tr.end; tile += tr.step, ++it) {
        if ((it & 3) != ew) continue;
        const TileCoord c = tile_coord(P, tile, pl);
        if (!wait(meta_full(it & (kXEtau - 1)), (uint32_t)((it / kXEtau) & 1))) { failed = true; break; }
        const int etau16 = s_etau[(it & (kXEtau - 1)) * kTile + pl], etau = etau16 == kBadTau16 ? kBadTau : etau16;
        if (!wait(t_full(ew), (uint32_t)((it >> 2) & 1))) { failed = true; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t acc[kSl][8];
        load_levels(acc, tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(ew * buf_cols), R);
        release_levels(t_empty(ew));
        double h[4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
          h[r] = scaled_double<true>(__ll2double_rn(exact_y(acc, r)), s_rowexp[r] + etau - kYUnit, etau == kBadTau);
        if (!c.valid) continue;
        double *o = P.halo_out + (((long long)c.b * P.nf + c.q) * 2 * np + tile_pencil(P, tile, pl)) * P.halo_nd;
        const long long side = (long long)np * P.halo_nd;
        if (P.halo_nd == 2) {
          *reinterpret_cast<double2 *>(o) = make_double2(h[0], h[2]);
          *reinterpret_cast<double2 *>(o + side) = make_double2(h[1], h[3]);
        } else {
          const bool second = P.halo_deg_mask == 2;
          o[0] = second ? h[2] : h[0];
          o[side] = second ? h[3] : h[1];
        }
      }
    } else {
    const int units = (UPWIND ? 1 : P.nseg[0]) * UPS;
    const bool rows_out = axis == 2 && P.out_box_bytes != 0;
    unsigned char *box = s_out + (warp - kXProdWarps) * P.out_box_bytes;
    int it = 0;
    for (int tile = tr.first; tile < tr.end; tile += tr.step, ++it) {
      // units of this warp: ew and ew + 4 of the tile, rotated from tile to tile so that units that
      // also write an intermediate go round; with two units in a tile, every second tile
      int u0 = (ew + it) & 3;
      if (u0 >= units) continue;
      const TileCoord c = tile_coord(P, tile, pl);
      const bool interior = c.valid && P.int_lo1 <= c.t1 && c.t1 < P.int_hi1 && P.int_lo2 <= c.t2 && c.t2 < P.int_hi2;
      TO *fb = static_cast<TO *>(P.out);
      if (interior)
        fb += (long long)P.nf * P.nops * (P.contig ? P.int0 + (long long)c.lb * n3 : P.intpre[c.b]) +
              (long long)c.q * P.nops * n3 + (long long)(c.t1 - P.int_lo1) * f_t1 + (long long)(c.t2 - P.int_lo2) * f_t2;
      double *sb = P.scratch_out;
      long long gx = 0, gy = 0;  // offsets from the intermediate to the neighbours' ghost copies
      if ((AXIS != 2) && sb != nullptr && c.valid) {
        sb += ((long long)(P.sc_local ? P.sc_local[c.lb] : c.lb) * P.nf + c.q) * (long long)P.sc_box +
              (long long)(sc_s1 + c.t1) * c_t1 + (long long)(sc_s2 + c.t2) * c_t2;
        if (P.ghost_x) {
          const int xs = sc_s2 + c.t2;  // t2 is the x axis in the stages that write intermediates
          const long long jump = (long long)P.nf * (long long)P.sc_box;
          // (no copy where the block has no such neighbour: it computes that strip itself)
          const int *nl = P.nl + c.lb * 4;
          if (xs < 2 * g) { if (nl[0] >= 0) gx = (long long)(nl[0] - c.lb) * jump + N; }
          else if (xs >= N) { if (nl[1] >= 0) gx = (long long)(nl[1] - c.lb) * jump - N; }
          if (P.ghost_y) {
            const int ys = sc_s1 + c.t1;  // t1 is the y axis (z stage)
            if (ys < 2 * g) { if (nl[2] >= 0) gy = (long long)(nl[2] - c.lb) * jump + (long long)N * ss1; }
            else if (ys >= N) { if (nl[3] >= 0) gy = (long long)(nl[3] - c.lb) * jump - (long long)N * ss1; }
          }
        }
      }
      if (!wait(meta_full(it & (kXEtau - 1)), (uint32_t)((it / kXEtau) & 1))) { failed = true; break; }
      const int etau16 = s_etau[(it & (kXEtau - 1)) * kTile + pl], etau = etau16 == kBadTau16 ? kBadTau : etau16;
      const bool bad = etau == kBadTau;
      const bool safe = !bad && etau + rlo >= kLo && etau + rhi <= kHi;
      const int tb = it & (nbuf - 1), tu = nbuf == 2 ? it >> 1 : it >> 2;
      if (!wait(t_full(tb), (uint32_t)(tu & 1))) { failed = true; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(tb * buf_cols);
      // one TMA store of this warp's output box (its previous store has read it, see box_free)
      auto box_free = [&]() {
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
      };
      auto box_store = [&](int op, int o) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {  // (fb: this pencil's row of op 0; every block starts at a multiple of 512 values)
          const unsigned long long at = reinterpret_cast<char *>(fb) - static_cast<char *>(P.out);
          const int row = (int)(at / (N * sizeof(TO))) + op * N * N;
          asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                           reinterpret_cast<uint64_t>(&P.tmap_out)),
                       "r"(o), "r"(row), "r"(smem_u32(box))
                       : "memory");
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      };
      if constexpr (UPWIND) {
        // the shift's signs along this pencil, one bit per point
        const uint32_t signs =
            interior ? P.upwind[(c.lb * 3 + 2 - axis) * N * N + tile_pencil(P, tile, pl)] : 0u;
#pragma unroll 1
        for (int u = u0; u < units; u += 4) {
          const int o = u * kXUnit;
          TO *f0 = fb + (long long)P.seg_op[0][0] * n3 + o * f_ax;
          const uint32_t ta = tbase + (uint32_t)o, rel = u + 4 >= units ? t_empty(tb) : 0u;
          const uint32_t w = signs >> o;
          const bool all = __all_sync(0xffffffffu, safe && interior);
          if (all && axis == 2 && rows_out) {
            box_free();
            rows_upwind<TO, true, true>(ta, R, N, etau, s_rowexp + o, N, f0, 1, true, w, rel, box);
            box_store(P.seg_op[0][0], o);
          } else if (all) {
            rows_upwind<TO, false, true>(ta, R, N, etau, s_rowexp + o, N, f0, f_ax, true, w, rel, nullptr);
          } else {
            rows_upwind<TO, false, false>(ta, R, N, etau, s_rowexp + o, N, f0, f_ax, interior, w, rel, nullptr);
          }
        }
      } else {
#pragma unroll 1
      for (int u = u0; u < units; u += 4) {
        const int sg = u >= UPS ? 1 : 0, o = (u - sg * UPS) * kXUnit;
        const int mode = P.seg_mode[0][sg];
        const bool wf = (mode == 0 || mode == 3) && interior, ws = (mode == 2 || mode == 3) && c.valid;
        const int *rexp = s_rowexp + sg * N + o;
        TO *f0 = fb + (long long)P.seg_op[0][sg] * n3 + o * f_ax;
        double *s0 = sb + o * c_ax;
        const uint32_t ta = tbase + (uint32_t)(sg * N + o);
        const uint32_t rel = u + 4 >= units ? t_empty(tb) : 0u;
        // warp-uniform choices: tcgen05.ld is a warp-wide instruction
        const bool all_f = __all_sync(0xffffffffu, safe && wf), any_s = __any_sync(0xffffffffu, ws);
        if (axis == 2 && rows_out && all_f) {
          box_free();
          rows_fast<TO, true, true, false>(ta, R, etau, rexp, f0, 1, nullptr, 0, 0, 0, rel, box);
          box_store(P.seg_op[0][sg], o);
        } else if (all_f && !any_s) {
          rows_fast<TO, false, true, false>(ta, R, etau, rexp, f0, f_ax, nullptr, 0, 0, 0, rel, nullptr);
        } else {
          const bool all_s = __all_sync(0xffffffffu, safe && ws), any_f = __any_sync(0xffffffffu, wf);
          if (AXIS != 2 && all_f && all_s)
            rows_fast<TO, false, true, true>(ta, R, etau, rexp, f0, f_ax, s0, c_ax, gx, gy, rel, nullptr);
          else if (AXIS != 2 && all_s && !any_f)
            rows_fast<TO, false, false, true>(ta, R, etau, rexp, f0, 0, s0, c_ax, gx, gy, rel, nullptr);
          else
            rows_any<TO>(ta, R, etau, rexp, f0, f_ax, s0, c_ax, gx, gy, wf, ws, rel);
        }
      }
    }
    }
    // the output boxes must have been read before the CTA leaves
    if (rows_out && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  } else if (warp == kXProdWarps + kXEpiWarps) {
    // ================================================================ MMA issue
    asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
    if (lane == 0) {
      bool issued = false;
      int it = 0;
      if (!mbar_wait_bounded(b_full, 0u, WL)) failed = true;
      // (it touches no global memory, but the limit of its first wait for a tile must not count the time that
      // the launch before still takes: the producers are held until then)
      chain_wait();
      for (int tile = tr.first; tile < tr.end; tile += tr.step, ++it) {
        const int buf = it & 1, tb = it & (nbuf - 1), tu = nbuf == 2 ? it >> 1 : it >> 2;
        if (failed || !mbar_wait_bounded(a_full(buf), (uint32_t)((it >> 1) & 1), WL) ||
            (tu > 0 && !mbar_wait_bounded(t_empty(tb), (uint32_t)((tu - 1) & 1), WL))) {
          failed = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a0 = smem_u32(sA) + (uint32_t)(buf * A_BYTES), b0 = smem_u32(sB);
        const uint32_t cb = tmem + (uint32_t)(tb * buf_cols);
        // digit s of the pencils against operator digits 0 .. 3-s, stacked along N: each lands on the
        // columns of its level s + t
#pragma unroll
        for (int s = 0; s < kSl; ++s) {
          const uint32_t idesc = (1u << 4) | ((uint32_t)(((kSl - s) * R) >> 3) << 17) | ((uint32_t)(kTile >> 4) << 24);
#pragma unroll
          for (int kk = 0; kk < KP / 16; ++kk)
            mma_16bit(cb + (uint32_t)(s * R), smem_desc(a0 + (uint32_t)(s * SLICE + kk * 256), 128, KP * 16),
                      smem_desc(b0 + (uint32_t)(kk * 256), 128, KP * 16), idesc, (s | kk) ? 1u : 0u);
        }
        mma_commit(t_full(tb));
        mma_commit(a_empty(buf));
        issued = true;
      }
      // every MMA issued completes before TMEM is released
      if (issued) {
        mma_commit(drain);
        mbar_wait_bounded(drain, 0u);
      }
    }
  } else if (warp == kXProdWarps + kXEpiWarps + 1) {
    // ================================================================ TMA issue
    asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
    if (lane == 0 && kind) {
      chain_wait();
      const uint64_t tmap = reinterpret_cast<uint64_t>(&P.tmap);
      int it = 0;
      for (int tile = tr.first; tile < tr.end; tile += tr.step, ++it) {
        const int sb = nstg == 2 ? it & 1 : 0, su = nstg == 2 ? it >> 1 : it;
        const int job = fdiv(tile, P.inv_tpj), tj = tile - job * P.tiles_per_job, t1_0 = tj * (kTile / N);
        int nb[2] = {0, 0}, q = 0;
        if constexpr (ITER || DIRECT) {  // (looked up before the wait for the staging buffer)
          const int lb = fdiv(job, P.inv_nf), b = P.contig ? P.b0 + lb : P.blocks[lb];
          q = job - lb * P.nf;
          nb[0] = __ldg(P.nbr + b * 26 + dir_index_dev(axis == 0 ? -1 : 0, axis == 1 ? -1 : 0, axis == 2 ? -1 : 0));
          nb[1] = __ldg(P.nbr + b * 26 + dir_index_dev(axis == 0 ? 1 : 0, axis == 1 ? 1 : 0, axis == 2 ? 1 : 0));
        }
        if (su > 0 && !mbar_wait_bounded(s_empty(sb), (uint32_t)((su - 1) & 1), WL)) { failed = true; break; }
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_full(sb)), "r"(P.tma_bytes)
                     : "memory");
        if constexpr (ITER) {
          const int np = P.n1 * P.n2, bytes = kTile * P.halo_nd * 8;
#pragma unroll
          for (int up = 0; up < 2; ++up) {
            const double *src = P.halo_in + ((((long long)nb[up] * P.nf + q) * 2 + (up ? 0 : 1)) * np + tj * kTile) * P.halo_nd;
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_u32(stg0) + (uint32_t)(sb * stg_bytes + P.halo_stg + up * bytes)),
                "l"(src), "r"(bytes), "r"(s_full(sb))
                : "memory");
          }
        }
        if constexpr (DIRECT) {
          // own points and the two ghost boxes from the output slot [job][op][z][y][x]
          auto box = [&](const CUtensorMap &m, uint32_t off, int cx, int cy, int j) {
            const int cz = (j * P.nops + P.direct_op) * N + t1_0;
            asm volatile(
                "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
                "%4}], [%5];" ::"r"(smem_u32(stg0) + (uint32_t)(sb * stg_bytes) + off),
                "l"(reinterpret_cast<uint64_t>(&m)), "r"(cx), "r"(cy), "r"(cz), "r"(s_full(sb))
                : "memory");
          };
          if (axis == 2) {
            for (int bx = 0; bx < N / 8; ++bx) box(P.tmap, bx * kTile * kXRowBytes, bx * 8, 0, job);
          } else {
            box(P.tmap, 0, 0, 0, job);
          }
#pragma unroll
          for (int up = 0; up < 2; ++up)
            box(P.tmap_ghost, kTile * N * ES + up * (kTile * 4 * ES), axis == 2 && !up ? N - 4 : 0,
                axis == 1 && !up ? N - 4 : 0, (nb[up] - P.b0) * P.nf + q);
          continue;
        }
        const int cz = P.in_start[0] + job * P.tma_zstep + (axis == 0 ? 0 : t1_0);
        const int cy = P.in_start[1] + (axis == 0 ? t1_0 : 0);
        for (int bx = 0; bx < P.tma_boxes; ++bx) {
          const uint32_t dst = smem_u32(stg0) + (uint32_t)(sb * stg_bytes + bx * kTile * kXRowBytes);
          const int cx = P.in_start[2] + bx * (kXRowBytes / ES);
          asm volatile(
              "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
              "%4}], [%5];" ::"r"(dst),
              "l"(tmap), "r"(cx), "r"(cy), "r"(cz), "r"(s_full(sb))
              : "memory");
        }
      }
      // every copy lands before the CTA leaves (the producers may have given up on theirs)
      for (int k = max(0, it - nstg); k < it; ++k)
        mbar_wait_bounded(s_full(nstg == 2 ? k & 1 : 0), (uint32_t)((nstg == 2 ? k >> 1 : k) & 1));
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
  }

  if (failed) atomicExch(P.status, (int)CFD_ERR_TIMEOUT);
  __syncwarp();
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kXProdWarps + kXEpiWarps) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

}  // namespace
}  // namespace cfd
