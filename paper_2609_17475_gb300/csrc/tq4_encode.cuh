// TQ4 encoder with one warp per vector, shared by the append kernel's general
// path and the fused append + decode step.
#pragma once
#include <cmath>

#include "common.cuh"
#include "tq4.cuh"

namespace jfkv {

template <int E>
__device__ __forceinline__ void load_bf16(const uint16_t* src, float (&x)[E]) {
  if constexpr (E == 8) {
    const uint4 w = *reinterpret_cast<const uint4*>(src);
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { x[2 * i] = bf16lo_to_f32(ws[i]); x[2 * i + 1] = bf16hi_to_f32(ws[i]); }
  } else {
    const uint2 w = *reinterpret_cast<const uint2*>(src);
    x[0] = bf16lo_to_f32(w.x); x[1] = bf16hi_to_f32(w.x);
    x[2] = bf16lo_to_f32(w.y); x[3] = bf16hi_to_f32(w.y);
  }
}

// Count of the 15 ascending thresholds T_k with u > T_k, by a branch-free
// 4-level search, and the thresholds bracketing u (lo < u <= hi; -inf / +inf
// past the ends).
__device__ __forceinline__ int bracket15(float u, const float (&T)[15], float& lo, float& hi) {
  const bool b3 = u > T[7];
  lo = b3 ? T[7] : -INFINITY;
  hi = b3 ? INFINITY : T[7];
  const float t2 = b3 ? T[11] : T[3];
  const bool b2 = u > t2;
  lo = b2 ? t2 : lo;
  hi = b2 ? hi : t2;
  const float t1 = b3 ? (b2 ? T[13] : T[9]) : (b2 ? T[5] : T[1]);
  const bool b1 = u > t1;
  lo = b1 ? t1 : lo;
  hi = b1 ? hi : t1;
  const float t0 = b3 ? (b2 ? (b1 ? T[14] : T[12]) : (b1 ? T[10] : T[8]))
                      : (b2 ? (b1 ? T[6] : T[4]) : (b1 ? T[2] : T[0]));
  const bool b0 = u > t0;
  lo = b0 ? t0 : lo;
  hi = b0 ? hi : t0;
  return (b3 ? 8 : 0) + (b2 ? 4 : 0) + (b1 ? 2 : 0) + (b0 ? 1 : 0);
}

// (s_hi, s_lo) += b for a double-float accumulator (Knuth's TwoSum; the
// error term of s_hi + b is exact)
__device__ __forceinline__ void two_sum_acc(float& sh, float& sl, float b) {
  const float s = __fadd_rn(sh, b);
  const float bb = __fsub_rn(s, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  sh = s;
  sl = __fadd_rn(sl, err);
}

// RN32(sqrt(s)) for the double-float sum s = sh + sl (error about 2^-40 s):
// rounded from r = RN32(sqrt(sh)) and the exact residual sh - r^2 (one fma).
// sure: the result is farther than 2^-10 half-ulp from a rounding boundary and
// s is in the safe range.  sl first leaves what sh can hold to sh: summed up, it
// may be more than an ulp of it, r then more than one off, and the result not
// sure (one vector in ~80 of the append's, each a wait for fp64: 9 rows of
// 24/4/256, 5.2 us of device time, 2.8 now).
__device__ __forceinline__ float rho_from_sum(float sh, float sl, bool& sure) {
  const float hi = __fadd_rn(sh, sl);
  sl = __fsub_rn(sl, __fsub_rn(hi, sh));                 // exact: |sl| <= |sh|
  sh = hi;
  const float r = __fsqrt_rn(sh);
  const float res = __fmaf_rn(-r, r, sh);                // exact: s_hi - r^2
  // sqrt(s) = r + dl up to ~2^-41 r; rounding boundaries at half an ulp on
  // either side (the spacing below a power of two is half the one above)
  const float dl = __fmul_rn(__fadd_rn(res, sl), __fdiv_rn(0.5f, r));
  const float up = __int_as_float(__float_as_int(r) + 1);
  const float dn = __int_as_float(__float_as_int(r) - 1);
  const float half = (dl > 0.f) ? 0.5f * (up - r) : 0.5f * (r - dn);
  const float ad = fabsf(dl);
  sure = (sh >= 0x1p-100f) && (sh <= 0x1p+120f) && (fabsf(ad - half) > half * 0x1p-10f) &&
         !(ad > 2.f * half);
  return (ad < half) ? r : (dl > 0.f ? up : dn);
}

// Encode one vector of D bf16 elements (src) with a whole warp: returns this
// lane's E = D/32 indices (element E lane + e in bits 4e .. 4e+3) and sets
// rho (the fp32 norm; every lane gets the same value).  kind 0: K, 1: V.
template <int D>
__device__ __forceinline__ uint32_t tq4_encode(const uint16_t* src, int kind, const Tq4Params& prm,
                                               int lane, float& rho_out) {
  constexpr int E = D / 32;
  float x[E];
  load_bf16<E>(src + lane * E, x);
  const uint32_t sbits = ((kind ? prm.sv : prm.sk)[(lane * E) >> 5]) >> ((lane * E) & 31);

  // rho = RN32(sqrt(s)), s the fp64 sum of squares.  Squares of bf16 values
  // are exact in fp32; their sum is carried as a double-float (TwoSum, error
  // about 2^-40 s) and its square root rounded from r = RN32(sqrt(s_hi)) and
  // the exact residual s_hi - r^2 (one fma).  When the result lies within
  // 2^-10 half-ulp of a rounding boundary, or s is out of the safe range, the
  // warp recomputes s in fp64 (GB300's fp64 rate is low, so this stays rare).
  float sh = 0.f, sl = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) two_sum_acc(sh, sl, __fmul_rn(x[e], x[e]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(0xffffffffu, sh, o);
    const float bl = __shfl_xor_sync(0xffffffffu, sl, o);
    two_sum_acc(sh, sl, bh);
    sl = __fadd_rn(sl, bl);
  }
  float rho;
  {
    bool sure;
    rho = rho_from_sum(sh, sl, sure);
    if (!sure) {   // uniform: every lane holds the same (sh, sl)
      double s = 0.0;
#pragma unroll
      for (int e = 0; e < E; ++e) s += (double)x[e] * (double)x[e];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      rho = __double2float_rn(sqrt(s));
    }
  }

  // fast path: fp32 butterfly, decided where no threshold is within 2^-15 rho
  float u[E];
#pragma unroll
  for (int e = 0; e < E; ++e) u[e] = ((sbits >> e) & 1u) ? -x[e] : x[e];
  warp_fwht<float, E>(u, lane);
  float T[15];
#pragma unroll
  for (int k = 0; k < 15; ++k) T[k] = rho * prm.tq[k];
  const float M = rho * 0x1p-15f;
  bool near = !(rho >= 1e-30f && rho <= 1e36f) || prm.exact_all;
  // thresholds are farther apart than 2M, so only the two bracketing ones can
  // lie within M of u
  uint32_t word = 0, nearmask = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    float lo, hi;
    const int z = bracket15(u[e], T, lo, hi);
    if (u[e] - lo <= M || hi - u[e] <= M) nearmask |= 1u << e;
    word |= (uint32_t)z << (4 * e);
  }
  near = near || (nearmask != 0);
  if (__any_sync(0xffffffffu, near)) {
    // exact path: fp64 butterfly; an element within M of a threshold compares
    // against the contract's threshold products T_k = fp64(fp64(sqrt(D) rho)
    // t_k) for its two bracketing thresholds (all 15 when the norm is outside
    // the fast path's range)
    double ud[E];
#pragma unroll
    for (int e = 0; e < E; ++e) ud[e] = ((sbits >> e) & 1u) ? -(double)x[e] : (double)x[e];
    warp_fwht<double, E>(ud, lane);
    const double r = (double)rho * sqrt((double)D);
    const bool all = !(rho >= 1e-30f && rho <= 1e36f) || prm.exact_all;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (all || ((nearmask >> e) & 1u)) {
        const int zf = (word >> (4 * e)) & 0xF;
        const int k0 = all ? 0 : max(zf - 1, 0), k1 = all ? 15 : min(zf + 1, 15);
        int z = k0;
        for (int k = k0; k < k1; ++k) z += (ud[e] > r * (double)prm.t[k]) ? 1 : 0;
        word = (word & ~(0xFu << (4 * e))) | ((uint32_t)z << (4 * e));
      }
    }
  }

  rho_out = rho;
  return word;
}

// Store a lane's indices and (lane 0) the fp16 norm into slot `vrow` (head *
// P + slot) of a page record.
template <int D>
__device__ __forceinline__ void tq4_store(uint8_t* pg, int64_t codes_region, int64_t norm_region,
                                          int kind, int64_t vrow, int lane, uint32_t word,
                                          float rho) {
  constexpr int E = D / 32;
  uint8_t* dst = pg + kind * codes_region + vrow * (D / 2);
  if constexpr (E == 8)
    reinterpret_cast<uint32_t*>(dst)[lane] = word;
  else
    reinterpret_cast<uint16_t*>(dst)[lane] = (uint16_t)word;
  if (lane == 0) {
    const __half h = __float2half_rn(fminf(rho, 65504.f));
    *reinterpret_cast<uint16_t*>(pg + 2 * codes_region + kind * norm_region + vrow * 2) =
        __half_as_ushort(h);
  }
}

}  // namespace jfkv
