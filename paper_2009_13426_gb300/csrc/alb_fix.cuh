// 64-bit fixed-point arithmetic of the FP32 form's residual refinement.
//
// The residual of an equilibrium solve is a difference of sums whose terms
// agree to about 1e-7, wanted to 1e-12: FP32 cannot form it, and the FP64
// pipe (2 operations per clock and SM on GB300) bounds a step that forms it
// there. Populations per unit density lie in (0, 1), so they are held here as
// 64-bit integers in units of 2^-63 (Q63): a sum costs two integer
// instructions, is exact, and may wrap modulo 2^64 on the way, since only the
// final residual has to fit. All of it issues on the integer and FP32 pipes.
//
//   exponent   y = s / ln 2 in octaves, Q25 in 32 bits (|y| < 64): the
//              multipliers are rounded to that grid once (5e-9 to 1e-8, below
//              the FP32 rounding of the multipliers they come from), and every
//              y_i = base + lambda . P(xi_i) is then exact integer arithmetic,
//              so the populations belong to one exponential family.
//   population p = 2^-y: Q63 table of 2^-(j/512), the rest of the exponent by
//              its degree-3 polynomial in FP32, rounded to 2^-32 of the table
//              value; for 0 <= y < 31 (FIX_OCTAVES) within 5e-10 relative
//              (1.2e-10 rounding, 1e-10 polynomial, the truncation to 2^-63
//              at most 2.4e-10). Colder states take the FP64 refinement.
//
// The functions also compile as plain host C++, so the same code is checked on
// the CPU against 64-bit arithmetic.
#pragma once

#include <math.h>

#include "alb_cvt.cuh"
#include "exp_table.h"

namespace alb {

constexpr int FIX_BITS = 25;          // fraction bits of the exponent
constexpr int FIX_OCTAVES = 31;       // accepted exponents: 0 <= y < 31 octaves
constexpr uint32_t FIX_Y_END = (uint32_t)FIX_OCTAVES << FIX_BITS;
// a multiplier in units of 2^-25 octave
constexpr float FIX_SCALE = 48408812.0f;  // 2^25 / ln 2
// Exponents above this magnitude (44 < 64 ln 2) could wrap in 32 bits.
constexpr float FIX_S_MAX = 44.0f;
// Largest step taken multiplicatively (the factor's polynomial: 3e-14).
constexpr float FIX_STEP_MAX = 9e-4f;
static_assert(FIXT_BITS == 9, "the index and remainder below assume 512 table entries");

// Q63 population 2^-y of an exponent y (Q25 octaves) with 0 <= y < 31; other
// exponents give some value (the caller rejects them).
// y = j/512 - r/2^25 octaves with j the next table index and 0 <= r < 2^16,
// so that 2^-y = 2^-(j/512) 2^(r/2^25), 2^(r/2^25) - 1 in [0, 1.36e-3).
ALB_CVT_FN uint64_t fix_exp(uint32_t y, const uint64_t* tab) {
  const uint32_t t = y + 0xffffu;
  const uint64_t T = tab[(t >> 16) & 511u];
  const uint32_t n = t >> FIX_BITS;
  // r as a float without a conversion instruction: 2^23 + r has r in its low bits
  const float r = cvt_f32_of_bits((~t & 0xffffu) | 0x4b000000u) - 8388608.0f;
  // 2^(r/2^25) - 1 = x + x^2/2 + x^3/6, x = r ln2 / 2^25, in units of 2^-32
  // (below 2^23); added to 2^23 it is rounded to an integer in the low bits
  const float a1 = 88.722839111673f;          // 2^7 ln 2
  const float a2 = 9.163913992275265e-7f;     // 2^-18 (ln 2)^2 / 2
  const float a3 = 6.310086594660513e-15f;    // 2^-43 (ln 2)^3 / 6
  const float q = fmaf(r, fmaf(r, fmaf(r, a3, a2), a1), 8388608.0f);
  const uint32_t qi = cvt_bits_f32(q) - 0x4b000000u;
  const uint64_t P = T + (uint64_t)(uint32_t)(T >> 32) * qi;
#ifdef __CUDA_ARCH__
  const uint32_t lo = __funnelshift_r((uint32_t)P, (uint32_t)(P >> 32), n);
  const uint32_t hi = (uint32_t)(P >> 32) >> (n & 31u);
  return ((uint64_t)hi << 32) | lo;
#else
  return P >> (n & 31u);
#endif
}

// Scale of the factors of one multiplicative update whose exponent changes are
// all at most `bound` (<= FIX_STEP_MAX) in magnitude: e = exp(-d) - 1 in units of
// 2^-(32 + k), k as large as 31 bits of magnitude allow, so that e keeps its FP32
// precision and a sequence of shrinking steps converges.
struct FixStep {
  float c1, c2, c3;  // e 2^(32 + k) = c1 d + c2 d^2 + c3 d^3
  uint32_t k;
};
ALB_CVT_FN FixStep fix_step(float bound) {
  const int eb = (int)(cvt_bits_f32(bound) >> 23) - 127;  // bound < 2^(eb + 1)
  int k = -3 - eb;
  k = k < 0 ? 0 : (k > 31 ? 31 : k);
  const float s = cvt_f32_of_bits((uint32_t)(127 + 32 + k) << 23);  // 2^(32 + k)
  return FixStep{-s, 0.5f * s, -0.16666667f * s, (uint32_t)k};
}

// Q63 population P times exp(-d) (the factor by a degree-3 polynomial in FP32).
ALB_CVT_FN uint64_t fix_scale(uint64_t P, float d, const FixStep& c) {
  // e 2^(32 + k), below 2^31 in magnitude, rounded to an integer
  const float q = d * fmaf(d, fmaf(d, c.c3, c.c2), c.c1);
#ifdef __CUDA_ARCH__
  const int e = __float2int_rn(q);
#else
  const int e = (int)lrintf(q);
#endif
  const uint32_t lo = (uint32_t)P, hi = (uint32_t)(P >> 32);
#ifdef __CUDA_ARCH__
  const uint32_t w = __umulhi(lo, (uint32_t)e);
#else
  const uint32_t w = (uint32_t)(((uint64_t)lo * (uint32_t)e) >> 32);
#endif
  // (lo * e) >> 32 for signed e
  const int32_t wl = (int32_t)(w - (lo & (uint32_t)(e >> 31)));
  const int64_t t = (int64_t)(int32_t)hi * (int64_t)e + (int64_t)wl;
#ifdef __CUDA_ARCH__
  const uint32_t th = (uint32_t)((uint64_t)t >> 32);
  const uint32_t sl = __funnelshift_r((uint32_t)t, th, c.k);
  return P + (((uint64_t)(uint32_t)((int32_t)th >> c.k) << 32) | sl);
#else
  return P + (uint64_t)(t >> c.k);
#endif
}

// A double in Q63, modulo 2^64 (bits below 2^-63 are dropped).
ALB_CVT_FN uint64_t fix_of_f64(double v) {
  uint32_t h, l;
  cvt_bits_f64(v, &h, &l);
  const int s = (int)((h >> 20) & 0x7ffu) - 1012;  // left shift of the 53-bit significand
  const uint64_t m = ((uint64_t)((h & 0xfffffu) | 0x100000u) << 32) | l;
  const uint64_t u = s >= 0 ? (s < 64 ? m << (s & 63) : 0u) : (s > -64 ? m >> (-s & 63) : 0u);
  return (h & 0x80000000u) ? 0u - u : u;
}

// A Q63 residual (|g| < 1, two's complement) in FP32: absolute error below
// 2^-55 for residuals that matter, relative 2^-24 for larger ones.
ALB_CVT_FN float fix_residual_f32(uint64_t g) {
  const int hi = (int)(uint32_t)(g >> 32);
  return fmaf((float)hi, 4.656612873077393e-10f,
                 (float)(uint32_t)g * 1.0842021724855044e-19f);  // 2^-31, 2^-63
}

// A Q63 population in FP32, rounded to nearest (0 < P).
ALB_CVT_FN float fix_to_f32(uint64_t P) {
  const uint32_t hi = (uint32_t)(P >> 32), lo = (uint32_t)P;
  const int lz = cvt_clz(hi);  // 32 if the high word is empty
#ifdef __CUDA_ARCH__
  const uint32_t top = __funnelshift_lc(lo, hi, lz);
#else
  const uint32_t top = lz == 0 ? hi : (lz == 32 ? lo : (hi << lz) | (lo >> (32 - lz)));
#endif
  const uint32_t rest = lz < 32 ? lo << (lz & 31) : 0u;
  // the dropped bits stay as a sticky bit below the 24 kept ones
  const uint32_t b = cvt_bits_f32((float)(top | (rest != 0u ? 1u : 0u)));
  return cvt_f32_of_bits(P == 0u ? 0u : b - ((uint32_t)(31 + lz) << 23));
}

// A Q63 population in FP64 (exact to 53 bits).
ALB_CVT_FN double fix_to_f64(uint64_t P) {
  return (double)P * 1.0842021724855044e-19;  // 2^-63
}

}  // namespace alb
