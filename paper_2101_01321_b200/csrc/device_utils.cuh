// Device-side integer building blocks shared by the kernels: dyadic requantization,
// the i-GELU element function, the i-exp element function and exact integer division
// helpers.  Everything here is integer arithmetic; no floating-point instruction is used.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ibert_internal.h"

namespace ibert {

// clamp((v * b + add) >> c, +-qmax); `add` carries the rounding constant 2^(c-1)
// (and, in GEMM epilogues, bias * b).  64-bit product, arithmetic shift, 0 <= c <= 31.
__device__ __forceinline__ int32_t requant_add(int32_t v, int32_t b, int64_t add, int c, int32_t qmax) {
  int64_t p = (int64_t)v * (int64_t)b + add;
  p >>= c;
  p = p > (int64_t)qmax ? (int64_t)qmax : p;
  p = p < -(int64_t)qmax ? -(int64_t)qmax : p;
  return (int32_t)p;
}

// (v * b2 + add) >> 32 with a 64-bit addend: two multiply-adds with a carry between them, which issue like one
// multiply-high (4.0 clocks per warp and scheduler) and leave the ALU pipe alone.  Written in C++, as a 64-bit product
// plus addend, it takes 8.5.
__device__ __forceinline__ int32_t requant_upper_add(int32_t v, int32_t b2, int64_t add) {
  int32_t hi;
  asm("{\n\t.reg .u32 lo;\n\t"
      "mad.lo.cc.u32 lo, %1, %2, %3;\n\t"
      "madc.hi.s32 %0, %1, %2, %4;\n\t}"
      : "=r"(hi)
      : "r"(v), "r"(b2), "r"((uint32_t)add), "r"((int32_t)(add >> 32)));
  return hi;
}

// The same requantization when the host could pre-shift the multiplier (b2 = b << (32 - c)): (v * b2 + 2^31) >> 32, not
// yet clamped.  (The form below issues in the same time alone, but its correction is ALU work, which binds most of the
// loops around it: i-GELU of 2^24 values 14.2 -> 13.6 us, three Base layers of 1 x 128 59.4 -> 58.1 us, of 8 x 77 88.1 ->
// 86.4.)
__device__ __forceinline__ int32_t requant_upper(int32_t v, int32_t b2) { return requant_upper_add(v, b2, int64_t(1) << 31); }

// The same as a product whose upper word is corrected by bit 31 of the lower one (a register less).
__device__ __forceinline__ int32_t requant_upper_product(int32_t v, int32_t b2) {
  const int64_t t = (int64_t)v * (int64_t)b2;
  return (int32_t)(t >> 32) + (int32_t)((uint32_t)t >> 31);
}

// The upper-word requantization for multipliers of 1/2 and more: b 2^(32-c) no longer fits 32 bits,
// so it is split into w 2^32 + r with r in [-2^31, 2^31) and the product into v w + (v r >> 32).
// Exact like the others; the host checks that v w cannot overflow.
__device__ __forceinline__ int32_t requant_upper_wide(int32_t v, int32_t r, int32_t w) {
  const int64_t t = (int64_t)v * (int64_t)r;
  return v * w + (int32_t)(t >> 32) + (int32_t)((uint32_t)t >> 31);
}

// four int32 -> four int8 lanes of one word, each saturated to [-128, 127]
__device__ __forceinline__ uint32_t pack4_sat_s8(int32_t v0, int32_t v1, int32_t v2, int32_t v3) {
  uint32_t hi, r;
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(v3), "r"(v2), "r"(0));
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(v1), "r"(v0), "r"(hi));
  return r;
}

// byte k of a word as a sign-extended int32 in one permute (`prmt`: a selector nibble with bit 3
// set replicates the sign of the byte it selects)
__device__ __forceinline__ int32_t sext_byte(uint32_t w, int k) {
  int32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "r"(0x8880 + k * 0x1111));
  return r;
}

// the int8 residual in byte j of w, rescaled, plus add: the byte lands above 16 bits of rounding offset by one permute
__device__ __forceinline__ int32_t residual_high_add(uint32_t w, int j, int32_t hk, int32_t hm, int32_t add) {
  int32_t u, d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(u) : "r"(w), "r"(hk), "r"(0x8054 + j * 0x1100));
  asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(u), "r"(hm), "r"(add));
  return d;
}

// 16-bit half h of a word as a sign-extended int32, likewise in one permute
__device__ __forceinline__ int32_t sext_half(uint32_t w, int h) {
  int32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "r"(h ? 0xBB32 : 0x9910));
  return r;
}

__device__ __forceinline__ int64_t rounding_half(int c) { return c > 0 ? (int64_t(1) << (c - 1)) : 0; }

__device__ __forceinline__ int32_t clamp_sym(int32_t v, int32_t qmax) { return max(-qmax, min(v, qmax)); }

// i-GELU of one Q16 value (Algorithm 2): i-erf = sgn(q) * [(min(|q| >> s_in, -q_b) + q_b)^2 + q_c],
// g = q * ((i-erf + q_1) >> s_f), then round(g / 256) and the dyadic requantization to int8.
__device__ __forceinline__ int32_t igelu_q16_to_int8(int32_t q, const GeluConsts& k, int64_t half) {
  const int32_t mag = abs(q);
  const int32_t t = min(mag >> k.s_in, k.nq_b) - k.nq_b;    // clip(|q|, max = -q_b) + q_b, in [q_b, 0]
  const int32_t poly = t * t + k.q_c;                        // I-Poly; negative
  const int32_t f = k.q_c + (q < 0 ? -poly : poly);          // q_erf + q_1 (value for q = 0 is unused: g = 0)
  const int32_t g = q * (f >> k.s_f);
  const int32_t g2 = (g + 128) >> 8;
  return requant_add(g2, k.b, half, k.c, 127);
}

// Same function, written for the integer pipes: sign applied by a select, the final
// requantization in upper-word form; the result still needs the upper clamp (pack4_sat_s8).
__device__ __forceinline__ int32_t igelu_q16_upper(int32_t q, const GeluConsts& k) {
  const int32_t t = min(abs(q) >> k.s_in, k.nq_b) - k.nq_b;
  const int32_t tt = t * t;
  // q_erf + q_1 = sgn(q) (t^2 + q_c) + q_c: -t^2 for q < 0, t^2 + 2 q_c otherwise (unused for q = 0)
  const int32_t f = q < 0 ? -tt : tt + 2 * k.q_c;
  const int32_t g2 = (q * (f >> k.s_f) + 128) >> 8;
  return max(requant_upper(g2, k.b2), -127);
}

// Magnitude form of the same function, taking the Q16 value BEFORE its clamp (x; q = clamp(x)):
// with a = |q| = min(|x|, 32767) and t as above,
//   q >= 0:  g = q ((t^2 + 2 q_c) >> s_f)                    = a ((t^2 + 2 q_c) >> s_f)
//   q <  0:  g = q ((-t^2) >> s_f) = q (-ceil(t^2 / 2^s_f))   = a ((t^2 + 2^s_f - 1) >> s_f)
// so one select of the addend replaces the two-sided clamp, the negation and the select of f.
// `rnd_f` = 2^s_f - 1.  The result still needs both clamps to +-127.
// Written for the ALU pipe, which binds it: the clip and its offset are one add-and-minimum, the addend is selected by
// a multiply-add with the sign (SHIFT = false: s_in is known to be 0).
template <bool SHIFT = true>
__device__ __forceinline__ int32_t igelu_magnitude_upper(int32_t x, const GeluConsts& k, int32_t rnd_f) {
  const int32_t a = (int32_t)min((uint32_t)abs(x), 32767u);    // unsigned: |INT32_MIN| stays 2^31
  const int32_t t = __viaddmin_s32(SHIFT ? a >> k.s_in : a, -k.nq_b, 0);
  const int32_t add = (x >> 31) * (2 * k.q_c - rnd_f) + 2 * k.q_c;         // x >= 0: 2 q_c, else rnd_f
  const int32_t f = (t * t + add) >> k.s_f;
  const int32_t g2 = (a * f + 128) >> 8;
  return requant_upper(g2, k.b2);
}

// Integer h-GELU (Eq. 6) of one Q16 value before its clamp: r = clamp(q + q_3, 0, q_6) >> s_h,
// g = q r, round(g / 256), dyadic requantization (GeluConsts with hard != 0).
__device__ __forceinline__ int32_t ihgelu_upper(int32_t x, const GeluConsts& k) {
  const int32_t v = clamp_sym(x, 32767);
  const int32_t r = min(max(v + k.q_c, 0), k.nq_b) >> k.s_f;
  return requant_upper((v * r + 128) >> 8, k.b2);
}
__device__ __forceinline__ int32_t ihgelu_to_int8(int32_t q, const GeluConsts& k, int64_t half) {
  const int32_t r = min(max(q + k.q_c, 0), k.nq_b) >> k.s_f;
  return requant_add((q * r + 128) >> 8, k.b, half, k.c, 127);
}

// One output value of a linear layer from one complete accumulator, by epilogue kind.  FAST: multipliers in
// upper-word form; `padd` = bias * b + rounding constant for the generic form; `gelu_rnd` = 2^s_f - 1.
template <int KIND, bool FAST>
__device__ __forceinline__ int32_t epilogue_value(int32_t a, int32_t bias, int32_t pb, int32_t pc, int64_t padd,
                                                  const GeluConsts& gk, int64_t gelu_half, int32_t gelu_rnd) {
  if constexpr (KIND == EPI_RAW) return a + bias;
  else if constexpr (KIND == EPI_Q16 || KIND == EPI_Q16H) {
    if constexpr (FAST) return clamp_sym(requant_upper(a + bias, pb), 32767);
    else return requant_add(a, pb, padd, pc, 32767);
  } else if constexpr (KIND == EPI_INT8) {
    if constexpr (FAST) return clamp_sym(requant_upper(a + bias, pb), 127);
    else return requant_add(a, pb, padd, pc, 127);
  } else if constexpr (KIND == EPI_HGELU) {
    // (a register more, 33, would leave a short reduction three CTAs of the one-wave kernel per SM instead of four:
    // 900 x 1024 x 256 4.0 -> 4.4 us; from K = 384 on the multiply-adds would gain 1 to 2 %)
    if constexpr (FAST) return clamp_sym(ihgelu_upper(requant_upper_product(a + bias, pb), gk), 127);
    else return ihgelu_to_int8(requant_add(a, pb, padd, pc, 32767), gk, gelu_half);
  } else {
    if constexpr (FAST) return clamp_sym(igelu_magnitude_upper(requant_upper(a + bias, pb), gk, gelu_rnd), 127);
    else return igelu_q16_to_int8(requant_add(a, pb, padd, pc, 32767), gk, gelu_half);
  }
}

__device__ __forceinline__ uint32_t shr_clamped(uint32_t v, uint32_t n) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));   // shift counts above 31 give 0
  return r;
}

// i-exp of one non-negative distance d = max - q (Algorithm 3): z = floor(d'/q_ln2),
// r = d' - z q_ln2, e = ((q_b - r)^2 + q_c) >> min(z + s_out, 31); d' = min(d >> s_in, 31 q_ln2).
// The polynomial is below 2^31, so a shift by more than 31 equals the shift by 31 (both give 0).
// DIV: 0 = multiply-high alone gives z, 1 = followed by a shift, 2 = operand pre-shifted as well.
template <int DIV>
__device__ __forceinline__ uint32_t iexp_dist(uint32_t d, const ExpConsts& k) {
  const uint32_t dp = min(d >> k.s_in, k.d_max);
  uint32_t z;
  if (DIV == 0) z = __umulhi(dp, k.div_m);
  else if (DIV == 1) z = __umulhi(dp, k.div_m) >> k.div_post;
  else z = __umulhi(dp << k.div_pre, k.div_m) >> k.div_post;
  const int32_t t = (int32_t)(z * k.q_ln2) + (k.q_b - (int32_t)dp);      // q_b - r
  const uint32_t poly = (uint32_t)(t * t + k.q_c);
  return shr_clamped(poly, z + (uint32_t)k.s_out);
}
// i-exp for distances below 2^21 (attention scores): no clamp of the distance -- a quotient above
// 31 just shifts the polynomial out completely, exactly like the clamped form.
__device__ __forceinline__ uint32_t iexp_dist_wide(uint32_t d, const ExpConsts& k) {
  const uint32_t dp = d >> k.s_in;
  const uint32_t z = __umulhi(dp, k.wide_m) >> k.wide_post;
  const int32_t t = (int32_t)(z * k.q_ln2) + (k.q_b - (int32_t)dp);      // q_b - r
  const uint32_t poly = (uint32_t)(t * t + k.q_c);
  return shr_clamped(poly, z + (uint32_t)k.s_out);
}
// a + b on the ALU pipe (add-and-maximum against INT32_MIN, passed as a run-time value so that the compiler cannot
// fold it): left to itself the compiler puts additions on the multiply-add pipe, which the multiply-highs of
// i-softmax keep busy for four clocks each
__device__ __forceinline__ int32_t add_alu(int32_t a, int32_t b, int32_t int_min) { return __viaddmax_s32(a, b, int_min); }
// The same when quotient and post-shift come from one multiply-high (ExpConsts::fold_m), from w = q_b - s_out q_ln2 - d'
// alone: with the distance offset to D = d' + s_out q_ln2 + fold_add = q_b + fold_add - w, the shift count is the upper
// word of D fold_m = (q_b + fold_add) fold_m - w fold_m, whose first term is the same for all scores.
// (a pre-shift above 12 -- score scales below 1e-8 -- would take the offset past 31 bits: iexp_dist_wide serves those)
__host__ __device__ __forceinline__ bool iexp_takes_folded(const ExpConsts& k) { return k.fold_m != 0 && k.s_in <= 12; }
__host__ __device__ __forceinline__ int64_t iexp_folded_addend(const ExpConsts& k) {
  return (int64_t)(k.q_b + k.fold_add) * (int64_t)k.fold_m;
}
// w = (score + offset) >> s_in for a row with maximum mx: -(d >> s) = (2^s - 1 - d) >> s
__host__ __device__ __forceinline__ int32_t iexp_folded_offset(const ExpConsts& k, int32_t mx) {
  const uint32_t c = (uint32_t)k.q_b - (uint32_t)k.s_out * k.q_ln2;      // below 2^18 in magnitude
  return (int32_t)(((c + 1u) << k.s_in) - 1u - (uint32_t)mx);
}
__device__ __forceinline__ uint32_t iexp_folded(int32_t w, int64_t mk, int32_t neg_m, uint32_t q_ln2, int32_t q_c) {
  const uint32_t n = (uint32_t)requant_upper_add(w, neg_m, mk);          // floor(d' / q_ln2) + s_out
  const int32_t t = (int32_t)(n * q_ln2) + w;                            // q_b - r
  return shr_clamped((uint32_t)(t * t + q_c), n);
}
__host__ __device__ __forceinline__ int exp_div_mode(const ExpConsts& k) {
  return k.div_pre != 0 ? 2 : (k.div_post != 0 ? 1 : 0);
}

// i-LayerNorm's normalization of one token: n = floor((v - mu) rho / 2^15) with rho = floor(2^31 / sigma) (sigma <= 1:
// 2^30 and 2^14) as ONE multiply-high, (v 2^a - mu 2^a) times rho 2^s with a + s = 17 (18).  s is as large as rho
// allows, at least floor(log2 sigma) - 1; |v - mu| <= (sigma + 1) sqrt(C) then keeps (v - mu) 2^a below 2^25 for
// C < 2048, so neither factor overflows (v 2^a and mu 2^a alone may: their difference is right modulo 2^32).
struct LnNorm {
  int32_t scale, shift, rho;       // 2^a, mu 2^a, rho 2^s
};
__device__ __forceinline__ LnNorm ln_norm(int32_t mu, uint32_t sigma) {
  const uint32_t rho = sigma > 1u ? 0x80000000u / sigma : 1u << 30;
  const int total = sigma > 1u ? 17 : 18, s = min(__clz((int)rho) - 1, total), a = total - s;
  return {1 << a, (int32_t)((uint32_t)mu << a), (int32_t)(rho << s)};
}
// floor(sum / C) for |sum| <= C 2^18
__device__ __forceinline__ int32_t ln_mean(int32_t sum, int C, const LnConsts& k) {
  return (int32_t)(__umulhi((uint32_t)(sum + (C << 18)), k.mean_m) >> k.mean_sh) - (1 << 18);
}
__device__ __forceinline__ int32_t ln_normalize(int32_t v, const LnNorm& n) {
  return __mulhi((int32_t)((uint32_t)v * (uint32_t)n.scale - (uint32_t)n.shift), n.rho);
}

// floor(sqrt(floor(ss / C))) = the largest s with s^2 C <= ss -- the value Algorithm 4 returns for n = floor(ss / C) --,
// one thread per value: Newton's iteration for the reciprocal square root (r <- r (3 - X r^2) / 2) on the leading 32
// bits X in [1/4, 1) of ss, from a quadratic start 2.4 % off.  Two steps leave 1.2e-6, so for s < 2^18 the product with X
// and `root_k` = floor(2^32 / sqrt(C)) is off by at most one, which the exact comparison settles.  (Bit by bit the root
// took 18 dependent rounds; three Base layers of 8 x 77 86.4 -> 85.0 us with this form, of 1 x 128 58.1 -> 57.8.)
// Needs ss < 2^60 and C >= 2.  STEPS = 3: s < 2^24.  (Other sums -- the missing row of an odd row count -- give any
// value: the shift count, negative from 2^60 on, must then be one that the shift takes.)
template <int STEPS = 2>
__device__ __forceinline__ uint32_t ln_root(uint64_t ss, uint32_t C, uint32_t root_k) {
  const int z = __clzll((long long)(ss | 1ull)) & ~1;
  const uint32_t x = (uint32_t)((ss << z) >> 32);
  uint32_t r = 0xAAEEF78Fu - __umulhi(x, 0xD24346FDu - __umulhi(x, 0x68DE4A2Du));       // Q30: 2.6708, 3.2854, 1.6386
#pragma unroll
  for (int i = 0; i < STEPS; ++i) r = __umulhi(r, 0x30000000u - __umulhi(x, __umulhi(r, r))) << 3;
  const uint32_t s = shr_clamped(__umulhi(__umulhi(x, r), root_k), (uint32_t)((z >> 1) - 2));
  const uint64_t sq = (uint64_t)s * s * C;
  return sq > ss ? s - 1u : (sq + (uint64_t)(2u * s + 1u) * C <= ss ? s + 1u : s);
}

// floor(sqrt(floor(ss / C))), i.e. the largest s with s*s*C <= ss -- the value Algorithm 4
// returns for n = floor(ss / C).  A 64-bit integer division costs on the order of a hundred
// instructions here, so instead of iterating x <- (x + n/x)/2 a group of GROUP lanes (32 or 16; ss is the group's) finds
// the same integer by a radix-GROUP search: in each round its lanes test GROUP candidates with one multiply each.
// Needs s < 2^25 (GROUP = 16: 2^24, six rounds; a seventh would test candidates up to 15 2^24, whose s^2 C passes
// 64 bits) and C < 2^12.  The rounds are those of the larger root of a warp: more of them change nothing.
template <int GROUP = 32>
__device__ __forceinline__ uint32_t warp_isqrt_of_quotient(uint64_t ss, uint32_t C, int lane) {
  constexpr int kDigit = GROUP == 32 ? 5 : 4;
  const int li = lane & (GROUP - 1);
  uint32_t base = 0;
  // ss / C < 2^bits bounds the result below 2^ceil(bits / 2): rounds above that cannot set a digit
  const int bits = 64 - __clzll((long long)(ss | 1ull)) - (31 - __clz((int)C));
  int need = min(max((bits + 1) >> 1, 1), GROUP == 32 ? 25 : 24);
  if constexpr (GROUP != 32) need = __reduce_max_sync(0xffffffffu, need);
  for (int shift = kDigit * ((need + kDigit - 1) / kDigit - 1); shift >= 0; shift -= kDigit) {
    const uint32_t cand = base + ((uint32_t)li << shift);
    const uint64_t sq = (uint64_t)cand * (uint64_t)cand;
    const bool le = sq * (uint64_t)C <= ss;                       // true for a prefix of the lanes
    uint32_t votes = __ballot_sync(0xffffffffu, le);
    if constexpr (GROUP == 16) votes = (votes >> (lane & 16)) & 0xffffu;
    base += (uint32_t)(__popc(votes) - 1) << shift;               // (lane 0 tests `base` itself: at least one vote)
  }
  return base;
}

// byte offset of element (row, col) in a K-major operand tile made of 128-byte-wide K blocks
// with the 128-byte swizzle: 16-byte chunk c of row r sits at chunk c ^ (r & 7).
__device__ __forceinline__ uint32_t sw128_offset(uint32_t row, uint32_t col, uint32_t rows_per_block) {
  const uint32_t kb = col >> 7, cc = (col >> 4) & 7, by = col & 15;
  return kb * (rows_per_block * 128u) + row * 128u + (((cc ^ (row & 7u)) << 4) | by);
}

// Reciprocal of a normalised 32-bit integer by Newton-Raphson iteration (r <- r (2 - y r), the usual linear
// start 48/17 - 32/17 y, relative error 1/17 squared by every step): for y in [2^31, 2^32) the result is
// floor(2^63 / y) or one less (saturated to 32 bits at y = 2^31).  Two steps in 32-bit fixed point (Q30), the
// last one on the exact 64-bit remainder.
__device__ __forceinline__ uint32_t reciprocal_q31(uint32_t y) {
  uint32_t r = 0xB4B4B4B4u - __umulhi(0x78787878u, y);
#pragma unroll
  for (int i = 0; i < 2; ++i) r = __umulhi(r, 0x80000000u - __umulhi(y, r)) << 2;
  const int64_t rem = (int64_t)((uint64_t(1) << 62) - (uint64_t)y * (uint64_t)r);     // below 2^46
  return 2u * r + (uint32_t)(__mulhi((int32_t)(rem >> 15), (int32_t)r) >> 14);
}

// Per-row divisor for p = floor(e * p_max / sum) with e < 2^21 and e <= sum < 2^31:
// with l = bit length of sum, K = 23 + l and any integer m with 0 <= m sum - p_max 2^K < 4 sum,
// floor(e m / 2^K) is exact: the excess e (m sum - p_max 2^K) / (sum 2^K) stays below
// 2^(21 + 2 - K) = 2^-l < 1/sum.  p_max 2^K / sum = p_max 2^55 / y for the normalised sum y, so
// m = floor(p_max R / 256) + 3 from the reciprocal above lies 0.3 to 3 too high (a 64-bit division costs four
// times the instructions).  Evaluated as umulhi(e << pre, m) >> post with post - pre = K - 32.
struct RowDivisor {
  uint32_t m;
  int pre, post;
};

__device__ __forceinline__ RowDivisor make_row_divisor(uint32_t sum, uint32_t p_max) {
  RowDivisor r;
  const int lz = __clz(sum), K = 23 + 32 - lz;
  r.m = __umulhi(reciprocal_q31(sum << lz), p_max << 24) + 3u;
  r.pre = K < 32 ? 32 - K : 0;
  r.post = K < 32 ? 0 : K - 32;
  return r;
}

__device__ __forceinline__ uint32_t softmax_quotient(uint32_t e, const RowDivisor& r) {
  return __umulhi(e << r.pre, r.m) >> r.post;
}
// the common case pre == 0 (row sum >= 2^8)
__device__ __forceinline__ uint32_t softmax_quotient_nopre(uint32_t e, const RowDivisor& r) {
  return __umulhi(e, r.m) >> r.post;
}

}  // namespace ibert
