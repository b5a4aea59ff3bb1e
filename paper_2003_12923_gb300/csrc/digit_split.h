// Digit split of a float64 element and the integer join of the level sums (digits.cu, narrow.cu).
#pragma once
#include <cstdint>

namespace esmp2 {

// V 2^e as float64, V rounded to 53 bits; integer operations only
__device__ __forceinline__ double scale_i64(long long V, int e) {
  if (V == 0) return 0.0;
  unsigned long long u = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
  const int lz = __clzll((long long)u);
  u <<= lz;
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1);   // in [2^52, 2^53]
  const int eb = 1023 + 63 - lz + e;                          // biased exponent of the leading bit
  unsigned long long bits = ((unsigned long long)(eb - 1) << 52) + m;
  if (eb <= 0) bits = 0;
  if (eb >= 2047) bits = 0x7FF0000000000000ull;
  if (V < 0) bits |= 0x8000000000000000ull;
  return __longlong_as_double((long long)bits);
}

// A joined sum that has no value (a NaN or infinity among the operands); sums stay above -2^63.
constexpr long long kNoValue = (long long)(1ull << 63);
__device__ __forceinline__ double scale_or_nan(long long V, int e) {
  return V == kNoValue ? __longlong_as_double(0x7FF8000000000000ll) : scale_i64(V, e);
}

// Digits of one element, W = 6 bits each (7 where few products are summed: bf16 holds them exactly).  The
// magnitude is split, U = |Z| + sum_k 32 64^k over the lower P - 1 digits, so
// that digit p >= 2 of |Z| is field - 32 and digit 1 the rest (64 and 128 for W = 7); the sign goes to every digit, so -v has
// the negated digits and its products (with the dropped pairs of low weight) are exactly the
// negated ones.  |Z| by shifts of the significand (round half up): float64 arithmetic would cost two
// operations of its slow pipe.
// With one digit range the digits would have the mean -1/2 sign(v), and the pairs left out would shift
// every product the same way relative to v (No=30 Nv=400, eight levels: 5e-14 of E2, 1.4e-15 with both ranges): half of the elements, by the
// parity of their significand, take digits in [-31, 32] (field - 31) instead of [-32, 31].
__device__ __forceinline__ uint32_t digit_range(double v) {   // 0 or 1
  return (uint32_t)__popc((uint32_t)__double2loint(v) ^ ((uint32_t)__double2hiint(v) & 0xFFFFFu)) & 1u;
}
template <int P, int W = 6>
__device__ __forceinline__ long long digit_word(double v, int es) {
  constexpr long long ones = ((1ll << (W * (P - 1))) - 1) / ((1 << W) - 1);   // sum_k 2^(W k)
  const long long bias = ones * (1 << (W - 1)) - (digit_range(v) ? ones : 0ll);
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const int ef = (int)(u >> 52) & 0x7FF;
  const int sh = 1075 - ef + es - W * P;   // >= 54 - W P for every finite |v| < 2^(es - 1)
  unsigned long long m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  if (sh > 0) m = sh < 55 && ef != 0 ? ((m >> (sh - 1)) + 1) >> 1 : 0;
  else if (W * P > 54) m <<= min(-sh, W * P - 54);
  return (long long)m + bias;
}
__device__ __forceinline__ bool non_finite(double v) { return (~(uint32_t)__double2hiint(v) & 0x7FF00000u) == 0; }
// The signs of two elements as bf16 factors +-1.0, packed.
__device__ __forceinline__ uint32_t sign_pair(double v0, double v1) {
  return (((uint32_t)__double2hiint(v0) >> 16) & 0x8000u) | ((uint32_t)__double2hiint(v1) & 0x80000000u) | 0x3F803F80u;
}
// The same with a NaN factor for a NaN or infinity: all its digits become NaN, the tensor cores carry it
// into every level sum of its row (or, in the right factor, column), and no_value finds it there, so that
// such an element spoils the results that depend on it and never passes for a number.  (It takes no
// part in the scale of its slice, k_slice_exp: the other rows are what they would be without it.)
__device__ __forceinline__ uint32_t sign_pair_nan(double v0, double v1) {
  uint32_t s = sign_pair(v0, v1);
  if (non_finite(v0)) s |= 0x7FC0u;
  if (non_finite(v1)) s |= 0x7FC00000u;
  return s;
}
__device__ __forceinline__ bool no_value(float leading_sum) { return leading_sum != leading_sum; }
// The ranges of two elements, packed as the difference of their constants in digit_pair.
__device__ __forceinline__ uint32_t range_pair(double v0, double v1) { return digit_range(v0) | (digit_range(v1) << 16); }
// Digit p (1-based) of two elements as packed bf16: 128 + field is the bf16 with the field in its low
// mantissa bits, so one packed fused multiply-add gives sign (field - 32) (digit 1: sign field) exactly.
template <int P, int W = 6>
__device__ __forceinline__ uint32_t digit_pair(long long U0, long long U1, uint32_t sg, uint32_t rg, int p) {
  static_assert(W == 6 || W == 7, "a field fits the mantissa of 128 + field");
  const int sh = W * (P - p);
  const uint32_t w = (__byte_perm((uint32_t)(U0 >> sh), (uint32_t)(U1 >> sh), 0x5410) & (W == 6 ? 0x003F003Fu : 0x007F007Fu)) | 0x43004300u;
  // -128, or -160 (W = 7: -192) and one less in the other range (the next bf16), times the sign
  const uint32_t c = (p == 1 ? 0xC300C300u : (W == 6 ? 0xC320C320u : 0xC340C340u) - rg) ^ (sg & 0x80008000u);
  uint32_t r;
  asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(sg), "r"(c));
  return r;
}

// Integer-valued accumulators v[0 .. NL-1] (levels 2 .. NL + 1 of one element) joined at the weight of
// the last one, for NL <= 8: sum_l v[l] 64^(NL-1-l).  SMALL: every |v| < 2^22, so that the integer is
// read off the bits of v + 1.5 2^23 (two full-rate operations; conversions run at an eighth of the rate);
// else |v| <= 2^24 (exact in fp32), converted.  Level l holds l + 1 digit products a step of K, so a pair
// stays within K 2^(2W-2) ((l + 1) 2^W + l + 2) < 2^31 for W = 6, l <= 6, K <= 1820 and W = 7, l <= 4, K <= 480.
template <int NL, bool SMALL, int W = 6, int NV = NL>
__device__ __forceinline__ long long join_levels(const float (&v)[NV]) {
  constexpr uint32_t C = 0x4B400000u;   // bits of 1.5 2^23
  auto bits = [&](int l) -> uint32_t {
    return SMALL ? __float_as_uint(v[l] + 12582912.0f) : (uint32_t)__float2int_rn(v[l]);
  };
  auto pair = [&](int l) -> int {       // two levels fit 32 bits
    return (int)(bits(l) * (1u << W) + bits(l + 1) - (SMALL ? C * ((1u << W) + 1u) : 0u));
  };
  long long V = pair(0);
#pragma unroll
  for (int l = 2; l + 1 < NL; l += 2) V = V * (1 << (2 * W)) + pair(l);
  if constexpr (NL & 1) V = V * (1 << W) + (int)(bits(NL - 1) - (SMALL ? C : 0u));
  return V;
}
// v / 64 and v / 128 rounded half away from zero (odd in v)
__device__ __forceinline__ int round64(int v) { return (v + 31 + (v >= 0 ? 1 : 0)) >> 6; }
__device__ __forceinline__ int round128(int v) { return (v + 63 + (v >= 0 ? 1 : 0)) >> 7; }

}  // namespace esmp2
