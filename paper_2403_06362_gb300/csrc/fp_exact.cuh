// fp_exact.cuh -- fp64 results computed on the integer pipes, bit for bit
// equal to the fp64 operations they replace.
//
// This GPU retires two fp64 lanes per clock per SM against 128 integer
// lanes, and its fp64 unit spends the same time on a warp instruction
// whatever the number of live lanes.  The fp64 transport kernels are bound by
// that unit, so every fp64 step whose exact result can be assembled from
// integer operations is moved off it:
//   floor_nonneg   floor(t) for 0 <= t < 2^63
//   floor_small    floor(t) for 0 <= t < 2^20
//   abs_le         |x| <= h for h >= 0
//   recip_rn       1/y correctly rounded (IEEE round to nearest even)
//   sqrt_rn        sqrt(x) correctly rounded
//   llrint_nonneg  llrint(v) for 0 <= v < 2^62
//   okey, d_lt ..  comparisons of doubles (sign-magnitude order keys)
//   mul_small      RN(j h) for a small integer j
// One fp64 addition that saves many integer instructions is the better trade
// where that unit is not the bound:
//   two_u_minus_1  2u - 1 for a draw u = n 2^-53 (exact: (2n - 2^53) 2^-53)
//   llrint_add     llrint(v) by an addition of 2^52
// All of them compile for host and device; the host copies let tests compare
// them with the host's IEEE arithmetic.
#pragma once
#include <cstdint>

#include "mc_log.cuh"  // to_bits, from_bits

namespace mcx {

using mclog::from_bits;
using mclog::to_bits;

__host__ __device__ __forceinline__ int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

__host__ __device__ __forceinline__ uint64_t mulhi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

__host__ __device__ __forceinline__ float rcp_f32(float x) {
#ifdef __CUDA_ARCH__
  return __frcp_rn(x);
#else
  return 1.0f / x;
#endif
}

// 2u - 1 for u = n 2^-53, 0 <= n < 2^53: the low 52 bits of n behind the
// exponent of 1 are 1 + (n mod 2^52) 2^-52, and one exact subtraction of 1 (n
// >= 2^52) or 2 leaves (2n - 2^53) 2^-53, +0 for n = 2^52.  Assembled on the
// integer pipes (leading zeros, shifts, exponent) it takes some 17 more
// instructions, worth more there than the 16 cycles of the fp64 unit: 3 * 10^7
// pulse sources 40.4 -> 37.9 ms, 300 000 slab histories of 9 flights 243 ->
// 234 us, box fp64 event schedule 11.0 -> 10.6 ms.
__host__ __device__ __forceinline__ double two_u_minus_1(uint64_t n) {
  return from_bits((n & ((1ull << 52) - 1ull)) | (1023ull << 52)) - ((n >> 52) != 0ull ? 1.0 : 2.0);
}

// floor(t) for 0 <= t < 2^63 (t finite, not negative zero excluded).
__host__ __device__ __forceinline__ uint64_t floor_nonneg(double t) {
  const uint64_t b = to_bits(t);
  const int e = (int)(b >> 52) - 1023;
  if (e < 0) return 0ull;
  const uint64_t m = (b & ((1ull << 52) - 1ull)) | (1ull << 52);
  return e <= 52 ? m >> (52 - e) : m << (e - 52);
}

// The bits of x for comparisons.  On the device they come through a move that
// the compiler does not see through: given a plain bit cast it recognises
// bits & ~2^63 as |x| and issues that to the fp64 unit, where it takes as
// long as an addition, and bits << 1 == 0 as a comparison with zero.  (65 of
// the 126 fp64 instructions of a box flight were such; without them 3 * 10^6
// histories took 37.9 ms instead of 45.7.)
__host__ __device__ __forceinline__ uint64_t raw_bits(double x) {
#ifdef __CUDA_ARCH__
  uint64_t b;
  asm("mov.b64 %0, %1;" : "=l"(b) : "d"(x));
  return b;
#else
  return to_bits(x);
#endif
}
__host__ __device__ __forceinline__ uint64_t mag_bits(double x) { return raw_bits(x) & ~(1ull << 63); }

// |x|.
__host__ __device__ __forceinline__ double abs_bits(double x) { return from_bits(mag_bits(x)); }

// |x| <= h for h >= 0 (finite): non-negative doubles order like their bits.
__host__ __device__ __forceinline__ bool abs_le(double x, double h) {
  return mag_bits(x) <= to_bits(h);
}

// q = RN(2^105 / M) for 2^52 <= M < 2^53 (ties cannot occur: 2^106 = (2q + 1) M
// would make M a power of two, and M = 2^52 divides exactly).  An fp32
// reciprocal of m = M 2^-52 gives Q = 2^32 / m (1 - e) with |e| < 2^-22, and
// 2^84 e = 2^84 - M Q exactly from the low words.  Then
//   2^53 / m = 2^21 Q (1 + e + e^2) + O(2^53 e^3 < 2^-13)
// puts q within a unit, and the exact remainder fixes and rounds it.  (Half
// the instructions of a table reduction with a polynomial.)
__host__ __device__ __forceinline__ uint64_t recip_mantissa(uint64_t M) {
  const uint32_t m32 = (uint32_t)(M >> 21);  // m 2^31
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint2float_rn(m32) * 0x1p-31f));
  const uint32_t Q = __float2uint_rz(fminf(y * 0x1p32f, 4294967040.0f));
#else
  const float y = 1.0f / ((float)m32 * 0x1p-31f) * 0x1p32f;
  const uint32_t Q = y < 4294967040.0f ? (uint32_t)y : 4294967040u;
#endif
  const long long e = (long long)(0ull - M * (uint64_t)Q);  // 2^84 (1 - M Q 2^-84), below 2^62 in magnitude
  const int eh = (int)(e >> 32);                             // e 2^52
  // 2^21 Q e = Q (e 2^84) 2^-63, and 2^21 Q e^2 from e's high word
  const long long t1 = ((long long)eh * (long long)Q + (long long)(((uint64_t)(uint32_t)e * Q) >> 32)) >> 31;
  const uint32_t e2 = (uint32_t)(((long long)eh * eh) >> 32);  // e^2 2^72, below 2^30
  const uint32_t t2 = (uint32_t)(((uint64_t)e2 * Q) >> 51);    // Q e^2 2^21
  uint64_t q = ((uint64_t)Q << 21) + (uint64_t)t1 + t2 + 1ull;  // (1: half of what the truncations take)
  long long rem = (long long)(0ull - q * M);  // 2^105 - q M (its low word: |rem| < 2^63)
  if (rem < 0) { --q; rem += (long long)M; }
  if (rem >= (long long)M) { ++q; rem -= (long long)M; }
  if ((uint64_t)rem * 2ull > M) ++q;
  return q;
}

// RN(1 / y) on the integer pipes for normal y whose reciprocal is normal
// (biased exponent 1..2044); the library division otherwise (zero,
// subnormal, huge, inf, NaN).
__host__ __device__ __forceinline__ double recip_rn(double y) {
  const uint64_t b = to_bits(y);
  const uint64_t sign = b & (1ull << 63);
  const uint32_t E = (uint32_t)(b >> 52) & 0x7FFu;
  if (E == 0u || E > 2044u) return 1.0 / y;
  const uint64_t frac = b & ((1ull << 52) - 1ull);
  if (frac == 0ull) return from_bits(sign | ((uint64_t)(2046u - E) << 52));  // a power of two
  const uint64_t q = recip_mantissa(frac | (1ull << 52));  // in [2^52, 2^53)
  return from_bits(sign | (((uint64_t)(2045u - E) << 52) + (q - (1ull << 52))));
}

// RN(sqrt(x)) for a positive normal x.  With x = A 2^(2k - 64), A in
// [2^62, 2^64), the result is RN(sqrt(N)) 2^(k - 53), N = A 2^42.  An fp32
// reciprocal square root y (relative error below 2^-20) gives sqrt(A) with
// scale 2^63, and two steps s += (x - s^2) y / 2 on 64-bit products, each
// shrinking the error by y's own, leave it below 2^-59; rounded to 53 bits
// it is within one unit, and the exact remainder N - q^2 (its low word: it is
// far below 2^63) rounds it.  A tie cannot occur: (q + 1/2)^2 is no integer.
// About 75 integer instructions; the fp64 unit's square root is a dozen of
// its own, 16 cycles per SM and warp each.
__host__ __device__ __forceinline__ double sqrt_rn(double x) {
  const uint64_t b = to_bits(x);
  const int E = (int)(b >> 52);  // positive: no sign
  const uint64_t m = (b & ((1ull << 52) - 1ull)) | (1ull << 52);
  const int odd = (E + 1) & 1;   // E - 1023 odd: one more doubling
  const uint64_t A = m << (10 + odd);
  const int k = (E - 1023 - odd) / 2 + 1;  // x = A 2^(2k - 64), E - 1023 - odd even
  const uint32_t ah = (uint32_t)(A >> 32);
#ifdef __CUDA_ARCH__
  const float y0 = rsqrtf(__uint2float_rn(ah) * 0x1p-32f);
  const uint32_t y = __float2uint_rz(fminf(y0 * 0x1p31f, 4294967040.0f));
#else
  const float y0 = 1.0f / std::sqrt((float)ah * 0x1p-32f);
  const uint32_t y = y0 * 0x1p31f < 4294967040.0f ? (uint32_t)(y0 * 0x1p31f) : 4294967040u;
#endif
  uint64_t s = mulhi64(A, (uint64_t)y << 32);  // sqrt(x) 2^63
  long long d = (long long)((A >> 2) - mulhi64(s, s));  // (x - s^2) 2^62, below 2^44
  s += (uint64_t)(((d >> 13) * (long long)y) >> 18);
  d = (long long)((A >> 2) - mulhi64(s, s));  // below 2^24
  s += (uint64_t)((d * (long long)y) >> 31);
  uint64_t q = (s + 512ull) >> 10;
  const long long rem = (long long)((A << 42) - q * q);
  if (rem > (long long)q) ++q;
  else if (rem <= -(long long)q) --q;
  // q in [2^52, 2^53]: the leading 1 (or the carry) adds into the exponent
  return from_bits(((uint64_t)(k + 1021) << 52) + q);
}

// A double's leading bits as an fp32 (truncated: relative error below 2^-23),
// |x| in [2^-120, 2^120], and whether x is in that range.
__host__ __device__ __forceinline__ bool f32_range(double x) {
  const uint32_t e = (uint32_t)(raw_bits(x) >> 52) & 0x7ffu;
  return e - 903u <= 240u;
}
__device__ __forceinline__ float f32_trunc(double x) {
  const uint64_t b = raw_bits(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  return __uint_as_float((hi & 0x80000000u) | ((((hi & 0x7fffffffu) << 3) | (lo >> 29)) - (896u << 23)));
}

// RN(1 / y) for a normal y with a normal reciprocal, biased exponent
// 1..2044 (a flight direction's component, say), without branches.
__host__ __device__ __forceinline__ double recip_normal(double y) {
  const uint64_t b = to_bits(y);
  const uint64_t q = recip_mantissa((b & ((1ull << 52) - 1ull)) | (1ull << 52));  // in [2^52, 2^53]
  const uint32_t E = (uint32_t)(b >> 52) & 0x7FFu;
  return from_bits((b & (1ull << 63)) + ((uint64_t)(2044u - E) << 52) + q);
}

// floor(t) for 0 <= t < 2^20, from the high word alone.
__host__ __device__ __forceinline__ uint32_t floor_small(double t) {
  const uint32_t h = (uint32_t)(raw_bits(t) >> 32), sh = 1043u - (h >> 20);
  return ((h & 0xfffffu) | 0x100000u) >> (sh < 31u ? sh : 31u);
}

// llrint(v) (round half to even) for 0 <= v < 2^62, from the bits.
__host__ __device__ __forceinline__ long long llrint_nonneg(double v) {
  const uint64_t b = to_bits(v);
  const int E = (int)(b >> 52);  // biased exponent: v = m 2^(E - 1075)
  const uint64_t m = (b & ((1ull << 52) - 1ull)) | (1ull << 52);
  if (E >= 1075) return (long long)(m << (E - 1075));
  // at most 63: below 1/2 (and zero) everything is shifted out, less than a half
  const int sh = 1075 - E < 63 ? 1075 - E : 63;
  const uint64_t q = m >> sh, rem = m << (64 - sh);  // rem: the bits shifted out, at the top
  const uint64_t half = 1ull << 63;
  return (long long)(q + ((rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull));
}

// The same by the rounding of v + 2^52, whose low bits are the integer, for v <
// 2^51; above, from the bits.
__host__ __device__ __forceinline__ long long llrint_add(double v) {
  if ((uint32_t)(raw_bits(v) >> 52) < 1023u + 51u)
    return (long long)(raw_bits(v + 4503599627370496.0) & ((1ull << 52) - 1ull));
  return llrint_nonneg(v);
}

// Order key of a non-NaN double: a < b  <=>  okey(a) < okey(b); -0 and +0
// share the key 0.
__host__ __device__ __forceinline__ long long okey(double x) {
  const long long m = (long long)mag_bits(x);
  return (long long)raw_bits(x) < 0 ? -m : m;
}
__host__ __device__ __forceinline__ bool d_lt(double a, double b) { return okey(a) < okey(b); }
__host__ __device__ __forceinline__ bool d_pos(double a) { return (long long)raw_bits(a) > 0; }        // a > 0
__host__ __device__ __forceinline__ bool d_neg(double a) { return raw_bits(a) > (1ull << 63); }         // a < 0
__host__ __device__ __forceinline__ bool d_zero(double a) { return (raw_bits(a) << 1) == 0ull; }        // a == 0

// RN(j h) for an integer 0 <= j < 2^11 and a normal h > 0 whose product
// stays normal: the exact product m_h j has at most 64 bits, rounded once.
__host__ __device__ __forceinline__ double mul_small(uint32_t j, double h) {
  if (j == 0u) return 0.0;
  const uint64_t b = to_bits(h);
  const uint64_t m = (b & ((1ull << 52) - 1ull)) | (1ull << 52);
  const uint64_t p = m * (uint64_t)j;  // < 2^64
  const int lz = clz64(p);             // 0..11
  const int sh = 11 - lz;              // bits below the 53 kept
  uint64_t q = p >> sh;
  if (sh > 0) {
    const uint64_t rem = p & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;  // may carry to 2^53
  }
  // value = q 2^(E_h + sh - 1075): biased exponent E_h + sh with q's leading
  // 1 at bit 52 (a carry to 2^53 moves into the exponent by itself)
  return from_bits((b & ~((1ull << 52) - 1ull)) + ((uint64_t)sh << 52) + (q - (1ull << 52)));
}

// A positive normal x as q 2^-s with a 32-bit q in [2^31, 2^32) (truncated),
// and floor(a x) within one for 0 <= a from it: a lookup guess that an exact
// comparison then corrects.
__host__ __device__ __forceinline__ void fixed_of(double x, uint32_t& q, int& s) {
  const uint64_t b = to_bits(x);
  q = (uint32_t)((((b & ((1ull << 52) - 1ull)) | (1ull << 52))) >> 21);
  s = 31 - ((int)(b >> 52) - 1023);
}
__host__ __device__ __forceinline__ uint64_t guess_floor_mul(double a, uint32_t q, int s) {
  const uint64_t b = to_bits(a);
  if ((b << 1) == 0ull) return 0ull;
  const int e = (int)(b >> 52) - 1023;
  const uint64_t m32 = (((b & ((1ull << 52) - 1ull)) | (1ull << 52))) >> 21;  // a ~ m32 2^(e - 31)
  const int sh = 31 + s - e;
  if (sh >= 64) return 0ull;
  if (sh <= 0) return 1ull << 40;
  return (m32 * (uint64_t)q) >> sh;
}

// llrint(w 2^32) for w >= 0 (2^32 w < 2^62): the scaling as an exponent add.
__host__ __device__ __forceinline__ long long fix32_nonneg(double w) {
  const uint64_t b = to_bits(w);
  if ((b >> 52) == 0ull) return 0;  // zero or below 2^-1022
  return llrint_nonneg(from_bits(b + (32ull << 52)));
}

// x 2^k for a normal x whose product stays normal (an exponent add).
__host__ __device__ __forceinline__ double scale_pow2(double x, int k) {
  return from_bits(to_bits(x) + ((uint64_t)(int64_t)k << 52));
}

}  // namespace mcx
