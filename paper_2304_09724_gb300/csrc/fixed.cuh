// Block fixed-point arithmetic on the integer pipe, for the Cauchy-Kovalevskaya recursion.
//
// Why.  One FP64 instruction holds a scheduler's FP64 unit for 64 clocks per warp (0.5 lanes per
// clock), while IMAD.WIDE (32 x 32 + 64 bits) takes 2.  A product of two 59-bit numbers costs three
// of them, so a sum of products in fixed point runs ten times as fast as in FP64 and leaves the
// FP64 unit to the rest of the kernel, which runs at the same time on other warps.
//
// Format.  x = X 2^-61 times a power of two of its own for each field and total degree.  Leading
// coefficients (degree 0) have |x| < 1, all others |x| < 1/4.  X is held as h 2^31 + l with
// |l| <= 2^30 (Fx), so |h| <= 2^30 or 2^28.  A coefficient of a product of two series is a sum of at
// most 12 products, at most two of them with a leading factor: hh = sum h h' and hl = sum (h l' + l h')
// stay below 2^63 (|hl| <= 2^30 (2 (2^30 + 2^28) + 20 * 2^28) = 0.94 * 2^63).  The l l' terms are left
// out (at most 2^-62 each, of either sign) and the sum is rounded once, to 2^-61: a leading
// coefficient in [1/2, 1) is rounded to a multiple of 2^-53 in FP64.  (A 32-bit l would split without
// a mask, but leaves l l' of up to 2^-60 out: 4 to 5 times the error.)  Magnitudes are collected on the
// way; a point whose values leave the format is repeated in another scale.
#pragma once
#include <cstdint>

#if defined(__CUDACC__)
#define FX_FN __host__ __device__ __forceinline__
#define FX_DEV __device__ __forceinline__
#else
#define FX_FN inline
#define FX_DEV inline
#endif

namespace shweno {

constexpr int FX_S = 31;  // bits of the low limb
constexpr int FX_Q = 61;  // fraction bits of a coefficient
constexpr int FX_C = 58;  // fraction bits of a constant
constexpr int FX_D = 57;  // fraction bits of the second pass's data (room for end values of 8 times the data)

struct Fx {
  int32_t h, l;
};
struct FxAcc {
  int64_t hh, hl;
};
// Magnitudes seen: OR of h + 2^28, or of the high word + 2^27, over the operands.  In range: |h| < 2^28, the high
// word within +-2^27 (|x| < 1/4).  Checking every operand suffices: a sum of products of operands in range
// stays below 2, where h still holds it, but for the time update (four times mu + p, plus mv: below 5.5 for gamma
// up to 3) and the difference of two end values.  Those are checked by the high word, which holds any 64-bit
// value (what wraps at 4 is out of range still).
struct FxRange {
  uint32_t h, t = 0;
  FX_FN bool bad() const { return (h >> 29) != 0 || (t >> 28) != 0; }
};

// 64-bit values that are to be split carry FX_HALF (half a unit of h): the split then floors.
constexpr int64_t FX_HALF = int64_t(1) << (FX_S - 1);

// Start of a sum: half a unit in the last place (rounds to nearest), and FX_HALF if it is to be split.
template <int Q = FX_Q>
FX_FN FxAcc fx_zero(bool split = false) {
  return FxAcc{split ? FX_HALF >> (2 * FX_S - Q) : 0, int64_t(1) << (Q - FX_S - 1)};
}
// c + a b.  As PTX: the compiler widens the limbs and multiplies 64 x 64 bits (three instructions).
FX_FN int64_t fx_wide(int32_t a, int32_t b, int64_t c) {
#if defined(__CUDA_ARCH__)
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return c + (int64_t)a * b;
#endif
}
FX_FN void fx_mac(FxAcc& s, Fx a, Fx b) {
  s.hh = fx_wide(a.h, b.h, s.hh);
  s.hl = fx_wide(a.h, b.l, s.hl);
  s.hl = fx_wide(a.l, b.h, s.hl);
}
// s += a * c 2^-30 with an integer c (c = 2^30: adds a itself)
FX_FN void fx_mac_int(FxAcc& s, Fx a, int32_t c) {
  s.hh = fx_wide(a.h, c, s.hh);
  s.hl = fx_wide(a.l, c, s.hl);
}
template <int Q = FX_Q>
FX_FN int64_t fx_sum(const FxAcc& s) {
  if (2 * FX_S - Q == 1) return s.hh + s.hh + (s.hl >> (Q - FX_S));
  return (int64_t)((uint64_t)s.hh << (2 * FX_S - Q)) + (s.hl >> (Q - FX_S));
}
// z + FX_HALF as limbs
FX_FN Fx fx_split(int64_t z, FxRange& r) {
  Fx v;
  v.h = (int32_t)(z >> FX_S);
  v.l = (int32_t)((uint32_t)z & 0x7fffffffu) - (int32_t)FX_HALF;
  r.h |= (uint32_t)(v.h + (1 << 28));
  return v;
}
// The same for any 64-bit value.  (2D: for all, one word to keep; vortex 2048^2 98.7 ms, with the other check beside
// it 101.)
FX_FN Fx fx_split_any(int64_t z, FxRange& r) {
  FxRange in{0};
  r.t |= (uint32_t)((int32_t)(z >> 32) + (1 << 27));
  return fx_split(z, in);
}
// For any 64-bit value, as an operand of sums of at most four products with constants below 1 (second
// pass): |x| < 1/2.
FX_FN Fx fx_split_wide(int64_t z, FxRange& r) {
  FxRange in{0};
  r.h |= (uint32_t)((int32_t)(z >> 32) + (1 << 28));
  return fx_split(z, in);
}
FX_FN int64_t fx_join(Fx a) { return (int64_t)((uint64_t)(int64_t)a.h << FX_S) + a.l; }

// ------------------------------------------------------------------ to and from double
FX_FN int32_t fx_hi(double x) {
#if defined(__CUDA_ARCH__)
  return __double2hiint(x);
#else
  uint64_t u;
  __builtin_memcpy(&u, &x, 8);
  return (int32_t)(u >> 32);
#endif
}
FX_FN uint64_t fx_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  __builtin_memcpy(&u, &x, 8);
  return u;
#endif
}
FX_FN double fx_from_bits(uint64_t u) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)u);
#else
  double x;
  __builtin_memcpy(&x, &u, 8);
  return x;
#endif
}
FX_FN int fx_clz(uint64_t u) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)u);
#else
  return u ? __builtin_clzll(u) : 64;
#endif
}
// e with |x| < 2^e from the high word's magnitude bits (biased exponent - 1022)
FX_FN int fx_exp(int32_t hi_abs) { return (hi_abs >> 20) - 1022; }
// x 2^-e in fixed point, rounded to nearest; |x| < 2^(e + FX_Q + 1 - Q).  Far smaller values give 0.
template <int Q = FX_Q>
FX_FN int64_t fx_from_double(double x, int e) {
  const uint64_t u = fx_bits(x);
  const uint64_t m = ((u & 0xfffffffffffffull) | 0x10000000000000ull) << 9;  // |x| = m 2^(fx_exp - 62)
  // X = m 2^(fx_exp - 62 - e + Q): a right shift by n + 1
  uint32_t n = (uint32_t)(FX_Q - Q + e - fx_exp((int32_t)(u >> 32) & 0x7fffffff));
  if (n > 63) n = 63;
  const int64_t t = (int64_t)(((m >> n) + 1) >> 1);
  return (int64_t)u < 0 ? -t : t;
}
// z 2^(e - 61) rounded to nearest; 0 and infinity beyond the normal range
FX_FN double fx_to_double(int64_t z, int e) {
  if (z == 0) return 0.0;
  const uint64_t s = z < 0 ? 0x8000000000000000ull : 0ull;
  uint64_t m = z < 0 ? (uint64_t)-z : (uint64_t)z;
  const int c = fx_clz(m);
  m <<= c;                                  // leading one in bit 63: |z| = m 2^-c
  const uint64_t f = (m >> 11) + ((m >> 10) & 1);  // 53 bits, round half up (a carry moves the exponent)
  const int b = 1022 + (64 - c) + e - FX_Q;  // biased exponent
  if (b < 1) return 0.0;
  if (b > 2046) return fx_from_bits(s | 0x7ff0000000000000ull);
  return fx_from_bits(s | (((uint64_t)b << 52) + (f - 0x10000000000000ull)));
}

}  // namespace shweno
