// rcp.cuh -- correctly rounded double reciprocal on the integer and FP32 pipes.
//
// GB300's FP64 pipe issues one warp instruction per 64 clocks per SMSP, so the
// ~7 dependent FP64 operations of a double division sit squarely on the pivot
// chain of the band LU.  This reciprocal uses integer arithmetic instead.  For a
// normal b = +-m * 2^(E-1075) with 2^52 <= m < 2^53 (E the biased exponent),
//   1/b = (2^105 / m) * 2^(970-E),
// so the rounded significand is q = Q + [2R > m] where Q = floor(2^105/m) and
// R = 2^105 - Q*m (no ties are possible: 2^106/m is not an integer for m > 2^52).
// Q is found as a quotient by approximate reciprocal with remainder correction
// (Knuth, TAOCP Vol. 2, Sec. 4.3.1): a Newton step on a two-float (double-float)
// representation of m gives Q within 2^9; one correction Q += (2^105 - Q*m)/m,
// the remainder's high bits times y's 24-bit significand in one integer
// multiply, brings Q within one unit; the exact remainder then fixes Q and
// decides the rounding.
// The result is the IEEE round-to-nearest 1/b, bit for bit.  Zeros, subnormals,
// infinities, NaN and |b| >= 2^1021 (whose reciprocal is subnormal) go to the
// ordinary division.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace bandlu {

__host__ __device__ __forceinline__ float rcp_approx_f32(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}

__host__ __device__ __forceinline__ uint64_t dbits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}

__host__ __device__ __forceinline__ double bitsd(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}

__host__ __device__ __forceinline__ float bitsf(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  std::memcpy(&x, &u, 4);
  return x;
#endif
}

__host__ __device__ __forceinline__ uint32_t fbits(float x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__float_as_uint(x);
#else
  uint32_t u;
  std::memcpy(&u, &x, 4);
  return u;
#endif
}

// Correctly rounded 1/b for every b whose reciprocal is a normal number and
// whose significand is not a power of two: *special is set for zeros,
// subnormals, infinities, NaN and |b| >= 2^1021, and the value returned then is
// meaningless.  Straight-line code (no branches), so it interleaves with other
// work.
__host__ __device__ __forceinline__ double rcp_rn_fast(double b, bool *special) {
  const uint64_t bits = dbits(b);
  const uint64_t E = (bits >> 52) & 0x7ffull;
  const uint64_t frac = bits & ((1ull << 52) - 1);
  const uint64_t sign = bits & (1ull << 63);
  *special = (E == 0) | (E >= 2045);
  const uint64_t m = frac | (1ull << 52);
  // M = m / 2^29 = xh + xl/2^29 with xh = floor(M), 2^23 <= xh < 2^24, written straight
  // into a float's bits (exponent 2^23), and 0 <= xl < 2^29.
  const uint32_t xh = (uint32_t)(m >> 29);
  const int32_t xl = (int32_t)(m & ((1ull << 29) - 1));
  const float xhf = bitsf((150u << 23) | (xh & 0x7fffffu)), xlf = (float)xl * 0x1p-29f;
  // y ~ 1/xh: hardware seed plus one Newton step; then one Newton step for 1/M
  // carried as the unevaluated pair y + t (relative error below 2^-45, plus 2^-47 from
  // rounding xl to a float).
  const float y0 = rcp_approx_f32(xhf);
  const float y = fmaf(y0, fmaf(-xhf, y0, 1.0f), y0);
  const float e = fmaf(-xlf, y, fmaf(-xhf, y, 1.0f));  // 1 - M*y
  const float t = y * e;
  // Q = (y + t) * 2^76 ~ 2^105/m within 2^9; y*2^76 is an exact integer (y in [2^-24, 2^-23]).
  const uint32_t yb = fbits(y);
  const uint32_t ym = (yb & 0x7fffffu) | 0x800000u;  // y = ym * 2^(yexp - 150)
  const int yexp = (int)(yb >> 23);
  uint64_t Q = (uint64_t)ym << (yexp - 74);
  Q = (uint64_t)((int64_t)Q + (int64_t)(int32_t)(t * 0x1p76f));
  // one correction from the exact remainder (2^105 = 0 mod 2^64 and |R| < 2^62): Q += R/m,
  // R/m ~ (R >> 31) * y * 2^2 = (R >> 31) * ym / 2^(148 - yexp), floored, within one unit
  int64_t R = (int64_t)(0ull - Q * m);
  Q = (uint64_t)((int64_t)Q + (((int64_t)(int32_t)(R >> 31) * (int64_t)ym) >> (148 - yexp)));
  // now |Q - 2^105/m| < 1.01: the exact remainder fixes Q and decides the rounding
  R = (int64_t)(0ull - Q * m);
  const bool lo = R < 0, hi = R >= (int64_t)m;
  Q = lo ? Q - 1 : (hi ? Q + 1 : Q);
  R = lo ? R + (int64_t)m : (hi ? R - (int64_t)m : R);
  Q += ((uint64_t)R > m - (uint64_t)R) ? 1ull : 0ull;  // 2R > m: round up
  const uint64_t rbits = sign | ((2045 - E) << 52) | (Q - (1ull << 52));
  const uint64_t pbits = sign | ((2046 - E) << 52);  // significand 1: 1/b is a power of two
  return bitsd(frac == 0 ? pbits : rbits);
}

// The same quotient with the rounding decided without a second exact remainder: with
// V = 2^105/m and the exact remainder R = 2^105 - Q*m of Q within 2^9.6, V = Q + R/m, and R/m
// is formed in fixed point (43 or 44 fractional bits) as the remainder's high word times y's
// 24-bit significand, within 2^-12 of its value.  Rounding that sum is the answer unless its
// fraction lies within 2^-11 of one half (one operand in 1000).  About 30 instructions against
// rcp_rn_fast's 50; in the register windows (regwin.cuh) the shorter stream is what counts.
// Correctly rounded 1/b, unless *special is set: then the value returned is
// meaningless and the caller divides (zeros, subnormals, infinities, NaN,
// |b| >= 2^1021, and the rare quotients too close to a rounding boundary for the
// fixed-point remainder to decide).  Straight-line code (no branches), so it
// interleaves with other work.
// The two 32-bit halves are kept apart: every 64-bit step is one wide
// multiply-add, and of the remainder only the high word is formed.
__host__ __device__ __forceinline__ double rcp_rn_quick(double b, bool *special) {
  const uint64_t bits = dbits(b);
  const uint32_t hi = (uint32_t)(bits >> 32), mlo = (uint32_t)bits;
  const uint32_t mhi = (hi & 0xfffffu) | 0x100000u;  // m = mhi * 2^32 + mlo
  // M = m / 2^29 = xh + xl with xh = floor(M), 2^23 <= xh < 2^24, and 0 <= xl < 1 cut to
  // 23 bits; both written straight into a float's bits.
  const float xh = bitsf((150u << 23) | ((mhi << 3 | mlo >> 29) & 0x7fffffu));
  const float xl = bitsf((127u << 23) | ((mlo >> 6) & 0x7fffffu)) - 1.0f;
  // y ~ 1/xh: hardware seed plus one Newton step (relative error below 2^-23); then one Newton
  // step for 1/M carried as the unevaluated pair y + t (relative error below 2^-44.5: the square
  // of e <= 2^-22.4, 2^-46 from xl's cut and 2^-46 from rounding e).
  const float y0 = rcp_approx_f32(xh);
  const float y = fmaf(y0, fmaf(-xh, y0, 1.0f), y0);
  const float e = fmaf(-xl, y, fmaf(-xh, y, 1.0f));  // 1 - M*y
  const float t = y * e;                             // |t| < 2^-45.3
  // Q = (y + t) * 2^76 ~ 2^105/m.  y*2^76 is an exact integer; t*2^76 is taken to a multiple of
  // 2^9 (t*2^67, below 2^21.7, rounded to an integer by adding 1.5*2^23), so |Q - V| < 2^9.6.
  const uint32_t yb = fbits(y);
  const uint32_t ym = (yb & 0x7fffffu) | 0x800000u;  // y = ym * 2^(yexp - 150), yexp 103 or 104
  const int yexp = (int)(yb >> 23);
  const int32_t ti = (int32_t)(fbits(fmaf(t, 0x1p67f, 12582912.0f)) - 0x4b400000u);
  const uint64_t Q = (uint64_t)ym * (1u << (yexp - 74)) + (uint64_t)((int64_t)ti * 512);
  // X = Q*m - 2^105 modulo 2^64 (2^105 is 0 there; |X| < 2^62.6), of which the high word is
  // enough: V = Q - X/m with X/m ~ (X >> 32) * y * 2^3 = (X >> 32) * ym / 2^sh, off by
  // 2^9.6 * 2^-22.4 (y for 1/M) and 2^-20 (X's low word).
  const uint32_t Ql = (uint32_t)Q, Qh = (uint32_t)(Q >> 32);
  const int32_t Xh = (int32_t)((uint32_t)(((uint64_t)Ql * mlo) >> 32) + Ql * mhi + Qh * mlo);
  const int sh = 147 - yexp;  // 43 or 44
  const int64_t P = (int64_t)Xh * -(int64_t)(int32_t)ym + (int64_t)((uint64_t)(1u << (sh - 33)) << 32);
  const int32_t Ph = (int32_t)(P >> 32);
  const uint64_t V = Q + (uint64_t)(int64_t)(Ph >> (sh - 32));  // floor(Q - X/m + 1/2)
  const uint32_t edge = (uint32_t)((Ph >> (sh - 43)) + 1) & 0x7ffu;  // its fraction, in units of 2^-11, plus one
  *special = (edge < 2u) | ((hi & 0x7ff00000u) - 0x100000u >= (2044u << 20));
  // significand V - 2^52 under exponent 2045 - E; V = 2^53 (a power of two) carries into the exponent
  const uint32_t rh = (((2044u << 20) - (hi & 0x7ff00000u)) | (hi & 0x80000000u)) + (uint32_t)(V >> 32);
  return bitsd(((uint64_t)rh << 32) | (uint32_t)V);
}

#ifdef __CUDACC__
// Out of line, so that the rarely taken division is never if-converted (an
// unconditional FP64 division in every thread costs more than the reciprocal).
__device__ __noinline__ static double rcp_division(double b) { return 1.0 / b; }
#endif

// Correctly rounded 1/b (IEEE binary64, round to nearest even).
__host__ __device__ __forceinline__ double rcp_rn(double b) {
  bool special;
  double r = rcp_rn_quick(b, &special);
#ifdef __CUDA_ARCH__
  if (special) r = rcp_division(b);
#else
  if (special) r = 1.0 / b;
#endif
  return r;
}

// ---------------------------------------------------------------------------
// x / d, correctly rounded, for a divisor known before the dividend (the
// diagonal of U in the back substitution), on the integer pipes.  With
// |d| = md * 2^(Ed-1075) and x alike (52-bit fractions, 2^52 <= m < 2^53), d gets
// ahead of time, off the dependence chain, a 63-bit reciprocal
//   R = 2^115/md within 1.5  (div_known_prep),
// and the quotient then is one truncated multiplication: Q = the high 64 bits of
// (mx * 2^11) * R ~ 2^62 * mx/md, short by less than 5 (three low partial products
// are dropped) and long by less than 1.5.  It has 62 or 63 bits, so rounding it to
// 53 is decided unless its low bits lie within that error of the rounding boundary
// (one quotient in 64 to 128); those, and dividends, divisors or quotients that
// are not normal numbers, take the ordinary division.  About 25 short-latency
// instructions: on GB300 the four dependent FP64 operations of a quotient from a
// two-term reciprocal cost 64 clk each.
__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

struct Divisor {
  uint32_t rl, rh;  // R
  uint32_t eb;      // (1021 - Ed) << 20 modulo 2^32: the quotient's exponent field less the dividend's, less
                    // one (the significand's leading bit adds it); kNoDivisor for a d that is not normal
  uint32_t sign;    // d's sign bit
};
constexpr uint32_t kNoDivisor = 0x80000000u;  // fails every range test of div_quick

__host__ __device__ __forceinline__ Divisor div_known_prep(double d) {
  const uint64_t bits = dbits(d);
  const uint32_t hi = (uint32_t)(bits >> 32);
  const uint32_t ed = (hi >> 20) & 0x7ffu;
  const uint64_t m = (bits & ((1ull << 52) - 1)) | (1ull << 52);
  // 1 / (md / 2^52) = V / 2^53 to nearest, 2^52 <= V <= 2^53 (2^53: a power of two)
  const uint64_t yb = dbits(rcp_rn(bitsd((1023ull << 52) | (bits & ((1ull << 52) - 1)))));
  const uint64_t V = ((yb & ((1ull << 52) - 1)) | (1ull << 52)) << ((yb >> 52) - 1022);
  // R0 = V * 2^10, within 2^9 of 2^115/md; one correction from the exact remainder
  uint64_t R = V << 10;
  const int64_t X = (int64_t)(0ull - R * m);  // 2^115 - R0*md modulo 2^64, |X| <= 2^62
  R += (uint64_t)(((X >> 32) * (int64_t)(V >> 22)) >> 51);
  const bool ok = ed >= 1 && ed <= 2046;
  return Divisor{(uint32_t)R, (uint32_t)(R >> 32), ok ? (1021u - ed) << 20 : kNoDivisor, hi & 0x80000000u};
}

// x / d, unless *unsure is set: then the value returned is meaningless.
// Straight-line code.
__host__ __device__ __forceinline__ double div_quick(double x, const Divisor &d, bool *unsure) {
  const uint64_t bits = dbits(x);
  const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
  const uint32_t ah = ((hi & 0xfffffu) | 0x100000u) << 11 | lo >> 21, al = lo << 11;  // mx * 2^11
  const uint64_t Q = (uint64_t)ah * d.rh + ((uint64_t)mulhi32(ah, d.rl) + mulhi32(al, d.rh));
  const uint32_t big = (uint32_t)(Q >> 62);  // 1: mx >= md, the quotient's significand is Q >> 10; 0: Q >> 9
  const uint32_t half = 256u << big;
  const uint64_t T = Q + (half + 5u);        // plus what Q may be short by
  const uint64_t V = T >> (9u + big);        // 2^52 <= V <= 2^53
  const uint32_t e = hi & 0x7ff00000u;
  const uint32_t low = (uint32_t)T & (2u * half - 1u);
  *unsure = (low < 8u) | (e - 0x100000u >= 0x7fe00000u) | (e + d.eb - 0x100000u >= 0x7fb00000u);
  const uint32_t rh = (e + d.eb + (big << 20) + (uint32_t)(V >> 32)) | ((hi & 0x80000000u) ^ d.sign);
  return bitsd(((uint64_t)rh << 32) | (uint32_t)V);
}

#ifdef __CUDACC__
__device__ __noinline__ static double div_division(double x, double d) { return x / d; }
#endif

// What the sweeps do with a dividend that div_quick is unsure of: the reference-BLAS
// zero test (a zero is kept, its sign with it, and not divided; *nonzero false), else
// the division.  A zero fails div_quick's range test, so it always comes here.  live
// false: x belongs to no row.
__host__ __device__ __forceinline__ double div_unsure(double x, double d, bool live, bool *nonzero) {
  const uint64_t bits = dbits(x);
  *nonzero = (((uint32_t)(bits >> 32) << 1) | (uint32_t)bits) != 0u;
#ifdef __CUDA_ARCH__
  return *nonzero && live ? div_division(x, d) : x;
#else
  return *nonzero && live ? x / d : x;
#endif
}

}  // namespace bandlu
