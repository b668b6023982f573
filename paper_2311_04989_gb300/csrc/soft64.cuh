// soft64.cuh -- FP64 division, square roots, comparisons, conversions and some sums without the FP64 pipe.
//
// GB300 issues one FP64 warp instruction per ~70 cycles and scheduler (measured: 126 M of them in the
// 7.43 ms of an FP64 k_faces, the pipe 87 % busy, the issue slots 7 %), and the FP64 division and square
// root of the compiler are about eight to ten of them each.  Here the significands are divided as integers:
// an FP32 reciprocal (square root) refined once to ~30 bits, two quotient digits from it, and an exact
// remainder that decides the last bit -- some 60 integer and FP32 instructions, which the idle issue slots
// take.  div64 and sqrt64 are correctly rounded (round to nearest even), so they return the bits of the IEEE
// operations they stand for; rsqrt64 is within 0.65 ulp.  Operands or results that are zero, subnormal,
// infinite or NaN take the operator itself (a zero dividend of div64 does not).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace grs {

// 1/x for x in [1, 2) and 1/sqrt(x) for x in [1, 4), at least 1/2; a relative error of 2^-22 is allowed for below
#ifdef __CUDACC__
__device__ __forceinline__ float rcp_apx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return fmaxf(y, 0.5f);
}
__device__ __forceinline__ float rsqrt_apx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return fmaxf(y, 0.5f);
}
#else   // a host build (the CPU tests of the integer arithmetic) brings its own
float rcp_apx(float x);
float rsqrt_apx(float x);
#endif

__device__ __forceinline__ uint64_t bits64(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double from64(uint64_t u) { return __longlong_as_double((long long)u); }
// low 64 bits of (hi:lo) >> s, 0 < s < 32
__device__ __forceinline__ uint32_t fsr(uint32_t lo, uint32_t hi, int s) { return __funnelshift_r(lo, hi, s); }
__device__ __forceinline__ uint64_t mulw(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

// a / b.  Significands A, B (53 bits), A doubled if below B, so the ratio r = A/B lies in [1, 2):
//   R     reciprocal 2^84/B from below, short by at most 12 units of its 32 bits (one Newton step on the FP32
//         reciprocal)
//   q1    r 2^30 from below, short by at most 14;  rem = A 2^30 - q1 B < 2^57 exactly
//   Q     q1 2^28 + (rem 2^28/B) = r 2^58 from below, short by at most 28
//   M     round(r 2^52), or one more: (Q + 32 + 32) >> 6; the sign of A 2^53 - (2 M - 1) B (its low 64 bits:
//         it is smaller than 2^55) tells which.  It is never zero: a quotient is never halfway between two
//         53-bit numbers.
__device__ __forceinline__ double div64(double a, double b) {
  const uint64_t ua = bits64(a), ub = bits64(b);
  const uint32_t ah = (uint32_t)(ua >> 32), bh = (uint32_t)(ub >> 32), bl = (uint32_t)ub;
  const uint32_t ea = (ah >> 20) & 0x7ffu, eb = (bh >> 20) & 0x7ffu;
  int e = (int)ea - (int)eb;
  const bool az = (ua << 1) == 0;
  // both normal and so the quotient, whichever its rounding: exponent e or e - 1
  if (!(eb - 1u < 2046u && (az || (ea - 1u < 2046u && (uint32_t)(e + 1021) < 2045u)))) return a / b;
  uint64_t A = (ua & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const uint64_t B = (ub & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const uint32_t Bh = (uint32_t)(B >> 32);
  const int lt = A < B;
  A <<= lt;
  e -= lt;
  const uint32_t Al = (uint32_t)A, Ah = (uint32_t)(A >> 32);
  // FP32 reciprocal of the leading 23 bits (odd, so it is below 1), biased down by 2^-21
  const float y = rcp_apx(__uint_as_float((fsr(bl, Bh, 29) & 0x7ffffeu) | 0x3f800001u));
  const uint32_t Y = ((__float_as_uint(y) << 8) | 0x80000000u) - 2048u;
  const uint32_t t = __umulhi(fsr(bl, Bh, 21), Y);
  const uint32_t R = Y + __umulhi(Y, (0x80000000u - t) << 1) - 6u;
  const uint32_t q1 = __umulhi(fsr(Al, Ah, 22), R);
  const uint64_t p1 = mulw(q1, bl) + ((uint64_t)(q1 * Bh) << 32);
  const uint64_t rem = (A << 30) - p1;
  const uint32_t q2 = __umulhi((uint32_t)(rem >> 25), R);   // rem 2^27 / B
  const uint64_t Q = ((uint64_t)q1 << 28) + ((uint64_t)q2 << 1) + 64u;
  const uint64_t M = Q >> 6;
  const uint32_t Ml = (uint32_t)M, Mh = (uint32_t)(M >> 32);
  const uint64_t MB = mulw(Ml, bl) + ((uint64_t)(Ml * Bh + Mh * bl) << 32);
  const int64_t d = (int64_t)((((A << 52) - MB) << 1) + B);
  const uint64_t m = M + ((uint64_t)(uint32_t)(e + 1022) << 52) - (uint64_t)(d < 0);
  const uint64_t sg = (ua ^ ub) & 0x8000000000000000ull;
  return from64(sg | (az ? 0ull : m));
}

// sqrt(x).  X = significand, doubled for an odd exponent: s = sqrt(X/2^52) in [1, 2):
//   Y     2^32/s from below, short by at most 16 units;  s1 = s 2^30 from below, short by at most 18
//   rem = X 2^8 - s1^2 exactly;  Q = s 2^58 = s1 2^28 + rem 2^28/(2 s) from below, short by at most 56
//   M     round(s 2^52) or one more, (Q + 60 + 32) >> 6; the sign of X 2^54 - (2 M - 1)^2 tells which (never zero, as above)
__device__ __forceinline__ double sqrt64(double x) {
  const uint64_t u = bits64(x);
  const uint32_t h = (uint32_t)(u >> 32);
  const uint32_t ex = h >> 20;
  if (ex - 1u >= 2046u) return sqrt(x);   // zero, subnormal, negative, infinite, NaN
  const int odd = (int)((ex & 1u) ^ 1u);  // the unbiased exponent ex - 1023 is odd
  const uint64_t X = ((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << odd;
  const uint32_t Xh = (uint32_t)(X >> 22);
  // leading bits as an FP32 number in [1, 4), odd in the last place so that the result is below 1
  const float f = __uint_as_float((0x3f800000u + ((uint32_t)odd << 23)) | (fsr((uint32_t)u, h, 29) & 0x7ffffeu) | 1u);
  const uint32_t Y0 = ((__float_as_uint(rsqrt_apx(f)) << 8) | 0x80000000u) - 2048u;
  const uint32_t er = 0x40000000u - __umulhi(Xh, __umulhi(Y0, Y0));
  const uint32_t Y = Y0 + __umulhi(Y0, er << 1) - 8u;
  const uint32_t s1 = __umulhi(Xh, Y);
  const uint64_t rem = (X << 8) - mulw(s1, s1);
  const uint32_t q2 = __umulhi((uint32_t)(rem >> 5), Y);   // rem 2^26 / (2 s1)
  const uint64_t Q = ((uint64_t)s1 << 28) + ((uint64_t)q2 << 2) + 92u;
  const uint64_t M = Q >> 6;
  const uint64_t T = 2 * M - 1;
  const uint32_t Tl = (uint32_t)T, Th = (uint32_t)(T >> 32);
  const uint64_t TT = mulw(Tl, Tl) + ((uint64_t)(2u * Tl * Th) << 32);
  const int64_t d = (int64_t)((X << 54) - TT);
  return from64(M + ((uint64_t)((ex + 1021u) >> 1) << 52) - (uint64_t)(d < 0));
}

// 1/sqrt(x): Y as in sqrt64, then one Newton step in 64 bits: e = 1 - X Y^2 (2^62 units, below 2^35), Y (1 + e/2)
__device__ __forceinline__ double rsqrt64(double x) {
  const uint64_t u = bits64(x);
  const uint32_t h = (uint32_t)(u >> 32);
  const uint32_t ex = h >> 20;
  if (ex - 1u >= 2046u) return rsqrt(x);
  const int odd = (int)((ex & 1u) ^ 1u);
  const uint64_t X = ((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << odd;
  const uint32_t Xh = (uint32_t)(X >> 22);
  const float f = __uint_as_float((0x3f800000u + ((uint32_t)odd << 23)) | (fsr((uint32_t)u, h, 29) & 0x7ffffeu) | 1u);
  const uint32_t Y0 = ((__float_as_uint(rsqrt_apx(f)) << 8) | 0x80000000u) - 2048u;
  const uint32_t er = 0x40000000u - __umulhi(Xh, __umulhi(Y0, Y0));
  const uint32_t Y = Y0 + __umulhi(Y0, er << 1) - 8u;
  const uint64_t e = 0x4000000000000000ull - __umul64hi(X << 10, mulw(Y, Y));
  const uint64_t y = ((uint64_t)Y << 32) + (mulw(Y, (uint32_t)(e >> 4)) >> 27);   // 2^64/s from below
  const uint64_t M = ((y >> 1) + 0x202ull) >> 10;                                 // nearest
  // exponent: x = s^2 2^(2k), 1/sqrt(x) = (M 2^-53) 2^-k
  const int k = ((int)ex - 1023 - odd) / 2;
  return from64(M + ((uint64_t)(uint32_t)(1021 - k) << 52));
}

// a * b by the FP64 pipe in a branch that is rarely taken: volatile, so that the compiler does not compute it
// ahead of the branch for every thread
__device__ __forceinline__ double mul_rare(double a, double b) {
#ifdef __CUDACC__
  double r;
  asm volatile("mul.rn.f64 %0, %1, %2;" : "=d"(r) : "d"(a), "d"(b));
  return r;
#else
  return a * b;
#endif
}

// a * b, correctly rounded, for products of the hot FP64 kernels that are no part of a fused multiply-add: ~45
// instructions of the idle issue slots for one of the FP64 pipe (70 cycles of a scheduler there).  Both
// significands shifted to 64 bits, the product's upper 64 bits with the lower ones folded into the last, rounded
// to nearest even.  Zero and operands or results out of the normal range: the operator.
__device__ __forceinline__ double mul64(double a, double b) {
  const uint64_t ua = bits64(a), ub = bits64(b);
  const uint32_t ah = (uint32_t)(ua >> 32), bh = (uint32_t)(ub >> 32);
  const uint32_t ea = (ah >> 20) & 0x7ffu, eb = (bh >> 20) & 0x7ffu;
  const int e = (int)(ea + eb) - 1023;            // exponent of the product, or one more
  if (!(ea - 1u < 2046u && eb - 1u < 2046u && (uint32_t)(e - 1) < 2044u)) return mul_rare(a, b);
  const uint32_t xh = 0x80000000u | fsr((uint32_t)ua, ah, 21), xl = (uint32_t)ua << 11;
  const uint32_t yh = 0x80000000u | fsr((uint32_t)ub, bh, 21), yl = (uint32_t)ub << 11;
  const uint64_t ll = mulw(xl, yl);
  const uint64_t m1 = mulw(xh, yl) + (ll >> 32);
  const uint64_t m2 = mulw(xl, yh) + (uint32_t)m1;
  uint64_t n = mulw(xh, yh) + (m1 >> 32) + (m2 >> 32);
  n |= (uint64_t)(((uint32_t)m2 | (uint32_t)ll) != 0u);
  const uint32_t top = (uint32_t)(n >> 63);       // the product of the significands is 2 or more
  n = top ? (n >> 1) | (n & 1u) : n;              // leading bit at 62
  n = (n + 0x1ffu + ((n >> 10) & 1u)) >> 10;      // 53 bits (54 after a carry, which steps the exponent)
  return from64(((ua ^ ub) & 0x8000000000000000ull) | (n + ((uint64_t)(uint32_t)(e + (int)top - 1) << 52)));
}

// x 2^-K, exactly for a normal result
template <int K>
__device__ __forceinline__ double scale64(double x) {
  const uint64_t u = bits64(x);
  const uint32_t e = (uint32_t)(u >> 52) & 0x7ffu;
  if (e - (K + 1u) < 2046u - K) return from64(u - ((uint64_t)K << 52));
  return mul_rare(x, 1.0 / (1 << K));
}

// whether x is finite, from the exponent bits of its high word (integer operations only: on GB300 an
// FP64 comparison is an instruction of the narrow FP64 pipe)
__device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// FP64 comparisons on the encodings (an FP64 comparison is an instruction of the narrow FP64 pipe)
// x < 0, false for -0 and NaN
__device__ __forceinline__ bool neg64(double x) {
  return (unsigned long long)__double_as_longlong(x) - 0x8000000000000001ull < 0x7ff0000000000000ull;
}
// x == 0 (either sign)
__device__ __forceinline__ bool zero64(double x) { return ((unsigned long long)__double_as_longlong(x) << 1) == 0ull; }
// a > b for b >= 0; false for a NaN a
__device__ __forceinline__ bool gtp64(double a, double b) {
  const long long u = __double_as_longlong(a);
  return u > (__double_as_longlong(b) & 0x7fffffffffffffffll) && u <= 0x7ff0000000000000ll;
}

// a > b for any signs; false for a NaN
__device__ __forceinline__ bool gt64(double a, double b) {
  const long long u = __double_as_longlong(a), v = __double_as_longlong(b);
  const long long ku = u ^ ((u >> 63) & 0x7fffffffffffffffll), kv = v ^ ((v >> 63) & 0x7fffffffffffffffll);
  const unsigned long long mu = (unsigned long long)u << 1, mv = (unsigned long long)v << 1;
  return ku > kv && mu <= 0xffe0000000000000ull && mv <= 0xffe0000000000000ull && (mu | mv) != 0ull;
}

// Precision conversions without the FP64 pipe (on GB300 an F2F conversion is an FP64-pipe
// instruction, ~1/64 of the FP32 rate), in integer arithmetic on the IEEE-754 encodings.
// FP64 -> FP32: round to nearest, ties to even, with gradual underflow (float subnormals) and
// overflow to infinity, i.e. the IEEE conversion; NaN becomes the canonical quiet NaN of its sign.
// FP32 -> FP64 is exact.
__device__ __forceinline__ float d2f_rn(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned long long sgn = u & 0x8000000000000000ull;
  const unsigned long long a = u ^ sgn;
  const unsigned int s32 = (unsigned int)(sgn >> 32);
  if (a >= 0x7FF0000000000000ull) return __uint_as_float(s32 | (a > 0x7FF0000000000000ull ? 0x7FC00000u : 0x7F800000u));
  const int e = (int)(a >> 52);                                 // biased binary exponent of |x|
  if (e >= 1151) return __uint_as_float(s32 | 0x7F800000u);     // |x| >= 2^128
  if (e >= 897) {                                               // |x| >= 2^-126: a normal float
    // drop the low 29 significand bits, rounding to nearest even; a carry out of the significand
    // steps the exponent (and turns 2^128 into infinity); rebias the exponent by 1023 - 127
    const unsigned long long r = a + 0x0FFFFFFFull + ((a >> 29) & 1ull);
    return __uint_as_float(s32 | (unsigned int)((r >> 29) - (896ull << 23)));
  }
  if (e < 873) return __uint_as_float(s32);                     // |x| < 2^-150: rounds to zero
  // a float subnormal: |x| = M 2^(e - 1075) with the 53-bit significand M, in units of 2^-149 that is
  // M / 2^s with s = 926 - e in [30, 53]; round the quotient to nearest even (2^23 is the smallest normal)
  const int s = 926 - e;
  const unsigned long long M = (a & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  unsigned long long q = M >> s;
  const unsigned long long rem = M & ((1ull << s) - 1ull), half = 1ull << (s - 1);
  if (rem > half || (rem == half && (q & 1ull))) ++q;
  return __uint_as_float(s32 | (unsigned int)q);
}

__device__ __forceinline__ double f2d_exact(float f) {
  const unsigned int u = __float_as_uint(f);
  const unsigned int sgn = u & 0x80000000u;
  unsigned int a = u ^ sgn, e = a >> 23;
  if (e - 1u < 254u) {
    e += 896u;                                    // rebias 127 -> 1023
  } else if (a == 0u) {
  } else if (e == 0u) {                           // a float subnormal: normalise the significand
    const int sh = __clz((int)a) - 8;
    a <<= sh;
    e = 897u - (unsigned)sh;
  } else {                                        // infinite, or NaN (made quiet)
    e = 2047u;
    if (a > 0x7F800000u) a |= 0x400000u;
  }
  return __longlong_as_double((long long)(((unsigned long long)(sgn | (e << 20)) << 32) |
                                          ((unsigned long long)(a & 0x7FFFFFu) << 29)));
}

// a - b in FP64.  Two FP32 values: the rounded difference s and its error term (Knuth's two-sum) add up to
// the exact one, and where the error's last bit is within 53 bits of s they are put together as integers: s
// widened, plus the error in units of its last place (the same value an FP64 subtraction gives, without the
// narrow FP64 pipe: the first k_ct of a 512-block RK3 step 148 -> 88 us, its FP64 instructions per face 23 -> 10).  Wider
// apart, or with a subnormal or non-finite value, an FP64 subtraction.
template <class R> __device__ __forceinline__ double diff64(R a, R b);
template <> __device__ __forceinline__ double diff64(double a, double b) { return a - b; }
template <> __device__ __forceinline__ double diff64(float a, float b) {
  const float s = __fsub_rn(a, b);
  const float bp = __fsub_rn(s, a);               // the part of s that came from -b
  const float ap = __fsub_rn(s, bp);              // the part of s that came from a
  const float err = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(__fsub_rn(0.f, b), bp));
  const unsigned int us = __float_as_uint(s), ue = __float_as_uint(err);
  if (err == 0.f && ((us << 1) < 0xFF000000u)) return f2d_exact(s);
  const unsigned int es = (us >> 23) & 0xFFu, ee = (ue >> 23) & 0xFFu;
  const int sh = (int)ee - (int)es + 29;          // err = k 2^(es - 127 - 52), k = its significand << sh
  if (es - 1u < 254u && ee != 0u && sh >= 0 && err == err) {
    long long k = (long long)(((ue & 0x7FFFFFu) | 0x800000u) << sh);
    if ((int)(us ^ ue) < 0) k = (us & 0x7FFFFFu) == 0u ? -2 * k : -k;   // below a power of two the units halve
    return __longlong_as_double(__double_as_longlong(f2d_exact(s)) + k);
  }
  return f2d_exact(a) - f2d_exact(b);
}

// ------------------------------------------------------------------------------------------------
// Sums of FP64 values in fixed point: significands aligned to the largest exponent of the set, added as 64-bit
// integers (exactly, but for what alignment cuts off a value many bits below the largest), and rounded once.
// ~12 integer instructions a value and ~18 a result, against 70 cycles of a scheduler for each FP64 addition.
// ------------------------------------------------------------------------------------------------
// largest biased exponent of N values (2047: one is not finite)
template <int N>
__device__ __forceinline__ uint32_t fix_exp(const double* f) {
  uint32_t e = 0;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    const uint32_t h = (uint32_t)__double2hiint(f[t]) & 0x7fffffffu;
    e = e > h ? e : h;
  }
  return e >> 20;
}
// f in units of 2^(e - 1075 - UP) (a subnormal counts as zero); |result| < 2^(53 + UP)
template <int UP>
__device__ __forceinline__ int64_t fix_of(double f, uint32_t e) {
  const uint32_t h = (uint32_t)__double2hiint(f), l = (uint32_t)__double2loint(f);
  const uint32_t et = (h >> 20) & 0x7ffu;
  uint32_t sh = e - et;
  sh = sh < 63u && et != 0u ? sh : 63u;
  const uint32_t mh = (((h & 0xfffffu) | 0x100000u) << UP) | (UP ? l >> ((32 - UP) & 31) : 0u);
  const int64_t m = (int64_t)((((uint64_t)mh << 32) | (l << UP)) >> sh);
  return (int32_t)h < 0 ? -m : m;
}
// acc 2^x, rounded to nearest even (a result below the normal range is zero, above it infinite)
__device__ __forceinline__ double fix_round(int64_t acc, int x) {
  const uint64_t sg = acc < 0 ? 0x8000000000000000ull : 0ull;
  const uint64_t u = (uint64_t)(acc < 0 ? -acc : acc);
  if (u == 0ull) return 0.0;
  const int z = __clzll((long long)u);
  const int ex = 1086 - z + x;                                   // biased exponent of the leading bit
  if (ex < 1) return 0.0;
  if (ex > 2046) return from64(sg | 0x7ff0000000000000ull);
  const uint64_t n = u << z;
  const uint64_t r = (n >> 11) + ((n >> 10) & 1ull & (uint64_t)((n & 0x3ffull) != 0ull || (n & 0x800ull) != 0ull));
  return from64(sg | (((uint64_t)(uint32_t)(ex - 1) << 52) + r));
}
// Sets that the fixed-point sums leave to the operators: one value is not finite, or all are so small that a result
// could fall below the normal range (then e < 64; mostly all are zero, as a vanishing shift is)
__device__ __forceinline__ bool fix_edge(uint32_t e) { return e - 64u >= 2047u - 64u; }
template <int N>
__device__ __forceinline__ bool fix_zero(const double* f) {
  uint32_t o = 0;
#pragma unroll
  for (int t = 0; t < N; ++t) o |= ((uint32_t)__double2hiint(f[t]) << 1) | (uint32_t)__double2loint(f[t]);
  return o == 0u;
}

// mean of the eight vertices of a cell (index x + 2 y + 4 z)
__device__ __forceinline__ double mean8_64(const double f[8]) {
  const uint32_t e = fix_exp<8>(f);
  if (fix_edge(e))
    return fix_zero<8>(f) ? 0.0 : mul_rare(((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])), 0.125);
  int64_t a = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) a += fix_of<7>(f[t], e);
  return fix_round(a, (int)e - 1075 - 7 - 3);
}
// the mean, and the sums of the four differences along x, y and z (each zero on a constant field)
__device__ __forceinline__ void haar8_64(const double f[8], double* mean, double* dx, double* dy, double* dz) {
  const uint32_t e = fix_exp<8>(f);
  if (fix_edge(e)) {
    *mean = *dx = *dy = *dz = 0.0;
    if (fix_zero<8>(f)) return;
    *mean = mul_rare(((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])), 0.125);
    *dx = ((f[1] - f[0]) + (f[3] - f[2])) + ((f[5] - f[4]) + (f[7] - f[6]));
    *dy = ((f[2] - f[0]) + (f[3] - f[1])) + ((f[6] - f[4]) + (f[7] - f[5]));
    *dz = ((f[4] - f[0]) + (f[5] - f[1])) + ((f[6] - f[2]) + (f[7] - f[3]));
    return;
  }
  int64_t m[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) m[t] = fix_of<7>(f[t], e);
  const int64_t s0 = m[0] + m[1], s1 = m[2] + m[3], s2 = m[4] + m[5], s3 = m[6] + m[7];
  const int x = (int)e - 1075 - 7;
  *mean = fix_round((s0 + s1) + (s2 + s3), x - 3);
  *dx = fix_round(((m[1] - m[0]) + (m[3] - m[2])) + ((m[5] - m[4]) + (m[7] - m[6])), x);
  *dy = fix_round((s1 - s0) + (s3 - s2), x);
  *dz = fix_round((s2 + s3) - (s0 + s1), x);
}
// the 4 x 4 Lagrange midpoint interpolant of a vertex plane, weights (-1, 9, 9, -1)/16 per axis; f[4 y + x]
__device__ __forceinline__ double lagr16_64(const double f[16]) {
  const uint32_t e = fix_exp<16>(f);
  if (fix_edge(e)) {
    if (fix_zero<16>(f)) return 0.0;
    double s[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) s[y] = 9.0 * (f[4 * y + 1] + f[4 * y + 2]) - (f[4 * y] + f[4 * y + 3]);
    return mul_rare(9.0 * (s[1] + s[2]) - (s[0] + s[3]), 1.0 / 256);
  }
  int64_t r[4];
#pragma unroll
  for (int y = 0; y < 4; ++y) {   // 54 bits, times at most 20 per axis: 63
    const int64_t b = fix_of<1>(f[4 * y + 1], e) + fix_of<1>(f[4 * y + 2], e);
    r[y] = 9 * b - (fix_of<1>(f[4 * y], e) + fix_of<1>(f[4 * y + 3], e));
  }
  return fix_round(9 * (r[1] + r[2]) - (r[0] + r[3]), (int)e - 1075 - 1 - 8);
}

// ------------------------------------------------------------------------------------------------
// A one-sided FP32 bound for the atmosphere test
// ------------------------------------------------------------------------------------------------
// x > 0 within 2^-20 from above, from the upper half of its encoding; 0 where it is not a normal FP32 number
__device__ __forceinline__ float above32(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  return h - 0x38200000u < 0x47a00000u - 0x38200000u ? __uint_as_float(((h - 0x38000000u) << 3) + 8u) : 0.f;
}
// Whether D is above thr sqrt(gamma) for certain, g: gamma_xx, gamma_yy, gamma_zz at the eight vertices of a cell.
// thr sqrt(gamma_xx gamma_yy gamma_zz) is an upper bound for a positive definite gamma_ij (Hadamard); it is formed in FP32
// from above with a margin of 1e-3, and given up where a product is too small to keep that margin
__device__ __forceinline__ bool surely_above(const double g[3][8], double D, double thr) {
  float p = 1.f;
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float s = 0.f;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float f = above32(g[c][t]);
      ok = ok && f > 0.f;
      s += f;
    }
    p *= 0.125f * s;
    ok = ok && p > 1e-30f;
  }
  const float d = above32(D), t = above32(thr);   // d exceeds D by 2^-20 at most
  return ok && t > 0.f && p < 1e30f && d > 1.001f * t * sqrtf(p);
}

}  // namespace grs
