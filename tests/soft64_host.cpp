// Host build of csrc/soft64.cuh: its integer arithmetic against the IEEE operations of this CPU, over random
// operands, all exponents, and significands at the ends of their range.  The FP32 approximations are perturbed by
// up to two units in the last place, more than the hardware's own error.  Prints "bad N" and the largest rsqrt error.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#define __device__
#define __forceinline__ inline
template <class T, class U> static T as(U u) { T t; static_assert(sizeof t == sizeof u, ""); memcpy(&t, &u, sizeof t); return t; }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) { return (unsigned long long)(((unsigned __int128)a * b) >> 64); }
static inline float __uint_as_float(unsigned u) { return as<float>(u); }
static inline unsigned __float_as_uint(float f) { return as<unsigned>(f); }
static inline long long __double_as_longlong(double d) { return as<long long>(d); }
static inline double __longlong_as_double(long long u) { return as<double>(u); }
static inline int __double2hiint(double d) { return (int)(as<unsigned long long>(d) >> 32); }
static inline int __double2loint(double d) { return (int)as<unsigned long long>(d); }
static inline unsigned __funnelshift_r(unsigned lo, unsigned hi, int s) { return (unsigned)((((unsigned long long)hi << 32) | lo) >> s); }
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline double rsqrt(double x) { return 1 / std::sqrt(x); }
#include "soft64.cuh"

static std::mt19937_64 rng(2311);
static float off(float y) { return as<float>(as<unsigned>(y) + (unsigned)((int)(rng() % 5) - 2)); }
namespace grs {
float rcp_apx(float x) { return std::fmin(std::fmax(off(1.0f / x), 0.5f), std::nextafter(1.0f, 0.0f)); }
float rsqrt_apx(float x) { return std::fmin(std::fmax(off((float)(1.0 / std::sqrt((double)x))), 0.5f), std::nextafter(1.0f, 0.0f)); }
}
using namespace grs;

static double draw(bool near1) {
  unsigned long long m = rng();
  switch (rng() % 6) {
    case 0: m &= ~0ull << (rng() % 53); break;
    case 1: m |= (1ull << (rng() % 53)) - 1; break;
    case 2: m = rng() % 64; break;
    case 3: m = 0xFFFFFFFFFFFFFull - rng() % 64; break;
    default: break;
  }
  const unsigned long long e = near1 ? 983 + rng() % 80 : rng() % 2048;
  return as<double>(((rng() & 1) << 63) | (e << 52) | (m & 0xFFFFFFFFFFFFFull));
}
static float drawf(bool near1) {
  unsigned m = (unsigned)rng() & 0x7FFFFFu;
  if (rng() % 4 == 0) m &= ~0u << (rng() % 23);
  return as<float>(((unsigned)(rng() & 1) << 31) | ((near1 ? 120u + (unsigned)(rng() % 16) : (unsigned)(rng() % 256)) << 23) | (m & 0x7FFFFFu));
}
static bool same(double a, double b) { return a != a ? b != b : (a == b && std::signbit(a) == std::signbit(b)); }

int main(int, char** v) {
  const long n = atol(v[1]);
  long bad = 0;
  double worst = 0;
  for (long i = 0; i < n; ++i) {
    double a = draw(i & 1), b = draw(i & 1);
    if (i % 7 == 0) a = b * (double)(int)(rng() % 1000);
    if (i % 11 == 0) a *= 0.0;
    bad += !same(div64(a, b), a / b) || !same(mul64(a, b), a * b);
    bad += gt64(a, b) != (a > b) || gt64(a, a) || gt64(b, b);
    bad += neg64(a) != (a < 0) || zero64(a) != (a == 0) || finite64(a) != std::isfinite(a);
    if (b >= 0) bad += gtp64(a, b) != (a > b) || gtp64(b, b) != (b > b);
    double x = std::fabs(draw(i & 1));
    if (i % 5 == 0) x *= x;
    bad += !same(sqrt64(x), std::sqrt(x)) || !same(sqrt64(-x), std::sqrt(-x));
    if (std::isnormal(x)) {
      const long double z = 1 / sqrtl((long double)x);
      const double zd = (double)z, ulp = std::nextafter(zd, INFINITY) - zd;
      worst = std::fmax(worst, std::fabs((double)((long double)rsqrt64(x) - z)) / ulp);
    }
    float f = drawf(i % 3), g = drawf(i % 3);
    if (i % 7 == 0) g = as<float>(as<unsigned>(f) + (unsigned)((int)(rng() % 64) - 32));
    if (i % 101 == 0) g = f;
    bad += !same(diff64(f, g), (double)f - (double)g) || !same(f2d_exact(f), (double)f);
    double w[8], big = 0;
    long double sum = 0;
    for (int t = 0; t < 8; ++t) {
      const unsigned long long e = i % 4 == 0 ? 1023 : i % 4 == 1 ? 1020 + rng() % 6 : i % 4 == 2 ? 1000 + rng() % 40 : 1022;
      unsigned long long m = rng() & 0xFFFFFFFFFFFFFull;
      if (i % 4 == 3) m |= 0xFFF0000000000ull;
      w[t] = rng() % 50 ? as<double>((i % 4 == 3 ? 0 : (rng() & 1) << 63) | (e << 52) | m) : 0.0;
      sum += w[t];
      big = std::fmax(big, std::fabs(w[t]));
    }
    const double mean = (double)(sum / 8);
    // each addend cut below 2^-59 of the largest, one rounding
    const double lim = std::ldexp(big, -58) + 0.502 * (std::nextafter(std::fabs(mean), INFINITY) - std::fabs(mean));
    bad += !(std::fabs((double)((long double)mean8_64(w) - sum / 8)) <= lim);
    // the differences: each addend cut below 2^-59 of the largest, one rounding; the plane: 2^-53 of the largest
    double hm, hd[3];
    haar8_64(w, &hm, hd, hd + 1, hd + 2);
    bad += !same(hm, mean8_64(w));
    for (int d = 0; d < 3; ++d) {
      long double z = 0;
      for (int q = 0; q < 8; ++q) z += (q >> d & 1) ? (long double)w[q] : -(long double)w[q];
      const double zd = std::fabs((double)z);
      bad += !(std::fabs((double)((long double)hd[d] - z)) <= std::ldexp(big, -55) + 0.502 * (std::nextafter(zd, INFINITY) - zd));
    }
    double pl[16], pb = 0;
    long double ps = 0;
    const long double wt[4] = {-1 / 16.0L, 9 / 16.0L, 9 / 16.0L, -1 / 16.0L};
    for (int q = 0; q < 16; ++q) {
      pl[q] = w[rng() % 8] * (1 + 1e-3 * (double)(rng() % 100));
      ps += wt[q & 3] * wt[q >> 2] * pl[q];
      pb = std::fmax(pb, std::fabs(pl[q]));
    }
    const double pd = std::fabs((double)ps);
    // sixteen cuts of 2^-53 of the largest with weights that add up to 25/16, one rounding
    bad += !(std::fabs((double)((long double)lagr16_64(pl) - ps)) <= std::ldexp(pb, -53) * 1.5625 * 1.01 + 0.502 * (std::nextafter(pd, INFINITY) - pd));
  }
  printf("bad %ld rsqrt %.4f\n", bad, worst);
  return 0;
}
