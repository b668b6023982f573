// Host build of csrc/soft64.cuh: the fixed-point sums of FP64 sets at the ends of the range -- an infinite or NaN value, all
// values subnormal or just above, all zero -- against the same sums by the operators.  Prints "bad N".
#include <cmath>
#include <cstdio>
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
namespace grs {
float rcp_apx(float x) { return 1.0f / x; }
float rsqrt_apx(float x) { return 1.0f / std::sqrt(x); }
}
using namespace grs;

static bool same(double a, double b) { return a != a ? b != b : a == b; }
// equal, or within what the sums are allowed elsewhere: a cut of 2^-53 of the largest (1.5625 of them in a plane) and a rounding
static bool near(double a, long double z, double big) {
  const double d = (double)z;
  if (!std::isfinite(d) || !std::isfinite(a)) return same(a, d);
  const double ulp = std::nextafter(std::fabs(d), INFINITY) - std::fabs(d);
  return std::fabs((double)((long double)a - z)) <= 1.6 * std::ldexp(big, -53) + 0.502 * ulp;
}

int main() {
  std::mt19937_64 rng(64);
  long bad = 0;
  const double edge[] = {INFINITY, -INFINITY, NAN, 4.9e-324, 1e-310, 2.2250738585072014e-308};
  for (int it = 0; it < 200000; ++it) {
    double f[16];
    // 0: ordinary values and one edge value; 1: all subnormal; 2: exponents 1 .. 80; 3: all zero of either sign; 4: huge
    const int kind = it % 5;
    for (double& v : f) {
      const unsigned long long m = rng() & 0xFFFFFFFFFFFFFull, s = (rng() & 1) << 63;
      const unsigned long long e = kind == 0 ? 1000 + rng() % 40 : kind == 1 ? 0 : kind == 2 ? 1 + rng() % 80 : 2030 + rng() % 10;
      v = kind == 3 ? as<double>(s) : as<double>(s | (e << 52) | m);
    }
    if (kind == 0) f[rng() % 16] = edge[rng() % 6];
    double big = 0;
    for (double v : f) big = std::fmax(big, std::isfinite(v) ? std::fabs(v) : 0.0);
    long double s8 = 0, d8[3] = {0, 0, 0}, pl = 0;
    for (int t = 0; t < 8; ++t) {
      s8 += f[t];
      for (int d = 0; d < 3; ++d) d8[d] += (t >> d & 1) ? (long double)f[t] : -(long double)f[t];
    }
    const long double w[4] = {-1 / 16.0L, 9 / 16.0L, 9 / 16.0L, -1 / 16.0L};
    for (int t = 0; t < 16; ++t) pl += w[t & 3] * w[t >> 2] * (long double)f[t];
    double m, dx, dy, dz;
    haar8_64(f, &m, &dx, &dy, &dz);
    bad += !same(m, mean8_64(f)) || !near(m, s8 / 8, big);
    bad += !near(dx, d8[0], 8 * big) || !near(dy, d8[1], 8 * big) || !near(dz, d8[2], 8 * big);
    bad += !near(lagr16_64(f), pl, 4 * big);
  }
  std::printf("bad %ld\n", bad);
  return 0;
}
