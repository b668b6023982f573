// Host build of csrc/soft64.cuh: surely_above, the FP32 bound by which gr_con2prim's first pass queues a cell, against the
// exact test D >= thr sqrt(gamma) over random positive definite metrics of all scales and D around the threshold.
// Prints "wrong N missed M fired F": cells queued below the threshold, cells well above the bound that were not queued
// although every product is in range, cells queued.
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


int main() {
  std::mt19937_64 rng(2311);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  long wrong = 0, missed = 0, fired = 0;
  for (int it = 0; it < 3000000; ++it) {
    // gamma = L L^T at a centre, vertices a little off it; scales 1e-16 .. 1e12, each axis its own in half of them
    const double s0 = std::pow(10.0, -16 + 28 * u(rng));
    double sc[3];
    for (double& v : sc) v = it & 1 ? s0 : s0 * std::pow(10.0, -6 + 12 * u(rng));
    const double l10 = it & 2 ? 0.0 : 2 * u(rng) - 1, l20 = it & 2 ? 0.0 : 2 * u(rng) - 1, l21 = it & 2 ? 0.0 : 2 * u(rng) - 1;
    const double d0 = 0.1 + u(rng), d1 = 0.1 + u(rng), d2 = 0.1 + u(rng), amp = it % 3 ? 1e-3 : 0.0;
    const double G[6] = {d0 * d0, d0 * l10, d0 * l20, l10 * l10 + d1 * d1, l10 * l20 + d1 * l21, l20 * l20 + l21 * l21 + d2 * d2};
    static const int I[6] = {0, 0, 0, 1, 1, 2}, J[6] = {0, 1, 2, 1, 2, 2};
    double g[3][8];
    long double m[6] = {0, 0, 0, 0, 0, 0};
    for (int t = 0; t < 8; ++t) {
      const double f = 1 + amp * u(rng);   // a common factor keeps every vertex positive definite
      for (int c = 0; c < 6; ++c) {
        const double v = G[c] * f * std::sqrt(sc[I[c]] * sc[J[c]]);
        m[c] += v / 8.0L;
        if (I[c] == J[c]) g[I[c]][t] = v;
      }
    }
    const long double det = m[0] * (m[3] * m[5] - m[4] * m[4]) - m[1] * (m[1] * m[5] - m[4] * m[2]) + m[2] * (m[1] * m[4] - m[3] * m[2]);
    const double thr = std::pow(10.0, -20 + 20 * u(rng));
    const double at = thr * (double)sqrtl(det), bound = thr * (double)sqrtl(m[0] * m[3] * m[5]);
    const double D = at * (it % 5 == 0 ? 1 - std::pow(10.0, -6 * u(rng)) : std::pow(10.0, -1 + 4 * u(rng)));
    const bool q = surely_above(g, D, thr);
    fired += q;
    wrong += q && D < at;
    const double lim = 1e-28;
    const bool ranged = m[0] > lim && m[0] * m[3] > lim && m[0] * m[3] * m[5] > lim && m[0] * m[3] * m[5] < 1e29 && D > 1e-37;
    missed += !q && ranged && D > 1.002 * bound;
  }
  std::printf("wrong %ld missed %ld fired %ld\n", wrong, missed, fired);
  return 0;
}
