// Host build of csrc/castlist.h: every combination of EOS, extrinsic curvature and caller's FP32 copies lists each pool
// that the stage then reads in FP32 once, with its own destination and length, and no entry of one array runs into another.
// Prints "bad N most M room R": wrong lists, the longest list, the list's capacity.
#include <cstdio>
#include <cstdint>
#include "castlist.h"
using namespace grs;

static double* D(long i) { return reinterpret_cast<double*>(0x100000L + 64 * i); }
static float* F(long i) { return reinterpret_cast<float*>(0x900000L + 64 * i); }

int main() {
  int bad = 0, most = 0;
  for (int mask = 0; mask < 32; ++mask) {
    const int eos = mask & 1 ? GR_EOS_TABLE : GR_EOS_IDEAL;
    const bool kz = mask & 2, w32 = mask & 4, m32 = mask & 8, cast = mask & 16;
    MetricView m{};
    StateView s{};
    Shadow sh{};
    m.k_zero = kz;
    for (int c = 0; c < 16; ++c) { m.v[c] = D(100 + c); sh.M[c] = F(100 + c); if (m32) m.v32[c] = F(500 + c); }
    for (int q = 0; q < 7; ++q) s.W[q] = D(q);
    for (int q = 0; q < 6; ++q) { sh.W[q] = F(q); if (w32) s.W32[q] = F(400 + q); }
    for (int d = 0; d < 3; ++d) { s.B[d] = D(50 + d); sh.B[d] = F(50 + d); sh.nface[d] = 1000 + d; if (w32) s.B32[d] = F(450 + d); }
    sh.ncell = 77;
    sh.nvert = 99;
    CastList L;
    if (!stage_casts(m, s, sh, eos, cast, L)) ++bad;
    int want = 0;
    auto has = [&](const double* a, float* b, long long n) {
      ++want;
      int seen = 0;
      for (int k = 0; k < L.count && k < CastList::kMax; ++k) seen += L.src[k] == a && L.dst[k] == b && L.n[k] == n;
      bad += seen != 1;
    };
    if (!w32) {
      for (int q = 0; q < (eos == GR_EOS_TABLE ? 6 : 5); ++q) has(D(q), F(q), 77);
      for (int d = 0; d < 3; ++d) has(D(50 + d), F(50 + d), 1000 + d);
    }
    for (int c = 0; cast && !m32 && c < (kz ? 10 : 16); ++c) has(D(100 + c), F(100 + c), 99);
    bad += L.count != want;
    most = L.count > most ? L.count : most;
  }
  // a full list refuses the next pool and is not changed by it
  CastList L{};
  for (int k = 0; k < CastList::kMax; ++k) bad += !L.add(D(k), F(k), k + 1);
  bad += L.add(D(900), F(900), 5) || L.count != CastList::kMax;
  for (int k = 0; k < CastList::kMax; ++k) bad += L.src[k] != D(k) || L.dst[k] != F(k) || L.n[k] != k + 1;
  std::printf("bad %d most %d room %d\n", bad, most, CastList::kMax);
  return 0;
}
