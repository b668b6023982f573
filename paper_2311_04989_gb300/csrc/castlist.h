// castlist.h -- the FP64 -> FP32 conversions of a mixed stage as one list for k_cast (host side, no CUDA calls)
#pragma once

#include "internal.h"

namespace grs {

// Pools to convert in one launch.  The fullest stage needs every entry of the input view: a table (six W pools), B, and
// the metric with K_ij, none with a caller's FP32 copy.
struct CastList {
  static constexpr int kW = 6, kB = 3, kM = 16;
  static constexpr int kMax = kW + kB + kM;
  const double* src[kMax];
  float* dst[kMax];
  long long n[kMax];
  int count;
  // false, and nothing written, when the list is full
  bool add(const double* s, float* d, long long m) {
    if (count < 0 || count >= kMax) return false;
    src[count] = s;
    dst[count] = d;
    n[count] = m;
    ++count;
    return true;
  }
};
static_assert(sizeof(InView<float>::W) / sizeof(float*) == CastList::kW && sizeof(InView<float>::B) / sizeof(float*) == CastList::kB &&
                  sizeof(InView<float>::M) / sizeof(float*) == CastList::kM,
              "CastList must hold every pool of a stage's inputs");

// The conversions a mixed stage needs: W and B unless the caller gave copies, the metric unless the caller gave one or
// (cast_metric = false) the previous stage on this mesh made it.  False if they do not fit.
inline bool stage_casts(const MetricView& m, const StateView& s, const Shadow& sh, int eos, bool cast_metric, CastList& L) {
  L = CastList{};
  bool ok = true;
  if (!s.W32[0]) {
    const int nw = eos == GR_EOS_TABLE ? 6 : 5;   // rho, u~^i, p[, Y_e]
    for (int q = 0; q < nw; ++q) ok = ok && L.add(s.W[q], sh.W[q], sh.ncell);
    for (int d = 0; d < 3; ++d) ok = ok && L.add(s.B[d], sh.B[d], sh.nface[d]);
  }
  const int ncomp = (cast_metric && !m.v32[0]) ? (m.k_zero ? 10 : 16) : 0;
  for (int c = 0; c < ncomp; ++c) ok = ok && L.add(m.v[c], sh.M[c], sh.nvert);
  return ok;
}

}  // namespace grs
