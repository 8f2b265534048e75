// Which grids tensor generation may treat through an integer argument
// (tensor_gen.cu): host code without device dependencies.
#pragma once
#include <cmath>

namespace fsa {

// Integers r_j with s_j^2 = base^2 r_j, and the table length sum_j r_j n_j^2 + 1.
struct Radial {
  double base;
  int r[3];
  long long size;
};

// s: three steps (mesh steps, or pi / (2 L_j)), each the same multiple of
// num / den, those two being exact.  False where no base s_min / m, m <= 3,
// gives integers or the table would hold more than a quarter of the octant's
// `total` points (more evaluations saved than made, and room for two tables in
// the octant).
//
// The ratios are compared in extended precision, so what is left of a
// difference from an integer is the box's own: half-widths that are rounded
// multiples of one length (2^-53 each) put a squared ratio within 4 * 2^-53 of
// its integer, and a table then moves r by at most 2 * 2^-53, as much as the
// per-point evaluation rounds.  Any other box is not radial.  (Extended
// precision is software on the Arm hosts, 4 us for a grid: the ratios in
// double, off by 8 * 2^-53 at most, sort out most grids without it.)
inline bool radial_of(const double* s, const double* num, const double* den, const int* n, long long total,
                      Radial* out) {
  int lo = 0;
  for (int j = 1; j < 3; ++j)
    if (s[j] < s[lo]) lo = j;
  for (int m = 1; m <= 3; ++m) {
    out->base = s[lo] / m;
    long long size = 1;
    bool ok = true;
    for (int j = 0; j < 3 && ok; ++j) {
      const double q = s[j] / s[lo], v = q * q * (m * m), rv = std::nearbyint(v);
      ok = std::fabs(v - rv) <= 4e-15 * rv && rv * n[j] * n[j] < 1e9;
      if (ok) {
        out->r[j] = (int)rv;
        size += (long long)rv * n[j] * n[j];
      }
    }
    if (!ok || size > total / 4) continue;
    for (int j = 0; j < 3 && ok; ++j) {
      const long double q = (long double)num[j] * den[lo] / ((long double)den[j] * num[lo]), r = out->r[j];
      ok = fabsl(q * q * (m * m) - r) <= 4.5e-16L * r;
    }
    if (ok) {
      out->size = size;
      return true;
    }
  }
  return false;
}

}  // namespace fsa
