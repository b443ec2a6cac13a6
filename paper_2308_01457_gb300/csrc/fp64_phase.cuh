// exp(i theta) in FP64 for the regular-pair kernels, from a table in shared memory.
//
// FP64 issues one warp instruction per 16 clocks and SM, so these kernels are bound by the
// number of FP64 instructions: theta = n pi/64 + d with |d| <= pi/128 leaves three terms of
// each series, 18 FP64 instructions against about 45 of sincos.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

namespace fosb {

constexpr int kPhaseTab = 128;  // cos and sin of j pi/64

inline void make_phase_table(double (&tab)[kPhaseTab][2]) {
  for (int j = 0; j < kPhaseTab; ++j) {
    const long double a = j * (3.14159265358979323846264338327950288L / 64);
    tab[j][0] = double(std::cos(a));
    tab[j][1] = double(std::sin(a));
  }
}

// theta >= 0.  n is taken from the low bits of theta 64/pi + 1.5 2^52; pi/64 = c1 + c2 with c1 a
// double: n c1 and theta are multiples of 2^-57 (of 2^-52 theta below one), so the first FMA is
// exact up to theta near 2^20, and the table's index stays right far beyond.
__device__ __forceinline__ void expi_table(double theta, const double2* tab, double& cs, double& sn) {
  constexpr double kMagic = 6755399441055744.0;
  const double t = fma(theta, 20.371832715762604, kMagic);
  const double n = t - kMagic;
  const double2 T = tab[__double2loint(t) & (kPhaseTab - 1)];
  double d = fma(-n, 0.04908738521234052, theta);
  d = fma(-n, 1.9135106236677394e-18, d);
  const double d2 = d * d;
  const double sd = fma(d * d2, fma(d2, fma(d2, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), d);
  const double cm = d2 * fma(d2, fma(d2, -1.0 / 720.0, 1.0 / 24.0), -0.5);  // cos d - 1
  cs = T.x + fma(T.x, cm, -T.y * sd);
  sn = T.y + fma(T.y, cm, T.x * sd);
}

}  // namespace fosb
