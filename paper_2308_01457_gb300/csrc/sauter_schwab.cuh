// What the touching-pair kernels share: the tables of the Sauter-Schwab rule in the form
// (x, y) = xi (xh, yh) (built on the host) and the warp-level pieces.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <vector>

#include "fosb_internal.h"

namespace fosb {

constexpr int kSsMaxNss = 12;   // largest n_ss an entry point accepts
constexpr int kSsRegions = 13;  // 6 identical, 5 common edge, 2 common vertex, in this order
constexpr int kSsFields = 11;   // u1, u2, v1, v2, weight, u1v1, u1v2, u2v1, u2v2, u1 - v1, u2 - v2
constexpr int kSsTerms = 16;    // powers of phi^2 in the series: more than phi = 3 needs

// g_ss_table's contents for r.nss points per coordinate: field f of point (region, e1, e2, e3) at
// f * (13 n^3) + region * n^3 + (e1 n + e2) n + e3, with xh = u1 (P1 - P0) + u2 (P2 - P1), yh the
// same in v, and the weight of the three coordinates with every Jacobian factor but xi^3.
inline std::vector<double> make_ss_table(const Rules& r) {
  const int n = r.nss, n3 = n * n * n;
  std::vector<double> tab(size_t(kSsFields) * kSsRegions * n3);
  for (int i1 = 0; i1 < n; ++i1)
    for (int i2 = 0; i2 < n; ++i2)
      for (int i3 = 0; i3 < n; ++i3) {
        const double a = r.glx[i1], b = r.glx[i2], c = r.glx[i3], w = r.glw[i1] * r.glw[i2] * r.glw[i3];
        const double w3 = w * a * a * b, w2 = w * a * a, w2b = w2 * b, w1 = w * b;
        const double s[kSsRegions][5] = {
            {1, 1 - a + a * b, 1 - a * b * c, 1 - a, w3},
            {1 - a * b * c, 1 - a, 1, 1 - a + a * b, w3},
            {1, a * (1 - b + b * c), 1 - a * b, a * (1 - b), w3},
            {1 - a * b, a * (1 - b), 1, a * (1 - b + b * c), w3},
            {1 - a * b * c, a * (1 - b * c), 1, a * (1 - b), w3},
            {1, a * (1 - b), 1 - a * b * c, a * (1 - b * c), w3},
            {1, a * c, 1 - a * b, a * (1 - b), w2},
            {1, a, 1 - a * b * c, a * b * (1 - c), w2b},
            {1 - a * b, a * (1 - b), 1, a * b * c, w2b},
            {1 - a * b * c, a * b * (1 - c), 1, a, w2b},
            {1 - a * b * c, a * (1 - b * c), 1, a * b, w2b},
            {1, a, b, b * c, w1},
            {b, b * c, 1, a, w1}};
        // u1 - v1 and u2 - v2 of the identical and edge regions, without cancellation
        const double d[kSsRegions][2] = {
            {a * b * c, a * b},  {-a * b * c, -a * b},          {a * b, a * b * c},
            {-a * b, -a * b * c}, {-a * b * c, a * b * (1 - c)}, {a * b * c, -a * b * (1 - c)},
            {a * b, 0},          {a * b * c, 0},                {-a * b, 0},
            {-a * b * c, 0},     {-a * b * c, 0},               {0, 0},
            {0, 0}};
        for (int q = 0; q < kSsRegions; ++q) {
          const double f[kSsFields] = {s[q][0], s[q][1], s[q][2], s[q][3], s[q][4], s[q][0] * s[q][2],
                                       s[q][0] * s[q][3], s[q][1] * s[q][2], s[q][1] * s[q][3], d[q][0], d[q][1]};
          const size_t at = size_t(q) * n3 + (size_t(i1) * n + i2) * n + i3;
          for (int k = 0; k < kSsFields; ++k) tab[size_t(k) * kSsRegions * n3 + at] = f[k];
        }
      }
  return tab;
}

// Coefficients of S_m(phi) = sum_a w_a xi_a^{2+m} exp(i phi xi_a), m = 0, 1, 2: with M_n the rule's
// moment of xi^n, Re S_m = sum_j (-1)^j M_{2+m+2j}/(2j)! phi^{2j} (c[j][m]) and
// Im S_m = phi sum_j (-1)^j M_{3+m+2j}/(2j+1)! phi^{2j} (c[j][3+m]).
inline void make_ss_series(const Rules& r, double (&c)[kSsTerms][6]) {
  auto moment = [&](int n) {
    long double s = 0;
    for (int a = 0; a < r.nss; ++a) s += (long double)r.glw[a] * std::pow((long double)r.glx[a], n);
    return s;
  };
  long double fact = 1;  // (2j)!
  for (int j = 0; j < kSsTerms; ++j) {
    if (j > 0) fact *= (long double)(2 * j - 1) * (2 * j);
    const long double sg = j & 1 ? -1 : 1;
    for (int m = 0; m < 3; ++m) {
      c[j][m] = double(sg * moment(2 + m + 2 * j) / fact);
      c[j][3 + m] = double(sg * moment(3 + m + 2 * j) / (fact * (2 * j + 1)));
    }
  }
}

// The same for Q_m(phi) = sum_a w_a xi_a^m (i phi xi_a - 1) exp(i phi xi_a), m = 1 .. MM, the xi sums
// of exp(ikr)(ikr - 1)/r^3: Re Q_m = sum_j (-1)^j (2j-1)/(2j)! M_{m+2j} phi^{2j} (c[j][m-1]) and
// Im Q_m = phi sum_j (-1)^j 2j/(2j+1)! M_{m+2j+1} phi^{2j} (c[j][MM+m-1]).
template <int MM>
inline void make_ss_series_mfio(const Rules& r, double (&c)[kSsTerms][2 * MM]) {
  auto moment = [&](int n) {
    long double s = 0;
    for (int a = 0; a < r.nss; ++a) s += (long double)r.glw[a] * std::pow((long double)r.glx[a], n);
    return s;
  };
  long double fact = 1;  // (2j)!
  for (int j = 0; j < kSsTerms; ++j) {
    if (j > 0) fact *= (long double)(2 * j - 1) * (2 * j);
    const long double sg = j & 1 ? -1 : 1;
    for (int m = 1; m <= MM; ++m) {
      c[j][m - 1] = double(sg * (2 * j - 1) * moment(m + 2 * j) / fact);
      c[j][MM + m - 1] = double(sg * 2 * j * moment(m + 1 + 2 * j) / (fact * (2 * j + 1)));
    }
  }
}

// The table on the current device (assemble.cu), nullptr if it cannot be had.
const double* ss_table_device();

// 1/sqrt(x) for a normal x > 0: the hardware's FP64 seed (about 20 bits) and one third-order step,
// y <- y + y e (1/2 + 3/8 e) with e = 1 - x y^2, which leaves an error of order e^3.
__device__ __forceinline__ double ss_rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// Upper bound of k |x - y| over the two triangles: attained between vertices, which are formed
// in FP32 from the edge vectors (P0 = Q0).
__device__ __forceinline__ float ss_phase_bound(double k, const double (&EP)[2][3], const double (&EQ)[2][3]) {
  float P[3][3], Q[3][3], m2 = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    P[0][c] = Q[0][c] = 0.f;
    P[1][c] = float(EP[0][c]);
    P[2][c] = P[1][c] + float(EP[1][c]);
    Q[1][c] = float(EQ[0][c]);
    Q[2][c] = Q[1][c] + float(EQ[1][c]);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float x = P[a][0] - Q[b][0], y = P[a][1] - Q[b][1], z = P[a][2] - Q[b][2];
      m2 = fmaxf(m2, x * x + y * y + z * z);
    }
  return float(k) * sqrtf(m2) * 1.0001f;
}

// The series up to here (its rounding is then below 6e-16 of |S_m|, 8e-16 at phase 4; 15 terms);
// larger phases, which only meshes with edges beyond about half a wavelength reach, take sincos per point.
constexpr double kSsMaxPhase = 3.0;

// Number of phi^2 powers for phases up to ph: the first J with ph^{2J}/(2J)! < 2^-56 (the
// moments' decay only helps), at most kSsTerms; 0 above kSsMaxPhase.
__device__ __forceinline__ int ss_terms(float ph) {
  if (!(ph <= float(kSsMaxPhase))) return 0;
  const float p2 = ph * ph;
  float t = 1.f;
  int J = 0;
  while (J < kSsTerms && t > 1.3e-17f) {
    t *= p2 / float((2 * J + 1) * (2 * J + 2));
    ++J;
  }
  return J;
}

// First region and number of regions of a kind of touching pair (3 identical, 2 edge, 1 vertex).
template <int KIND>
__device__ __forceinline__ constexpr int ss_first_region() {
  return KIND == 3 ? 0 : (KIND == 2 ? 6 : 11);
}
template <int KIND>
__device__ __forceinline__ constexpr int ss_regions() {
  return KIND == 3 ? 6 : (KIND == 2 ? 5 : 2);
}

// Difference xh - yh, distance and phase of one point of the table (field f at tab[f * stride]):
// 1/rh and k rh.
template <int KIND>
__device__ __forceinline__ void ss_distance(const double* tab, int stride, const double (&uv)[4],
                                            const double (&EP)[2][3], const double (&EQ)[2][3], double k,
                                            double (&d)[3], double& rinv, double& phi) {
  if constexpr (KIND == 3) {  // EQ = EP: the coordinate differences are in the table
    const double a = __ldg(tab + 9 * stride), b = __ldg(tab + 10 * stride);
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = fma(a, EP[0][c], b * EP[1][c]);
  } else if constexpr (KIND == 2) {  // EQ[0] = EP[0], the shared edge
    const double a = __ldg(tab + 9 * stride);
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = fma(a, EP[0][c], fma(uv[1], EP[1][c], -uv[3] * EQ[1][c]));
  } else {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      d[c] = fma(uv[0], EP[0][c], fma(uv[1], EP[1][c], fma(-uv[2], EQ[0][c], -uv[3] * EQ[1][c])));
  }
  const double r2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
  rinv = ss_rsqrt(r2);
  phi = k * (r2 * rinv);
}

__device__ __forceinline__ double ss_dot(const double (&x)[3], const double (&y)[3]) {
  return fma(x[0], y[0], fma(x[1], y[1], x[2] * y[2]));
}

// XY - q.X - p.Y + (p.q) I0 from the reference moments (I0, u1, u2, v1, v2, u1v1, u1v2, u2v1, u2v2;
// complex): X = EP.u, Y = EQ.v, XY = u EP.EQ v.
__device__ __forceinline__ void ss_efio_entry(const double* mom, const double (&EP)[2][3], const double (&EQ)[2][3],
                                              const double (&p)[3], const double (&q)[3], double& ar, double& ai) {
  const double pq = ss_dot(p, q);
  ar = pq * mom[0];
  ai = pq * mom[1];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double qe = ss_dot(q, EP[s]), pf = ss_dot(p, EQ[s]);
    ar -= fma(qe, mom[2 + 2 * s], pf * mom[6 + 2 * s]);
    ai -= fma(qe, mom[3 + 2 * s], pf * mom[7 + 2 * s]);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const double ef = ss_dot(EP[s], EQ[t]);
      ar = fma(ef, mom[10 + 4 * s + 2 * t], ar);
      ai = fma(ef, mom[11 + 4 * s + 2 * t], ai);
    }
  }
}

// acc[i] summed over the warp's lanes, left in every lane.  Halving: each step a lane keeps one
// half of its values and adds its partner's, so NV sums cost about NV + 5 additions instead of
// the 5 NV of a butterfly; the sums are then broadcast from the lanes that hold them.
template <int NV>
__device__ __forceinline__ void ss_warp_sum(double (&acc)[NV], int lane) {
  double v[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = i < NV ? acc[i < NV ? i : 0] : 0.0;
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      if (i >= NV) continue;  // zero in every lane
      const double keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, h);
    }
  }
  // lane l now holds the sum of value l
#pragma unroll
  for (int i = 0; i < NV; ++i) acc[i] = __shfl_sync(0xffffffffu, v[0], i);
}

}  // namespace fosb
