// Adjoint (reverse-mode) shape gradient of the discrete EFIE quantities with respect to
// the mesh vertex coordinates X (V x 3), used for gradients of monostatic RCS.
//
// For fixed coefficient vectors the kernels accumulate the real gradient of
//   J_Z = sum_i lambda_i^T Z(X) u_i                                  (pair kernels)
//   J_P = sum_i sum_t sum_j w_{e_j,i} alpha_i (s_j l_j / 2) sum_q w_q pi_i.(x_q - P_j) exp(ik d_i.x_q)
//                                                                    (triangle kernel)
// J_P covers both the plane-wave right-hand side (w = lambda, alpha = -1, pi = p_i,
// d = d_i: the term lambda^T b) and the far-field matrix (w = u, alpha = -ik,
// pi = (I - xh xh^T) c_i, d = -xh_i: the term c^T A u).
//
// With RWG functions the area factors cancel: a triangle-pair block is
//   Blk_jk = s_j s'_k l_j l'_k sum_pq w_pq G(r) [-(ik/4)(x_p - P_j).(y_q - Q_k) - 1/(ik)]
// (w_pq = product of the 6-point weights, or 4 x the Sauter-Schwab reference weights), so
// J_Z per pair is sum_pq w_pq G(r) H(x, y) with the bilinear
//   H = -(ik/4)(S x.y - x.U - V.y + c) + (i/k) S,   S = sum W_jk, U = sum W_jk Q_k,
//   V = sum W_jk P_j, c = sum W_jk P_j.Q_k,  W_jk = s_j s'_k l_j l'_k sum_i lambda_{j,i} u_{k,i}.
// Its derivatives with respect to the quadrature points (G' = G (ik - 1/r)), the opposite
// vertices and the edge lengths are accumulated (real parts) and chained to the vertices.
#include <cuda_runtime.h>

#include "fosb_internal.h"
#include "fp64_phase.cuh"
#include "pair_tiles.cuh"
#include "sauter_schwab.cuh"

namespace fosb {

// this translation unit's copy of the quadrature rules (uploaded with the assembly's)
__constant__ double c_bary[6][3];
__constant__ double c_w[6];
__constant__ double c_glx[16];
__constant__ double c_glw[16];
__constant__ double c_wbary[6][3];         // w_q bary_qb
__constant__ double c_phase[kPhaseTab][2];  // make_phase_table
__constant__ double c_adj_series[kSsTerms][14];  // make_ss_series, then make_ss_series_mfio

void upload_rules_adjoint(const Rules& r) {
  double wb[6][3], ph[kPhaseTab][2];
  for (int q = 0; q < 6; ++q)
    for (int b = 0; b < 3; ++b) wb[q][b] = r.w[q] * r.bary[q][b];
  cudaMemcpyToSymbol(c_wbary, wb, sizeof(wb));
  make_phase_table(ph);
  cudaMemcpyToSymbol(c_phase, ph, sizeof(ph));
  double se[kSsTerms][6], sh[kSsTerms][8], sc[kSsTerms][14];
  make_ss_series(r, se);
  make_ss_series_mfio<4>(r, sh);
  for (int j = 0; j < kSsTerms; ++j)
    for (int i = 0; i < 14; ++i) sc[j][i] = i < 6 ? se[j][i] : sh[j][i - 6];
  cudaMemcpyToSymbol(c_adj_series, sc, sizeof(sc));
  cudaMemcpyToSymbol(c_bary, r.bary, sizeof(r.bary));
  cudaMemcpyToSymbol(c_w, r.w, sizeof(r.w));
  cudaMemcpyToSymbol(c_glx, r.glx, sizeof(r.glx));
  cudaMemcpyToSymbol(c_glw, r.glw, sizeof(r.glw));
}

namespace {

constexpr double kInv4Pi = 0.07957747154594767;

struct Cx {
  double r, i;
};
__device__ __forceinline__ Cx operator+(Cx a, Cx b) { return {a.r + b.r, a.i + b.i}; }
__device__ __forceinline__ Cx operator-(Cx a, Cx b) { return {a.r - b.r, a.i - b.i}; }
__device__ __forceinline__ Cx operator*(Cx a, Cx b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
__device__ __forceinline__ Cx operator*(Cx a, double s) { return {a.r * s, a.i * s}; }

__device__ __forceinline__ void tri_edge_data(const DevMesh& m, int64_t t, int v[3], int e[3], double sl[3],
                                              double l[3], double V[3][3]) {
  for (int a = 0; a < 3; ++a) {
    v[a] = m.tris[3 * t + a];
    e[a] = m.tri_edge[3 * t + a];
    for (int d = 0; d < 3; ++d) V[a][d] = m.verts[3 * v[a] + d];
  }
  for (int j = 0; j < 3; ++j) {
    const double* A = V[(j + 1) % 3];
    const double* B = V[(j + 2) % 3];
    double dx = B[0] - A[0], dy = B[1] - A[1], dz = B[2] - A[2];
    l[j] = sqrt(dx * dx + dy * dy + dz * dz);
    sl[j] = (m.tri_coef[3 * t + j] > 0 ? 1.0 : -1.0) * l[j];
  }
}

// gradient of l_j (edge opposite local vertex j) into the vertex gradient array g (3 x 3)
__device__ __forceinline__ void chain_lengths(const double V[3][3], const double l[3], const double gl[3],
                                              double g[3][3]) {
  for (int j = 0; j < 3; ++j) {
    int a = (j + 1) % 3, b = (j + 2) % 3;
    for (int d = 0; d < 3; ++d) {
      double e = (V[b][d] - V[a][d]) / l[j];
      g[b][d] += gl[j] * e;
      g[a][d] -= gl[j] * e;
    }
  }
}

__device__ __forceinline__ void add_grad(double* grad, int v, const double g[3], double sgn) {
  for (int d = 0; d < 3; ++d) atomicAdd(grad + 3 * v + d, sgn * g[d]);
}

// ------------------------------------------------------------------ regular pairs
// Unordered pairs t1 < t2 with the symmetrised W_jk (lambda u + u lambda).  H is bilinear in the
// barycentric coordinates, H = sum_ab lambda_a beta_b H_ab with H_ab = H(P_a, Q_b), and everything
// linear in G follows from the moments mu_ab = sum_pq w lambda_pa beta_qb G: only the real vector
// F d = w Re(G'/r H) d is summed per point.  Bound by the FP64 pipe: about 53 instructions per
// point pair and 1200 per triangle pair (576 of them the W_jk of 8 columns), against 143 and
// 1000 per ordered pair with every term summed per point.  T = 5120, 8 columns: 92.7 ms, 310.7 ms before.

// imaginary part of a b
__device__ __forceinline__ double cx_mul_im(Cx a, Cx b) { return fma(a.r, b.i, a.i * b.r); }
__device__ __forceinline__ Cx cx_axpy(double s, Cx a, Cx b) { return {fma(s, a.r, b.r), fma(s, a.i, b.i)}; }

// One side's G-linear and explicit gradient terms, accumulated into g (vertex gradients of this
// side).  X: this side's vertices relative to vertex 0, r_j / wq_j: sum_k W_jk and sum_k W_jk Q_k
// over the other side, mo_a = sum_b mu_ab, moq_a = sum_b mu_ab Q_b, U = sum W Q_k, MX / MO: sum of
// mu X_a / mu Q_b, MXO the sum of mu X_a.Q_b.
//   points:   dJ/dx = mik4 G (S y - U)          -> (k/4) Im(S moq_a - U mo_a)
//   vertices: dJ/dX_j = (ik/4)(r_j MO - wq_j I0) -> -(k/4) Im(...)
//   lengths:  l_j dJ/dl_j = sum_k W_jk K_jk, K_jk = -(ik/4)(MXO - Q_k.MX - X_j.MO + X_j.Q_k I0) + (i/k) I0.
__device__ __forceinline__ void adjoint_side(double k4, double kinv, Cx S, Cx I0, Cx MXO, const Cx (&MX)[3],
                                             const Cx (&MO)[3], const Cx (&U)[3], const Cx (&r)[3],
                                             const Cx (&wq)[3][3], const Cx (&mo)[3], const Cx (&moq)[3][3],
                                             const double (&X)[3][3], double (&g)[3][3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      double im = cx_mul_im(S, moq[a][d]) - cx_mul_im(U[d], mo[a]);
      im -= cx_mul_im(r[a], MO[d]) - cx_mul_im(wq[a][d], I0);
      g[a][d] = fma(k4, im, g[a][d]);
    }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    Cx t = MXO, xq = {0.0, 0.0};
    double im = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (j > 0) {
        t = cx_axpy(-X[j][d], MO[d], t);
        xq = cx_axpy(X[j][d], wq[j][d], xq);
      }
      im -= cx_mul_im(wq[j][d], MX[d]);
    }
    im += cx_mul_im(r[j], t);
    if (j > 0) im += cx_mul_im(xq, I0);
    const double lk = fma(k4, im, -kinv * cx_mul_im(r[j], I0));  // l_j dJ/dl_j
    const int a = (j + 1) % 3, b = (j + 2) % 3;
    double e[3], l2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      e[d] = X[b][d] - X[a][d];
      l2 = fma(e[d], e[d], l2);
    }
    const double rl = ss_rsqrt(l2), f = lk * (rl * rl);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      g[b][d] = fma(f, e[d], g[b][d]);
      g[a][d] = fma(-f, e[d], g[a][d]);
    }
  }
}

__global__ void __launch_bounds__(128) adjoint_regular_kernel(DevMesh m, double k, const double* __restrict__ lam,
                                                              const double* __restrict__ U, int64_t ld, int64_t nrhs,
                                                              double* grad) {
  __shared__ double2 tab[kPhaseTab];
  int64_t rg, cb;
  if (!pair_tile(m.nt, 4, blockIdx.y, blockIdx.x, rg, cb)) return;
  tab[threadIdx.x] = make_double2(c_phase[threadIdx.x][0], c_phase[threadIdx.x][1]);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t t1 = rg * 4 + (threadIdx.x >> 5);
  int64_t t2 = cb * 32 + lane;
  if (t1 >= m.nt) return;  // the whole warp
  bool live = t2 < m.nt && t1 < t2;
  int v1[3], v2[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) v1[a] = m.tris[3 * t1 + a];
  if (live) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      v2[a] = m.tris[3 * t2 + a];
      live = live && v2[a] != v1[0] && v2[a] != v1[1] && v2[a] != v1[2];
    }
  }
  if (!__any_sync(0xffffffffu, live)) return;
  double g1[3][3] = {};
  if (live) {
    double P[3][3], Q[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        P[a][d] = m.verts[3 * v1[a] + d] - m.verts[3 * v1[0] + d];
        Q[a][d] = m.verts[3 * v2[a] + d] - m.verts[3 * v2[0] + d];
      }
    // W_jk = s_j l_j s'_k l'_k/(4 pi) sum_i (lambda_j u_k + u_j lambda_k)
    Cx W[3][3] = {};
    {
      int64_t o1[3], o2[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        o1[j] = m.tri_edge[3 * t1 + j] * ld;
        o2[j] = m.tri_edge[3 * t2 + j] * ld;
      }
      const Cx* L = reinterpret_cast<const Cx*>(lam);
      const Cx* Uc = reinterpret_cast<const Cx*>(U);
#pragma unroll 1
      for (int64_t i = 0; i < nrhs; ++i) {
        Cx a[3], b[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          a[j] = L[o1[j] + i];
          b[j] = Uc[o1[j] + i];
        }
#pragma unroll
        for (int kk = 0; kk < 3; ++kk) {
          const Cx c = Uc[o2[kk] + i], d = L[o2[kk] + i];
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            Cx& w = W[j][kk];
            w.r = fma(a[j].r, c.r, fma(-a[j].i, c.i, fma(b[j].r, d.r, fma(-b[j].i, d.i, w.r))));
            w.i = fma(a[j].r, c.i, fma(a[j].i, c.r, fma(b[j].r, d.i, fma(b[j].i, d.r, w.i))));
          }
        }
      }
      const double A1 = 2.0 * m.tri_area[t1] * kInv4Pi, A2 = 2.0 * m.tri_area[t2];
#pragma unroll
      for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int kk = 0; kk < 3; ++kk) W[j][kk] = W[j][kk] * ((A1 * m.tri_coef[3 * t1 + j]) * (A2 * m.tri_coef[3 * t2 + kk]));
    }
    // sums over one side and the vertex values H_ab
    Cx rj[3], ck[3], S = {0.0, 0.0}, c = {0.0, 0.0}, Us[3] = {}, Vs[3] = {};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      rj[j] = W[j][0] + W[j][1] + W[j][2];
      ck[j] = W[0][j] + W[1][j] + W[2][j];
      S = S + rj[j];
    }
#pragma unroll
    for (int j = 1; j < 3; ++j)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        Us[d] = cx_axpy(Q[j][d], ck[j], Us[d]);
        Vs[d] = cx_axpy(P[j][d], rj[j], Vs[d]);
      }
    double pq[3][3] = {};
#pragma unroll
    for (int a = 1; a < 3; ++a)
#pragma unroll
      for (int b = 1; b < 3; ++b) {
        pq[a][b] = ss_dot(P[a], Q[b]);
        c = cx_axpy(pq[a][b], W[a][b], c);
      }
    const double k4 = 0.25 * k, kinv = 1.0 / k;
    Cx H[3][3];
    {
      Cx pu[3] = {}, vq[3] = {};
#pragma unroll
      for (int a = 1; a < 3; ++a)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          pu[a] = cx_axpy(P[a][d], Us[d], pu[a]);
          vq[a] = cx_axpy(Q[a][d], Vs[d], vq[a]);
        }
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const Cx B = cx_axpy(pq[a][b], S, c - pu[a] - vq[b]);
          H[a][b] = {fma(k4, B.i, -kinv * S.i), fma(-k4, B.r, kinv * S.r)};  // -(ik/4) B + (i/k) S
        }
    }
    // the point loop: mu and the real F d sums
    const double* xq = m.tri_qp + 18 * t1;
    const double* yq = m.tri_qp + 18 * t2;
    double gy[6][3] = {};
    Cx mu[3][3] = {};
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      const double x0 = xq[3 * p], x1 = xq[3 * p + 1], x2 = xq[3 * p + 2];
      Cx T[3] = {}, A[3] = {};
      double gx[3] = {};
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) T[b] = cx_axpy(c_wbary[p][a], H[a][b], T[b]);
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const double d[3] = {x0 - yq[3 * q], x1 - yq[3 * q + 1], x2 - yq[3 * q + 2]};
        const double r2 = fma(d[0], d[0], fma(d[1], d[1], d[2] * d[2]));
        const double rinv = ss_rsqrt(r2), kr = k * (r2 * rinv);
        double cs, sn;
        expi_table(kr, tab, cs, sn);
        const Cx G = {cs * rinv, sn * rinv};
        Cx h = {0.0, 0.0};  // w_p w_q H
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          A[b] = cx_axpy(c_wbary[q][b], G, A[b]);
          h = cx_axpy(c_wbary[q][b], T[b], h);
        }
        // F = Re(G (ikr - 1) H)/r^2
        const double hr = fma(kr, h.i, h.r), hi = fma(-kr, h.r, h.i);  // -(ikr - 1) H
        const double F = (rinv * rinv) * fma(G.i, hi, -G.r * hr);
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          gx[e] = fma(F, d[e], gx[e]);
          gy[q][e] = fma(-F, d[e], gy[q][e]);
        }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int b = 0; b < 3; ++b) mu[a][b] = cx_axpy(c_wbary[p][a], A[b], mu[a][b]);
#pragma unroll
        for (int e = 0; e < 3; ++e) g1[a][e] = fma(c_bary[p][a], gx[e], g1[a][e]);
      }
    }
    double g2[3][3] = {};
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int e = 0; e < 3; ++e) g2[b][e] = fma(c_bary[q][b], gy[q][e], g2[b][e]);
    // moments of G
    Cx m1[3], m2[3], I0 = {0.0, 0.0}, MP[3] = {}, MQ[3] = {}, MPQ = {0.0, 0.0}, mq[3][3] = {}, mp[3][3] = {};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      m1[a] = mu[a][0] + mu[a][1] + mu[a][2];
      m2[a] = mu[0][a] + mu[1][a] + mu[2][a];
      I0 = I0 + m1[a];
#pragma unroll
      for (int b = 1; b < 3; ++b)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          mq[a][d] = cx_axpy(Q[b][d], mu[a][b], mq[a][d]);
          mp[a][d] = cx_axpy(P[b][d], mu[b][a], mp[a][d]);
        }
    }
#pragma unroll
    for (int a = 1; a < 3; ++a)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        MP[d] = cx_axpy(P[a][d], m1[a], MP[d]);
        MQ[d] = cx_axpy(Q[a][d], m2[a], MQ[d]);
        MPQ = cx_axpy(P[a][d], mq[a][d], MPQ);
      }
    Cx wq[3][3] = {}, wp[3][3] = {};
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int b = 1; b < 3; ++b)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          wq[j][d] = cx_axpy(Q[b][d], W[j][b], wq[j][d]);
          wp[j][d] = cx_axpy(P[b][d], W[b][j], wp[j][d]);
        }
    adjoint_side(k4, kinv, S, I0, MPQ, MP, MQ, Us, rj, wq, m1, mq, P, g1);
    adjoint_side(k4, kinv, S, I0, MPQ, MQ, MP, Vs, ck, wp, m2, mp, Q, g2);
#pragma unroll
    for (int a = 0; a < 3; ++a) add_grad(grad, v2[a], g2[a], -1.0);  // J_Z enters the objective with a minus sign
  }
  // t1 is the warp's: one addition per vertex coordinate
  double s[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) s[i] = g1[i / 3][i % 3];
  ss_warp_sum<9>(s, lane);
  if (lane == 0)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double g[3] = {s[3 * a], s[3 * a + 1], s[3 * a + 2]};
      add_grad(grad, v1[a], g, -1.0);
    }
}

// ------------------------------------------------------------------ touching pairs
// One touching pair (t1 <= t2) per warp, Sauter-Schwab in the form (x, y) = xi (xh, yh) with the
// xi sums as power series in phi = k |xh - yh| (see efie_singular_kernel).  With the moments of G
// in the reference coordinates and H along xi a quadratic h0 + xi h1 + xi^2 h2, the sums of F d
// and of xi F d (chained to the vertices through u and v) are
//   F_0 = Re(Q_1 h0 + Q_2 h1 + Q_3 h2)/rh^3, F_1 = Re(Q_2 h0 + Q_3 h1 + Q_4 h2)/rh^3,
//   Q_m = sum_a w_a xi_a^m (i phi xi_a - 1) exp(i phi xi_a).
// Bound by the FP64 pipe: about 185 instructions per 5 points against 145 per point.  T = 5120,
// n_ss = 5, 8 columns: 7.8 ms, 39.3 ms before.
template <int KIND>
__device__ __forceinline__ void adjoint_ss_moments(const double* __restrict__ table, double k, int nss, int J,
                                                   const double (&EP)[2][3], const double (&EQ)[2][3], Cx h0,
                                                   const Cx (&hu)[4], const Cx (&huv)[4], int lane, double (&e)[18],
                                                   double (&f)[15]) {
  const int n3 = nss * nss * nss, stride = kSsRegions * n3, count = ss_regions<KIND>() * n3;
  const double* tab = table + ss_first_region<KIND>() * n3;
  for (int idx = lane; idx < count; idx += 32) {
    auto T = [&](int q) { return __ldg(tab + q * stride + idx); };
    const double uv[4] = {T(0), T(1), T(2), T(3)};
    double d[3], rinv, phi;
    ss_distance<KIND>(tab + idx, stride, uv, EP, EQ, k, d, rinv, phi);
    // Re S_0..2, Im S_0..2, Re Q_1..4, Im Q_1..4
    double s[14];
    if (J > 0) {
      const double p2 = phi * phi;
#pragma unroll
      for (int i = 0; i < 14; ++i) s[i] = c_adj_series[J - 1][i];
      for (int j = J - 2; j >= 0; --j)
#pragma unroll
        for (int i = 0; i < 14; ++i) s[i] = fma(s[i], p2, c_adj_series[j][i]);
#pragma unroll
      for (int i = 3; i < 6; ++i) s[i] *= phi;
#pragma unroll
      for (int i = 10; i < 14; ++i) s[i] *= phi;
    } else {
#pragma unroll
      for (int i = 0; i < 14; ++i) s[i] = 0.0;
      for (int a = 0; a < nss; ++a) {
        const double xi = c_glx[a], px = phi * xi;
        double sn, cs, w = c_glw[a];
        sincos(px, &sn, &cs);
        const double hr = -cs - px * sn, hi = px * cs - sn;
#pragma unroll
        for (int m = 1; m <= 4; ++m) {
          w *= xi;
          s[5 + m] += w * hr;
          s[9 + m] += w * hi;
          if (m >= 2) {
            s[m - 2] += w * cs;
            s[m + 1] += w * sn;
          }
        }
      }
    }
    const double g = T(4) * rinv, g3 = g * (rinv * rinv);
    Cx h1 = {0.0, 0.0}, h2 = {0.0, 0.0};
    e[0] = fma(g, s[0], e[0]);
    e[1] = fma(g, s[3], e[1]);
    const double ar = g * s[1], ai = g * s[4], br = g * s[2], bi = g * s[5];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double p = T(5 + q);
      e[2 + 2 * q] = fma(uv[q], ar, e[2 + 2 * q]);
      e[3 + 2 * q] = fma(uv[q], ai, e[3 + 2 * q]);
      e[10 + 2 * q] = fma(p, br, e[10 + 2 * q]);
      e[11 + 2 * q] = fma(p, bi, e[11 + 2 * q]);
      h1 = cx_axpy(uv[q], hu[q], h1);
      h2 = cx_axpy(p, huv[q], h2);
    }
    double F[2];
#pragma unroll
    for (int m = 0; m < 2; ++m)
      F[m] = g3 * (fma(s[6 + m], h0.r, -s[10 + m] * h0.i) + fma(s[7 + m], h1.r, -s[11 + m] * h1.i) +
                   fma(s[8 + m], h2.r, -s[12 + m] * h2.i));
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] = fma(F[0], d[c], f[c]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double fq = F[1] * uv[q];
#pragma unroll
      for (int c = 0; c < 3; ++c) f[3 + 3 * q + c] = fma(fq, d[c], f[3 + 3 * q + c]);
    }
  }
}

__global__ void __launch_bounds__(128) adjoint_singular_kernel(DevMesh m, double k, int nss,
                                                               const double* __restrict__ table,
                                                               const double* __restrict__ lam,
                                                               const double* __restrict__ U, int64_t ld, int64_t nrhs,
                                                               double* grad) {
  const int64_t pair = int64_t(blockIdx.x) * 4 + (threadIdx.x >> 5);
  if (pair >= m.ntouch) return;
  const int lane = threadIdx.x & 31;
  const TouchPair tp = m.touch[pair];
  const int64_t t1 = tp.t1, t2 = tp.t2;
  double EP[2][3], EQ[2][3], X1[3][3], X2[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double o = m.verts[3 * tp.p[0] + c];  // the shared vertex P0 = Q0
    EP[0][c] = m.verts[3 * tp.p[1] + c] - o;
    EP[1][c] = m.verts[3 * tp.p[2] + c] - m.verts[3 * tp.p[1] + c];
    EQ[0][c] = m.verts[3 * tp.q[1] + c] - o;
    EQ[1][c] = m.verts[3 * tp.q[2] + c] - m.verts[3 * tp.q[1] + c];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      X1[a][c] = m.verts[3 * m.tris[3 * t1 + a] + c] - o;
      X2[a][c] = m.verts[3 * m.tris[3 * t2 + a] + c] - o;
    }
  }
  // W_jk = s_j l_j s'_k l'_k 4/(4 pi) sum_i (lambda_j u_k [+ u_j lambda_k unless t1 = t2]), one entry
  // per lane 0-8; the 4 is the reference weights' Jacobian 2A 2A'/(A A')
  Cx W[3][3];
  {
    const int j = lane < 9 ? lane / 3 : 0, kk = lane < 9 ? lane % 3 : 0;
    const int64_t o1 = m.tri_edge[3 * t1 + j] * ld, o2 = m.tri_edge[3 * t2 + kk] * ld;
    const Cx* L = reinterpret_cast<const Cx*>(lam);
    const Cx* Uc = reinterpret_cast<const Cx*>(U);
    Cx w = {0.0, 0.0};
    const double mir = t1 != t2 ? 1.0 : 0.0;
    for (int64_t i = 0; i < nrhs; ++i) {
      const Cx a = L[o1 + i], b = Uc[o2 + i], c = Uc[o1 + i] * mir, d = L[o2 + i];
      w = w + a * b + c * d;
    }
    const double sc = (2.0 * m.tri_area[t1] * m.tri_coef[3 * t1 + j]) * (2.0 * m.tri_area[t2] * m.tri_coef[3 * t2 + kk]);
    w = w * (4.0 * kInv4Pi * sc);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        W[a][b] = {__shfl_sync(0xffffffffu, w.r, 3 * a + b), __shfl_sync(0xffffffffu, w.i, 3 * a + b)};
  }
  const double k4 = 0.25 * k, kinv = 1.0 / k;
  Cx S = {0.0, 0.0}, c0 = {0.0, 0.0}, Us[3] = {}, Vs[3] = {};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const Cx r = W[j][0] + W[j][1] + W[j][2], c = W[0][j] + W[1][j] + W[2][j];
    S = S + r;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      Us[d] = cx_axpy(X2[j][d], c, Us[d]);
      Vs[d] = cx_axpy(X1[j][d], r, Vs[d]);
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) c0 = cx_axpy(ss_dot(X1[j], X2[b]), W[j][b], c0);
  }
  // H(xi xh, xi yh) = h0 + xi h1 + xi^2 h2 with h1 linear in (u, v) and h2 in the products u v
  const Cx h0 = {fma(k4, c0.i, -kinv * S.i), fma(-k4, c0.r, kinv * S.r)};
  Cx hu[4], huv[4];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    Cx eu = {0.0, 0.0}, fv = {0.0, 0.0};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      eu = cx_axpy(EP[s][d], Us[d], eu);
      fv = cx_axpy(EQ[s][d], Vs[d], fv);
    }
    hu[s] = {-k4 * eu.i, k4 * eu.r};  // (ik/4) E_s.U
    hu[2 + s] = {-k4 * fv.i, k4 * fv.r};
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const double ef = k4 * ss_dot(EP[s], EQ[t]);
      huv[2 * s + t] = {ef * S.i, -ef * S.r};  // -(ik/4) S E_s.F_t
    }
  }
  const int J = ss_terms(ss_phase_bound(k, EP, EQ));
  const int terms = J > 0 ? min(J + 1, kSsTerms) : 0;  // the Q series carry a factor 2j - 1
  double e[18], f[15];
#pragma unroll
  for (int i = 0; i < 18; ++i) e[i] = 0.0;
#pragma unroll
  for (int i = 0; i < 15; ++i) f[i] = 0.0;
  if (tp.kind == 3) adjoint_ss_moments<3>(table, k, nss, terms, EP, EQ, h0, hu, huv, lane, e, f);
  else if (tp.kind == 2) adjoint_ss_moments<2>(table, k, nss, terms, EP, EQ, h0, hu, huv, lane, e, f);
  else adjoint_ss_moments<1>(table, k, nss, terms, EP, EQ, h0, hu, huv, lane, e, f);
  ss_warp_sum<18>(e, lane);
  ss_warp_sum<15>(f, lane);
  if (lane >= 2) return;
  // Lane 0 takes t1's side, lane 1 t2's, the same formulas with the sides exchanged: X, E this
  // side's vertices and edge vectors, O, Eo the other's, Wk this side's index first.
  const bool sw = lane == 1;
  auto pick = [&](double a, double b) { return sw ? b : a; };
  double X[3][3], O[3][3], E[2][3], Eo[2][3];
  Cx Wk[3][3], Ux[3], Mi[3], Mo[3], Mp[3][3];  // moments: this side's basis (1, u1, u2), the other's, products
  double g[3][3];                            // point gradients along the basis (F part)
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      X[a][d] = pick(X1[a][d], X2[a][d]);
      O[a][d] = pick(X2[a][d], X1[a][d]);
      if (a < 2) {
        E[a][d] = pick(EP[a][d], EQ[a][d]);
        Eo[a][d] = pick(EQ[a][d], EP[a][d]);
      }
      Wk[a][d] = {pick(W[a][d].r, W[d][a].r), pick(W[a][d].i, W[d][a].i)};
      g[a][d] = a == 0 ? pick(f[d], -f[d]) : pick(f[3 * a + d], -f[6 + 3 * a + d]);
    }
#pragma unroll
  for (int d = 0; d < 3; ++d) Ux[d] = {pick(Us[d].r, Vs[d].r), pick(Us[d].i, Vs[d].i)};
  const Cx I0 = {e[0], e[1]};
  Mi[0] = Mo[0] = Mp[0][0] = I0;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    Mi[1 + s] = {pick(e[2 + 2 * s], e[6 + 2 * s]), pick(e[3 + 2 * s], e[7 + 2 * s])};
    Mo[1 + s] = {pick(e[6 + 2 * s], e[2 + 2 * s]), pick(e[7 + 2 * s], e[3 + 2 * s])};
    Mp[1 + s][0] = Mi[1 + s];
    Mp[0][1 + s] = Mo[1 + s];
#pragma unroll
    for (int t = 0; t < 2; ++t)
      Mp[1 + s][1 + t] = {pick(e[10 + 4 * s + 2 * t], e[10 + 4 * t + 2 * s]),
                          pick(e[11 + 4 * s + 2 * t], e[11 + 4 * t + 2 * s])};
  }
  // point gradients linear in G: (k/4) Im(S sum phi_i G y - U sum phi_i G), phi = (1, u1, u2)
  Cx My[3] = {}, Mx[3] = {}, Mxy = {0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      Cx y = {0.0, 0.0};
#pragma unroll
      for (int t = 0; t < 2; ++t) y = cx_axpy(Eo[t][d], Mp[i][1 + t], y);
      g[i][d] = fma(k4, cx_mul_im(S, y) - cx_mul_im(Ux[d], Mp[i][0]), g[i][d]);
      if (i == 0) My[d] = y;
      else {
        Mx[d] = cx_axpy(E[i - 1][d], Mi[i], Mx[d]);
        Mxy = cx_axpy(E[i - 1][d], y, Mxy);
      }
    }
  // J_Z enters the objective with a minus sign; x = P0 (1 - u1) + P1 (u1 - u2) + P2 u2
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double ga[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) ga[d] = a < 2 ? g[a][d] - g[a + 1][d] : g[a][d];
    add_grad(grad, sw ? tp.q[a] : tp.p[a], ga, -1.0);
  }
  // opposite vertices and edge lengths (adjoint_side's formulas)
  double gv[3][3] = {};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const Cx r = Wk[j][0] + Wk[j][1] + Wk[j][2];
    Cx t = Mxy, xq = {0.0, 0.0};
    double im = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      Cx wq = {0.0, 0.0};
#pragma unroll
      for (int b = 0; b < 3; ++b) wq = cx_axpy(O[b][d], Wk[j][b], wq);
      gv[j][d] = fma(-k4, cx_mul_im(r, My[d]) - cx_mul_im(wq, I0), gv[j][d]);
      t = cx_axpy(-X[j][d], My[d], t);
      xq = cx_axpy(X[j][d], wq, xq);
      im -= cx_mul_im(wq, Mx[d]);
    }
    im += cx_mul_im(r, t) + cx_mul_im(xq, I0);
    const double lk = fma(k4, im, -kinv * cx_mul_im(r, I0));
    const int a = (j + 1) % 3, b = (j + 2) % 3;
    double ev[3], l2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      ev[d] = X[b][d] - X[a][d];
      l2 = fma(ev[d], ev[d], l2);
    }
    const double rl = ss_rsqrt(l2), fl = lk * (rl * rl);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      gv[b][d] = fma(fl, ev[d], gv[b][d]);
      gv[a][d] = fma(-fl, ev[d], gv[a][d]);
    }
  }
  const int64_t tt = sw ? t2 : t1;
#pragma unroll
  for (int a = 0; a < 3; ++a) add_grad(grad, m.tris[3 * tt + a], gv[a], -1.0);
}

// ------------------------------------------------------------------ plane-wave moments
// J_P term for one (triangle, column i): coefficient vector pi (complex 3), direction dd,
// alpha (complex), edge weights w (N x m, column i).  Thread per (triangle, column).
__global__ void adjoint_planewave_kernel(DevMesh m, double k, int64_t ncols, const double* pw /* ncols x 11 */,
                                         const double* wgt, int64_t ldw, double* grad) {
  int64_t gid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (gid >= m.nt * ncols) return;
  const int64_t t = gid / ncols, i = gid % ncols;
  const double* c = pw + 11 * i;  // d(3), Re pi(3), Im pi(3), alpha (re, im)
  const Cx pi3[3] = {{c[3], c[6]}, {c[4], c[7]}, {c[5], c[8]}};
  const Cx alpha = {c[9], c[10]};
  int v[3], e[3];
  double sl[3], l[3], V[3][3];
  tri_edge_data(m, t, v, e, sl, l, V);
  Cx kap[3];
  for (int j = 0; j < 3; ++j) {
    Cx w = {wgt[2 * (e[j] * ldw + i)], wgt[2 * (e[j] * ldw + i) + 1]};
    kap[j] = w * alpha * (0.5 * sl[j]);
  }
  double g[3][3] = {}, gl[3] = {0, 0, 0};
  for (int q = 0; q < 6; ++q) {
    double x[3];
    for (int d = 0; d < 3; ++d) x[d] = m.tri_qp[18 * t + 3 * q + d];
    double sn, cs;
    sincos(k * (c[0] * x[0] + c[1] * x[1] + c[2] * x[2]), &sn, &cs);
    Cx E = {cs * c_w[q], sn * c_w[q]};
    for (int j = 0; j < 3; ++j) {
      Cx pxp = {0, 0};
      for (int d = 0; d < 3; ++d) pxp = pxp + pi3[d] * (x[d] - V[j][d]);
      Cx kE = kap[j] * E;
      Cx term = kE * pxp;
      gl[j] += term.r / l[j];
      Cx ikd_pxp = Cx{0.0, k} * pxp;
      for (int d = 0; d < 3; ++d) {
        double gxd = (kE * (pi3[d] + ikd_pxp * c[d])).r;
        for (int a = 0; a < 3; ++a) g[a][d] += c_bary[q][a] * gxd;
        g[j][d] -= (kE * pi3[d]).r;  // explicit opposite vertex P_j
      }
    }
  }
  chain_lengths(V, l, gl, g);
  for (int a = 0; a < 3; ++a) add_grad(grad, v[a], g[a], 1.0);
}

inline unsigned cdiv(int64_t a, int64_t b) { return unsigned((a + b - 1) / b); }

}  // namespace

cudaError_t launch_adjoint_pairs(const DevMesh& m, double k, int nss, const double* lam, const double* U, int64_t ld,
                                 int64_t nrhs, double* grad, cudaStream_t s) {
  if (cdiv(m.nt, 4) > 65535u) return cudaErrorInvalidValue;
  const dim3 grid(unsigned(pair_tiles_width(m.nt)), unsigned(pair_tiles_rows(m.nt, 4)));
  adjoint_regular_kernel<<<grid, 128, 0, s>>>(m, k, lam, U, ld, nrhs, grad);
  note_launches(1);
  if (m.ntouch > 0) {
    const double* table = ss_table_device();
    if (!table) return cudaErrorInvalidSymbol;
    adjoint_singular_kernel<<<cdiv(m.ntouch, 4), 128, 0, s>>>(m, k, nss, table, lam, U, ld, nrhs, grad);
    note_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t launch_adjoint_planewave(const DevMesh& m, double k, int64_t ncols, const double* d_pw, const double* wgt,
                                     int64_t ldw, double* grad, cudaStream_t s) {
  if (ncols == 0) return cudaSuccess;
  adjoint_planewave_kernel<<<cdiv(m.nt * ncols, 128), 128, 0, s>>>(m, k, ncols, d_pw, wgt, ldw, grad);
  return launched();
}

}  // namespace fosb
