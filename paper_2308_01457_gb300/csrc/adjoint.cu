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

void upload_rules_adjoint(const Rules& r) {
  double wb[6][3], ph[kPhaseTab][2];
  for (int q = 0; q < 6; ++q)
    for (int b = 0; b < 3; ++b) wb[q][b] = r.w[q] * r.bary[q][b];
  cudaMemcpyToSymbol(c_wbary, wb, sizeof(wb));
  make_phase_table(ph);
  cudaMemcpyToSymbol(c_phase, ph, sizeof(ph));
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

// Per-pair state: the coefficient matrix W (already scaled by s s' l l'), origins and the
// local (origin-relative) opposite vertices of both triangles.
struct PairCoef {
  Cx W[3][3];
  Cx S, U[3], V[3], c;
};

__device__ void make_coef(const double P[3][3], const double Q[3][3], PairCoef& pc) {
  pc.S = {0, 0};
  pc.c = {0, 0};
  for (int d = 0; d < 3; ++d) pc.U[d] = pc.V[d] = Cx{0, 0};
  for (int j = 0; j < 3; ++j)
    for (int k = 0; k < 3; ++k) {
      Cx w = pc.W[j][k];
      pc.S = pc.S + w;
      double pq = P[j][0] * Q[k][0] + P[j][1] * Q[k][1] + P[j][2] * Q[k][2];
      pc.c = pc.c + w * pq;
      for (int d = 0; d < 3; ++d) {
        pc.U[d] = pc.U[d] + w * Q[k][d];
        pc.V[d] = pc.V[d] + w * P[j][d];
      }
    }
}

// Accumulators of one pair: real gradients at the points and complex moments.
struct PairAcc {
  double gx[6][3], gy[6][3];   // regular: per test / trial point
  Cx I0, Mx[3], My[3], Mxy;
};

// One point pair: x, y local coordinates (x - o1, y - o2), dvec = x - y (absolute),
// weight w (includes the 1/(4 pi) of G).  Returns the real gradient contributions with
// respect to x and y and adds the moments.
__device__ __forceinline__ void point_pair(double k, const PairCoef& pc, const double x[3], const double y[3],
                                           const double dvec[3], double w, double gx[3], double gy[3],
                                           PairAcc& A) {
  double r2 = dvec[0] * dvec[0] + dvec[1] * dvec[1] + dvec[2] * dvec[2];
  double rinv = rsqrt(r2);
  double r = r2 * rinv;
  double sn, cs;
  sincos(k * r, &sn, &cs);
  Cx G = {cs * rinv * w, sn * rinv * w};
  Cx Gp_over_r = G * Cx{-rinv * rinv, k * rinv};  // G'(r)/r = G (ik - 1/r)/r
  double xy = x[0] * y[0] + x[1] * y[1] + x[2] * y[2];
  Cx xU = pc.U[0] * x[0] + pc.U[1] * x[1] + pc.U[2] * x[2];
  Cx Vy = pc.V[0] * y[0] + pc.V[1] * y[1] + pc.V[2] * y[2];
  Cx B = pc.S * xy - xU - Vy + pc.c;
  const Cx mik4 = {0.0, -0.25 * k};
  Cx H = mik4 * B + Cx{0.0, 1.0 / k} * pc.S;
  Cx GH = Gp_over_r * H;
  Cx Gm = G * mik4;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Cx dHx = pc.S * y[d] - pc.U[d];  // (S y - U)
    Cx dHy = pc.S * x[d] - pc.V[d];  // (S x - V)
    gx[d] += GH.r * dvec[d] + (Gm * dHx).r;
    gy[d] += -GH.r * dvec[d] + (Gm * dHy).r;
  }
  A.I0 = A.I0 + G;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    A.Mx[d] = A.Mx[d] + G * x[d];
    A.My[d] = A.My[d] + G * y[d];
  }
  A.Mxy = A.Mxy + G * xy;
}

// Explicit (non point) terms of one pair: opposite vertices and edge lengths.
//   dJ/dP_j = (ik/4) sum_k W_jk (My - Q_k I0),  dJ/dQ_k = (ik/4) sum_j W_jk (Mx - P_j I0),
//   dJ/dl_j = sum_k W_jk K_jk / l_j,  K_jk = -(ik/4)(Mxy - Q_k.Mx - P_j.My + P_j.Q_k I0) + (i/k) I0.
__device__ void explicit_terms(double k, const PairCoef& pc, const PairAcc& A, const double P[3][3],
                               const double Q[3][3], const double l1[3], const double l2[3], double gP[3][3],
                               double gQ[3][3], double gl1[3], double gl2[3]) {
  const Cx ik4 = {0.0, 0.25 * k};
  for (int j = 0; j < 3; ++j) {
    gl1[j] = gl2[j] = 0.0;
    for (int d = 0; d < 3; ++d) gP[j][d] = gQ[j][d] = 0.0;
  }
  for (int j = 0; j < 3; ++j)
    for (int kk = 0; kk < 3; ++kk) {
      Cx w = pc.W[j][kk];
      Cx wik = w * ik4;
      for (int d = 0; d < 3; ++d) {
        gP[j][d] += (wik * (A.My[d] - A.I0 * Q[kk][d])).r;
        gQ[kk][d] += (wik * (A.Mx[d] - A.I0 * P[j][d])).r;
      }
      Cx QMx = A.Mx[0] * Q[kk][0] + A.Mx[1] * Q[kk][1] + A.Mx[2] * Q[kk][2];
      Cx PMy = A.My[0] * P[j][0] + A.My[1] * P[j][1] + A.My[2] * P[j][2];
      double pq = P[j][0] * Q[kk][0] + P[j][1] * Q[kk][1] + P[j][2] * Q[kk][2];
      Cx K = Cx{0.0, -0.25 * k} * (A.Mxy - QMx - PMy + A.I0 * pq) + Cx{0.0, 1.0 / k} * A.I0;
      double v = (w * K).r;
      gl1[j] += v / l1[j];
      gl2[kk] += v / l2[kk];
    }
}

// W_jk = s_j s'_k l_j l'_k sum_i lambda[e1_j, i] u[e2_k, i] (+ the mirrored term for
// touching pairs whose transpose block is not evaluated separately).
__device__ void load_w(const double* lam, const double* U, int64_t ld, int64_t m, const int e1[3], const int e2[3],
                       const double sl1[3], const double sl2[3], bool mirror, PairCoef& pc) {
  for (int j = 0; j < 3; ++j)
    for (int kk = 0; kk < 3; ++kk) {
      Cx acc = {0, 0};
      for (int64_t i = 0; i < m; ++i) {
        Cx a = {lam[2 * (e1[j] * ld + i)], lam[2 * (e1[j] * ld + i) + 1]};
        Cx b = {U[2 * (e2[kk] * ld + i)], U[2 * (e2[kk] * ld + i) + 1]};
        acc = acc + a * b;
        if (mirror) {
          Cx a2 = {lam[2 * (e2[kk] * ld + i)], lam[2 * (e2[kk] * ld + i) + 1]};
          Cx b2 = {U[2 * (e1[j] * ld + i)], U[2 * (e1[j] * ld + i) + 1]};
          acc = acc + a2 * b2;
        }
      }
      pc.W[j][kk] = acc * (sl1[j] * sl2[kk]);
    }
}

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
// One CTA (128 threads) per touching pair (t1 <= t2), Sauter-Schwab points in the
// orientation of the assembly; gradients at the points are chained immediately to the
// permuted vertices through the barycentric weights of chi.
__device__ __forceinline__ void chi_bary(double u1, double u2, double a[3]) {
  a[0] = 1.0 - u1;
  a[1] = u1 - u2;
  a[2] = u2;
}

__global__ void __launch_bounds__(128) adjoint_singular_kernel(DevMesh m, double k, int nss, const double* lam,
                                                               const double* U, int64_t ld, int64_t nrhs,
                                                               double* grad) {
  const TouchPair tp = m.touch[blockIdx.x];
  const int t1 = tp.t1, t2 = tp.t2;
  int v1[3], v2[3], e1[3], e2[3];
  double sl1[3], sl2[3], l1[3], l2[3], V1[3][3], V2[3][3];
  tri_edge_data(m, t1, v1, e1, sl1, l1, V1);
  tri_edge_data(m, t2, v2, e2, sl2, l2, V2);
  double Pp[3][3], Qp[3][3];  // permuted vertices (Sauter-Schwab order), absolute
  for (int a = 0; a < 3; ++a)
    for (int d = 0; d < 3; ++d) {
      Pp[a][d] = m.verts[3 * tp.p[a] + d];
      Qp[a][d] = m.verts[3 * tp.q[a] + d];
    }
  // local coordinates relative to the shared vertex Pp[0] == Qp[0]
  double P[3][3], Q[3][3];
  for (int a = 0; a < 3; ++a)
    for (int d = 0; d < 3; ++d) {
      P[a][d] = V1[a][d] - Pp[0][d];
      Q[a][d] = V2[a][d] - Qp[0][d];
    }
  PairCoef pc;
  load_w(lam, U, ld, nrhs, e1, e2, sl1, sl2, t1 != t2, pc);
  make_coef(P, Q, pc);
  PairAcc A;
  A.I0 = A.Mxy = Cx{0, 0};
  for (int d = 0; d < 3; ++d) A.Mx[d] = A.My[d] = Cx{0, 0};
  double gp[3][3] = {}, gq[3][3] = {};  // gradients w.r.t. the permuted vertices
  const int n2 = nss * nss, n4 = n2 * n2;
  auto visit = [&](double u1, double u2, double w1, double w2, double wt) {
    double ax[3], ay[3], x[3], y[3], dv[3];
    chi_bary(u1, u2, ax);
    chi_bary(w1, w2, ay);
    for (int d = 0; d < 3; ++d) {
      x[d] = u1 * (Pp[1][d] - Pp[0][d]) + u2 * (Pp[2][d] - Pp[1][d]);
      y[d] = w1 * (Qp[1][d] - Qp[0][d]) + w2 * (Qp[2][d] - Qp[1][d]);
      dv[d] = x[d] - y[d];
    }
    double gx[3] = {0, 0, 0}, gy[3] = {0, 0, 0};
    point_pair(k, pc, x, y, dv, 4.0 * wt * kInv4Pi, gx, gy, A);
    for (int a = 0; a < 3; ++a)
      for (int d = 0; d < 3; ++d) {
        gp[a][d] += ax[a] * gx[d];
        gq[a][d] += ay[a] * gy[d];
      }
  };
  for (int idx = threadIdx.x; idx < n4; idx += blockDim.x) {
    int a = idx / (n2 * nss), b = (idx / n2) % nss, c = (idx / nss) % nss, d = idx % nss;
    double xi = c_glx[a], e1 = c_glx[b], e2 = c_glx[c], e3 = c_glx[d];
    double w4 = c_glw[a] * c_glw[b] * c_glw[c] * c_glw[d];
    if (tp.kind == 3) {
      double w = w4 * xi * xi * xi * e1 * e1 * e2;
      visit(xi, xi * (1 - e1 + e1 * e2), xi * (1 - e1 * e2 * e3), xi * (1 - e1), w);
      visit(xi * (1 - e1 * e2 * e3), xi * (1 - e1), xi, xi * (1 - e1 + e1 * e2), w);
      visit(xi, xi * e1 * (1 - e2 + e2 * e3), xi * (1 - e1 * e2), xi * e1 * (1 - e2), w);
      visit(xi * (1 - e1 * e2), xi * e1 * (1 - e2), xi, xi * e1 * (1 - e2 + e2 * e3), w);
      visit(xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3), xi, xi * e1 * (1 - e2), w);
      visit(xi, xi * e1 * (1 - e2), xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3), w);
    } else if (tp.kind == 2) {
      double w0 = w4 * xi * xi * xi * e1 * e1, w1 = w0 * e2;
      visit(xi, xi * e1 * e3, xi * (1 - e1 * e2), xi * e1 * (1 - e2), w0);
      visit(xi, xi * e1, xi * (1 - e1 * e2 * e3), xi * e1 * e2 * (1 - e3), w1);
      visit(xi * (1 - e1 * e2), xi * e1 * (1 - e2), xi, xi * e1 * e2 * e3, w1);
      visit(xi * (1 - e1 * e2 * e3), xi * e1 * e2 * (1 - e3), xi, xi * e1, w1);
      visit(xi * (1 - e1 * e2 * e3), xi * e1 * (1 - e2 * e3), xi, xi * e1 * e2, w1);
    } else {
      double w = w4 * xi * xi * xi * e2;
      visit(xi, xi * e1, xi * e2, xi * e2 * e3, w);
      visit(xi * e2, xi * e2 * e3, xi, xi * e1, w);
    }
  }
  // block reduction: 18 + 18 point-chained reals and the 16 moment reals
  __shared__ double red[4][52];
  double vals[52];
  int o = 0;
  for (int a = 0; a < 3; ++a)
    for (int d = 0; d < 3; ++d) {
      vals[o++] = gp[a][d];
      vals[o++] = gq[a][d];
    }
  vals[o++] = A.I0.r; vals[o++] = A.I0.i; vals[o++] = A.Mxy.r; vals[o++] = A.Mxy.i;
  for (int d = 0; d < 3; ++d) {
    vals[o++] = A.Mx[d].r; vals[o++] = A.Mx[d].i; vals[o++] = A.My[d].r; vals[o++] = A.My[d].i;
  }
  for (int i = 0; i < 52; ++i) {
    double v = vals[i];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    vals[i] = v;
  }
  if ((threadIdx.x & 31) == 0)
    for (int i = 0; i < 52; ++i) red[threadIdx.x >> 5][i] = vals[i];
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int i = 0; i < 52; ++i) vals[i] = red[0][i] + red[1][i] + red[2][i] + red[3][i];
  o = 0;
  for (int a = 0; a < 3; ++a)
    for (int d = 0; d < 3; ++d) {
      gp[a][d] = vals[o++];
      gq[a][d] = vals[o++];
    }
  A.I0 = {vals[o], vals[o + 1]}; o += 2;
  A.Mxy = {vals[o], vals[o + 1]}; o += 2;
  for (int d = 0; d < 3; ++d) {
    A.Mx[d] = {vals[o], vals[o + 1]};
    A.My[d] = {vals[o + 2], vals[o + 3]};
    o += 4;
  }
  double gP[3][3], gQ[3][3], gl1[3], gl2[3];
  explicit_terms(k, pc, A, P, Q, l1, l2, gP, gQ, gl1, gl2);
  double g1[3][3], g2[3][3];
  for (int a = 0; a < 3; ++a)
    for (int d = 0; d < 3; ++d) {
      g1[a][d] = gP[a][d];
      g2[a][d] = gQ[a][d];
    }
  chain_lengths(V1, l1, gl1, g1);
  chain_lengths(V2, l2, gl2, g2);
  for (int a = 0; a < 3; ++a) {
    add_grad(grad, v1[a], g1[a], -1.0);
    add_grad(grad, v2[a], g2[a], -1.0);
    add_grad(grad, tp.p[a], gp[a], -1.0);
    add_grad(grad, tp.q[a], gq[a], -1.0);
  }
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
    adjoint_singular_kernel<<<unsigned(m.ntouch), 128, 0, s>>>(m, k, nss, lam, U, ld, nrhs, grad);
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
