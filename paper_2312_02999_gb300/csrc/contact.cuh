// Point-triangle / edge-edge distance, closest-feature classification and the
// PSD-projected IPC barrier Hessian of one pair (device, float64).
//
// Sec. 2.2: every vertex-triangle and edge-edge pair k of the proxy with
// unsigned distance d_k < d0 contributes kappa * b(d_k) (Eq. 3).  Reading of
// the unprinted barrier: b(d) = -(d - dhat)^2 ln(d / dhat).
//
// Distance structure used here: the closest points are an affine combination
// v = sum_i c_i(beta) X_i of the pair's four vertices, with beta the k <= 2
// free parameters of the closest-feature case (face interior: k = 2, edge
// interior: k = 1, vertex: k = 0; edge-edge interior: k = 2 ...).  With
// f(x, beta) = |v|^2 minimised over beta, the envelope theorem and implicit
// differentiation give
//   grad d^2 = 2 c (x) v,
//   hess d^2 = 2 (c c^T) (x) I_3 - F (2 E^T E)^-1 F^T,
//   F_k = 2 (c'_k (x) v + c (x) E_k),  E_k = sum_i c'_k[i] X_i = dv/dbeta_k.
// Both live in the (3 + k)-dimensional span of {c^ (x) e_a} u {q_m (x) v^}
// where (c^, q_1.. q_k) orthonormalises (c, c'_1.. c'_k) in R^4, so the 12x12
// pair Hessian kappa (b'' grad d grad d^T + b' hess d) is formed, projected
// onto the PSD cone (PositiveDefinite of Algorithm 1) and lifted back exactly
// in that small basis.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace fsim {

// Classification threshold for nearly parallel edges (no mollifier: those
// pairs take the closest of the four endpoint-to-segment distances).
#define FSIM_PARALLEL_EPS 1e-10

struct PairGeom {
  double c[4];      // affine coefficients, v = sum_i c_i X_i
  double cp[2][4];  // d c / d beta_k
  int k;            // number of free parameters (0..2)
  double v[3];      // difference vector of the closest points
  double d2;        // |v|^2
};

__device__ __forceinline__ double dot3(const double* a, const double* b) {
  return fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0]));
}

// Closest point of segment [A, B] to P: clamped parameter and squared distance.
__device__ __forceinline__ void seg_closest(const double* P, const double* A, const double* B,
                                            double& t, double& d2) {
  double e[3] = {B[0] - A[0], B[1] - A[1], B[2] - A[2]};
  double r[3] = {P[0] - A[0], P[1] - A[1], P[2] - A[2]};
  t = dot3(r, e) / dot3(e, e);
  t = fmin(fmax(t, 0.0), 1.0);
  double q[3] = {P[0] - (A[0] + t * e[0]), P[1] - (A[1] + t * e[1]), P[2] - (A[2] + t * e[2])};
  d2 = dot3(q, q);
}

__device__ __forceinline__ void geom_finish(PairGeom& g, const double X[4][3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d)
    g.v[d] = fma(g.c[3], X[3][d], fma(g.c[2], X[2][d], fma(g.c[1], X[1][d], g.c[0] * X[0][d])));
  g.d2 = dot3(g.v, g.v);
}

// point X[0] vs triangle X[1..3]
__device__ void pt_geometry(const double X[4][3], PairGeom& g) {
  const double* p = X[0];
  const double* a = X[1];
  const double* b = X[2];
  const double* c = X[3];
  double e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
  double e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
  double r[3] = {p[0] - a[0], p[1] - a[1], p[2] - a[2]};
  double a11 = dot3(e1, e1), a12 = dot3(e1, e2), a22 = dot3(e2, e2);
  double r1 = dot3(e1, r), r2 = dot3(e2, r);
  // (products and sums fused explicitly: pair_features_warp rounds alike)
  double det = fma(a11, a22, -(a12 * a12));
  double u = fma(a22, r1, -(a12 * r2)) / det;
  double w = fma(a11, r2, -(a12 * r1)) / det;
#pragma unroll
  for (int i = 0; i < 4; ++i) { g.c[i] = 0.0; g.cp[0][i] = 0.0; g.cp[1][i] = 0.0; }
  if (u >= 0.0 && w >= 0.0 && u + w <= 1.0) {
    g.k = 2;
    g.c[0] = 1.0; g.c[1] = -(1.0 - u - w); g.c[2] = -u; g.c[3] = -w;
    g.cp[0][1] = 1.0; g.cp[0][2] = -1.0;   // d/du
    g.cp[1][1] = 1.0; g.cp[1][3] = -1.0;   // d/dw
  } else {
    double t0, d0, t1, d1, t2, d2;
    seg_closest(p, a, b, t0, d0);
    seg_closest(p, b, c, t1, d1);
    seg_closest(p, c, a, t2, d2);
    int k = 0; double t = t0, dm = d0;
    if (d1 < dm) { k = 1; t = t1; dm = d1; }
    if (d2 < dm) { k = 2; t = t2; dm = d2; }
    const int ia = 1 + k, ib = 1 + (k + 1) % 3;   // pair-local ids of the edge
    g.c[0] = 1.0;
    if (t > 0.0 && t < 1.0) {
      g.k = 1;
      g.c[ia] = -(1.0 - t); g.c[ib] = -t;
      g.cp[0][ia] = 1.0; g.cp[0][ib] = -1.0;
    } else {
      g.k = 0;
      g.c[t <= 0.0 ? ia : ib] = -1.0;
    }
  }
  geom_finish(g, X);
}

// edge X[0]X[1] vs edge X[2]X[3]
__device__ void ee_geometry(const double X[4][3], PairGeom& g) {
  const double* a0 = X[0];
  const double* a1 = X[1];
  const double* b0 = X[2];
  const double* b1 = X[3];
  double u[3] = {a1[0] - a0[0], a1[1] - a0[1], a1[2] - a0[2]};
  double v[3] = {b1[0] - b0[0], b1[1] - b0[1], b1[2] - b0[2]};
  double w0[3] = {a0[0] - b0[0], a0[1] - b0[1], a0[2] - b0[2]};
  double A = dot3(u, u), B = dot3(u, v), C = dot3(v, v), D = dot3(u, w0), E = dot3(v, w0);
  double den = fma(A, C, -(B * B));
#pragma unroll
  for (int i = 0; i < 4; ++i) { g.c[i] = 0.0; g.cp[0][i] = 0.0; g.cp[1][i] = 0.0; }
  bool interior = false;
  if (den > FSIM_PARALLEL_EPS * A * C) {
    double s = fma(B, E, -(C * D)) / den;
    double t = fma(A, E, -(B * D)) / den;
    if (s > 0.0 && s < 1.0 && t > 0.0 && t < 1.0) {
      interior = true;
      g.k = 2;
      g.c[0] = 1.0 - s; g.c[1] = s; g.c[2] = -(1.0 - t); g.c[3] = -t;
      g.cp[0][0] = -1.0; g.cp[0][1] = 1.0;
      g.cp[1][2] = 1.0; g.cp[1][3] = -1.0;
    }
  }
  if (!interior) {
    double ta0, da0, ta1, da1, tb0, db0, tb1, db1;
    seg_closest(a0, b0, b1, ta0, da0);
    seg_closest(a1, b0, b1, ta1, da1);
    seg_closest(b0, a0, a1, tb0, db0);
    seg_closest(b1, a0, a1, tb1, db1);
    int k = 0; double t = ta0, dm = da0;
    if (da1 < dm) { k = 1; t = ta1; dm = da1; }
    if (db0 < dm) { k = 2; t = tb0; dm = db0; }
    if (db1 < dm) { k = 3; t = tb1; dm = db1; }
    const bool mid = t > 0.0 && t < 1.0;
    if (k < 2) {            // point a_k vs segment b: v = a_k - (b0 + t (b1 - b0))
      g.c[k] = 1.0;
      if (mid) {
        g.k = 1; g.c[2] = -(1.0 - t); g.c[3] = -t;
        g.cp[0][2] = 1.0; g.cp[0][3] = -1.0;
      } else {
        g.k = 0; g.c[t <= 0.0 ? 2 : 3] = -1.0;
      }
    } else {                // point b_(k-2) vs segment a: v = (a0 + t (a1 - a0)) - b
      g.c[k] = -1.0;
      if (mid) {
        g.k = 1; g.c[0] = 1.0 - t; g.c[1] = t;
        g.cp[0][0] = -1.0; g.cp[0][1] = 1.0;
      } else {
        g.k = 0; g.c[t <= 0.0 ? 0 : 1] = 1.0;
      }
    }
  }
  geom_finish(g, X);
}

__device__ __forceinline__ void pair_geometry(int type, const double X[4][3], PairGeom& g) {
  if (type == 0) pt_geometry(X, g);
  else ee_geometry(X, g);
}

__device__ __forceinline__ double pair_distance(int type, const double X[4][3]) {
  PairGeom g;
  pair_geometry(type, X, g);
  return sqrt(g.d2);
}

// float32 distance of a pair given in coordinates relative to its first
// vertex (rounding error ~1e-7 of the pair's own extent).  Used only as a
// conservative filter: callers act on it only when it is far (>= 2x) from
// the threshold they test, so the float64 decision is never changed.
__device__ __forceinline__ float seg_d2f(const float* P, const float* A, const float* B) {
  const float e0 = B[0] - A[0], e1 = B[1] - A[1], e2 = B[2] - A[2];
  const float r0 = P[0] - A[0], r1 = P[1] - A[1], r2 = P[2] - A[2];
  const float ee = e0 * e0 + e1 * e1 + e2 * e2;
  float t = ee > 0.f ? (r0 * e0 + r1 * e1 + r2 * e2) / ee : 0.f;
  t = fminf(fmaxf(t, 0.f), 1.f);
  const float q0 = r0 - t * e0, q1 = r1 - t * e1, q2 = r2 - t * e2;
  return q0 * q0 + q1 * q1 + q2 * q2;
}

__device__ float pair_distance_f(int type, const float X[4][3]) {
  if (type == 0) {
    const float* p = X[0]; const float* a = X[1]; const float* b = X[2]; const float* c = X[3];
    const float e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    const float e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
    const float r[3] = {p[0] - a[0], p[1] - a[1], p[2] - a[2]};
    const float a11 = e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2];
    const float a12 = e1[0] * e2[0] + e1[1] * e2[1] + e1[2] * e2[2];
    const float a22 = e2[0] * e2[0] + e2[1] * e2[1] + e2[2] * e2[2];
    const float r1 = e1[0] * r[0] + e1[1] * r[1] + e1[2] * r[2];
    const float r2 = e2[0] * r[0] + e2[1] * r[1] + e2[2] * r[2];
    const float det = a11 * a22 - a12 * a12;
    if (det > 0.f) {
      const float u = (a22 * r1 - a12 * r2) / det, w = (a11 * r2 - a12 * r1) / det;
      if (u >= 0.f && w >= 0.f && u + w <= 1.f) {
        const float q0 = r[0] - u * e1[0] - w * e2[0], q1 = r[1] - u * e1[1] - w * e2[1],
                    q2 = r[2] - u * e1[2] - w * e2[2];
        return sqrtf(q0 * q0 + q1 * q1 + q2 * q2);
      }
    }
    return sqrtf(fminf(fminf(seg_d2f(p, a, b), seg_d2f(p, b, c)), seg_d2f(p, c, a)));
  }
  const float* a0 = X[0]; const float* a1 = X[1]; const float* b0 = X[2]; const float* b1 = X[3];
  const float u[3] = {a1[0] - a0[0], a1[1] - a0[1], a1[2] - a0[2]};
  const float v[3] = {b1[0] - b0[0], b1[1] - b0[1], b1[2] - b0[2]};
  const float w0[3] = {a0[0] - b0[0], a0[1] - b0[1], a0[2] - b0[2]};
  const float A = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const float B = u[0] * v[0] + u[1] * v[1] + u[2] * v[2];
  const float C = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  const float D = u[0] * w0[0] + u[1] * w0[1] + u[2] * w0[2];
  const float E = v[0] * w0[0] + v[1] * w0[1] + v[2] * w0[2];
  const float den = A * C - B * B;
  if (den > 1e-6f * A * C) {
    const float s = (B * E - C * D) / den, t = (A * E - B * D) / den;
    if (s > 0.f && s < 1.f && t > 0.f && t < 1.f) {
      const float q0 = w0[0] + s * u[0] - t * v[0], q1 = w0[1] + s * u[1] - t * v[1],
                  q2 = w0[2] + s * u[2] - t * v[2];
      return sqrtf(q0 * q0 + q1 * q1 + q2 * q2);
    }
  }
  return sqrtf(fminf(fminf(seg_d2f(a0, b0, b1), seg_d2f(a1, b0, b1)),
                     fminf(seg_d2f(b0, a0, a1), seg_d2f(b1, a0, a1))));
}

// X relative to its first vertex, in float32
__device__ __forceinline__ void to_rel_f(const double X[4][3], float Y[4][3]) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int d = 0; d < 3; ++d) Y[k][d] = (float)(X[k][d] - X[0][d]);
}

// First two derivatives of the IPC barrier (reading of Eq. 3's b).
__device__ __forceinline__ void barrier_derivatives(double d, double inv_d, double dhat, double& b1,
                                                    double& b2) {
  const double u = d - dhat;
  const double L2 = 2.0 * log(d / dhat);
  const double q = u * inv_d;
  b1 = -u * (L2 + q);
  b2 = fma(q, q, -fma(4.0, q, L2));
}

__device__ __forceinline__ double barrier_value(double d, double dhat) {
  if (!(d < dhat)) return 0.0;
  const double u = d - dhat;
  return -u * u * log(d / dhat);
}

// The pair Hessian kappa (b'' grad d grad d^T + b' hess d) in the reduced
// basis {c^ (x) e_a} u {q_m (x) v^} (n = 3 + k <= 5 coordinates), before the
// PSD projection, with everything the lift back to the 12x12 blocks needs.
struct PairReduced {
  int n, k;
  double d;            // unsigned distance
  double gfac;         // kappa b'(d): gradient of vertex i = gfac c_i v^
  double c[4];         // affine coefficients
  double ch[4];        // c / |c|
  double q[2][4];      // orthonormal complement directions in R^4
  double vh[3];        // v / |v|
  double A[5][5];      // reduced Hessian (n x n used)
};

// The cost is float64 instructions (one per warp every 66 cycles per SM
// sub-partition, and a division is about 16 of them), so the divisions are
// reciprocals shared by their numerators, products feeding sums are fused,
// and only the upper triangle is formed.  With F' = F / 2 (F as at the top of
// this file) the reduced Hessian is
//   K2 v^ v^T + K1 (|c|^2 (I - v^ v^T) - F' (E^T E)^-1 F'^T),
//   K1 = kappa b' / d, K2 = kappa b'' |c|^2:
// the two parts that nearly cancel near a face or an edge interior are
// subtracted before the factor 1 / d.
__device__ __forceinline__ double dot4(const double* a, const double* b) {
  return fma(a[3], b[3], fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0])));
}

__device__ void pair_reduced(int type, const double X[4][3], double dhat, double kappa,
                             PairReduced& r) {
  PairGeom g;
  pair_geometry(type, X, g);
  const double d = sqrt(g.d2);
  const double inv_d = 1.0 / d;
  double b1, b2;
  barrier_derivatives(d, inv_d, dhat, b1, b2);
  const int k = g.k, n = 3 + k;
  r.n = n; r.k = k; r.d = d; r.gfac = kappa * b1;
  // orthonormal (c^, q_1 .. q_k) in R^4 by Gram-Schmidt; the coefficients
  // c^ . c'_k and q_m . c'_k of c'_k come out of it (q_2 . c'_1 = 0)
  const double cn2 = dot4(g.c, g.c);
  const double cn = sqrt(cn2), icn = 1.0 / cn;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    r.c[i] = g.c[i];
    r.ch[i] = g.c[i] * icn;
    r.q[0][i] = 0.0;
    r.q[1][i] = 0.0;
  }
  double chc[2] = {0.0, 0.0}, q00 = 0.0, q01 = 0.0, q11 = 0.0;
  double E[2][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    if (kk >= k) continue;
    chc[kk] = dot4(r.ch, g.cp[kk]);
    double w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = fma(-chc[kk], r.ch[i], g.cp[kk][i]);
    if (kk == 1) {
      q01 = dot4(r.q[0], w);
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i] = fma(-q01, r.q[0][i], w[i]);
    }
    const double w2 = dot4(w, w), iw = rsqrt(w2);
    if (kk == 0) q00 = w2 * iw;
    else q11 = w2 * iw;
#pragma unroll
    for (int i = 0; i < 4; ++i) r.q[kk][i] = w[i] * iw;
#pragma unroll
    for (int dd = 0; dd < 3; ++dd)
      E[kk][dd] = fma(g.cp[kk][3], X[3][dd],
                      fma(g.cp[kk][2], X[2][dd], fma(g.cp[kk][1], X[1][dd], g.cp[kk][0] * X[0][dd])));
  }
  // F' and (E^T E)^-1 F'^T
  double F[5][2], T[5][2];
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
    for (int a = 0; a < 3; ++a) F[a][kk] = kk < k ? fma(chc[kk], g.v[a], cn * E[kk][a]) : 0.0;
  }
  F[3][0] = q00 * d; F[3][1] = q01 * d;
  F[4][0] = 0.0;     F[4][1] = q11 * d;
  double G00 = 0.0, G01 = 0.0, G11 = 0.0;      // (E^T E)^-1
  if (k > 0) {
    const double e00 = dot3(E[0], E[0]);
    if (k == 1) {
      G00 = 1.0 / e00;
    } else {
      const double e01 = dot3(E[0], E[1]), e11 = dot3(E[1], E[1]);
      const double id = 1.0 / fma(e00, e11, -(e01 * e01));
      G00 = e11 * id; G01 = -e01 * id; G11 = e00 * id;
    }
  }
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    T[i][0] = fma(G00, F[i][0], G01 * F[i][1]);
    T[i][1] = fma(G01, F[i][0], G11 * F[i][1]);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) r.vh[a] = g.v[a] * inv_d;
  const double K1 = r.gfac * inv_d, K2 = kappa * b2 * cn2;
#pragma unroll
  for (int i = 0; i < 5; ++i)
#pragma unroll
    for (int j = i; j < 5; ++j) {
      double h = 0.0;
      if (i < n && j < n) {
        h = -fma(F[i][0], T[j][0], F[i][1] * T[j][1]);
        if (j < 3) {
          const double vv = r.vh[i] * r.vh[j];
          h = fma(cn2, (i == j ? 1.0 : 0.0) - vv, h);
          h = fma(K1, h, K2 * vv);
        } else {
          h *= K1;
        }
      }
      r.A[i][j] = h;
      r.A[j][i] = h;
    }
}

// Workspace of the one-warp forms, where the lanes share a pair's float64 work.
struct PairWarp {
  double X[4][3];       // the pair's vertices
  double D[3][3];       // edge vectors, vertex difference
  double C[3][4];       // c, c'_1, c'_2
  double W[3][4];       // v, E_1, E_2 (last entry 0)
  double Q[3][4];       // c^, q_1, q_2
  double F[5][2], T[5][2];
  double vh[3];
};

// Closest features of the pair at w.X (visible to the warp): its number of free
// parameters; C = c, c'_1, c'_2.  One lane per difference component, dot product,
// quotient and segment: about 25 float64 instructions where one lane needs 70
// (interior features), 65 where it needs 180.
__device__ __forceinline__ int pair_features_warp(int type, int lane, PairWarp& w) {
  constexpr unsigned full = 0xffffffffu;
  int k;
  if (lane < 9) {       // PT: b - a, c - a, p - a;  EE: a1 - a0, b1 - b0, a0 - b0
    const int q = lane / 3, dd = lane % 3;
    const int hi = type == 0 ? (q == 0 ? 2 : q == 1 ? 3 : 0) : (q == 0 ? 1 : q == 1 ? 3 : 0);
    const int lo = type == 0 ? 1 : (q == 0 ? 0 : 2);
    w.D[q][dd] = w.X[hi][dd] - w.X[lo][dd];
  }
  __syncwarp();
  double m = 0.0;
  if (lane < 5) {       // 0.0, 0.1, 1.1, 0.2, 1.2
    const int a = lane == 2 || lane == 4, b = lane == 0 ? 0 : lane < 3 ? 1 : 2;
    m = dot3(w.D[a], w.D[b]);
  }
  const double m0 = __shfl_sync(full, m, 0), m1 = __shfl_sync(full, m, 1),
               m2 = __shfl_sync(full, m, 2), m3 = __shfl_sync(full, m, 3),
               m4 = __shfl_sync(full, m, 4);
  const double det = fma(m0, m2, -(m1 * m1));
  const bool odd = lane & 1, ee = type != 0;
  // even lanes (a22 r1 - a12 r2) / det or (B E - C D) / det, odd (m0 m4 - m1 m3) / det
  const double par = fma(odd ? m0 : ee ? m1 : m2, odd || ee ? m4 : m3,
                         -((ee && !odd ? m2 : m1) * (odd || ee ? m3 : m4))) / det;
  const double pu = __shfl_sync(full, par, 0), pt = __shfl_sync(full, par, 1);
  bool inside;
  if (type == 0) {
    inside = pu >= 0.0 && pt >= 0.0 && pu + pt <= 1.0;
  } else {
    inside = det > FSIM_PARALLEL_EPS * m0 * m2 && pu > 0.0 && pu < 1.0 && pt > 0.0 && pt < 1.0;
  }
  double c = 0.0, c1 = 0.0, c2 = 0.0;             // this lane's vertex (lanes 0 .. 3)
  const int i4 = lane & 3;
  if (inside) {
    k = 2;
    if (type == 0) {
      c = i4 == 0 ? 1.0 : i4 == 1 ? -(1.0 - pu - pt) : i4 == 2 ? -pu : -pt;
      c1 = i4 == 1 ? 1.0 : i4 == 2 ? -1.0 : 0.0;
      c2 = i4 == 1 ? 1.0 : i4 == 3 ? -1.0 : 0.0;
    } else {
      const double f = i4 < 2 ? pu : pt;
      c = (odd ? f : 1.0 - f) * (i4 < 2 ? 1.0 : -1.0);
      c1 = i4 == 0 ? -1.0 : i4 == 1 ? 1.0 : 0.0;
      c2 = i4 == 2 ? 1.0 : i4 == 3 ? -1.0 : 0.0;
    }
  } else {
    // lane l: feature l, a point against a segment (PT: three, EE: four)
    const int nseg = type == 0 ? 3 : 4;
    auto feature = [&](int l, int& P, int& A, int& B) {
      if (type == 0) { P = 0; A = 1 + l; B = l == 2 ? 1 : 2 + l; }
      else { P = l; A = l < 2 ? 2 : 0; B = A + 1; }
    };
    int P, A, B;
    feature(i4 < nseg ? i4 : nseg - 1, P, A, B);
    double ts, ds;
    seg_closest(w.X[P], w.X[A], w.X[B], ts, ds);
    int best = 0;
    double dm = __shfl_sync(full, ds, 0);
    for (int l = 1; l < nseg; ++l) {
      const double dl = __shfl_sync(full, ds, l);
      if (dl < dm) { best = l; dm = dl; }
    }
    const double t = __shfl_sync(full, ts, best);
    feature(best, P, A, B);
    const double sg = type == 1 && best >= 2 ? -1.0 : 1.0;
    const bool mid = t > 0.0 && t < 1.0;
    k = mid ? 1 : 0;
    const double tb = mid ? t : t <= 0.0 ? 0.0 : 1.0;
    c = i4 == P ? sg : i4 == A ? -sg * (1.0 - tb) : i4 == B ? -sg * tb : 0.0;
    if (mid) c1 = i4 == A ? sg : i4 == B ? -sg : 0.0;
  }
  if (lane < 4) { w.C[0][lane] = c; w.C[1][lane] = c1; w.C[2][lane] = c2; }
  __syncwarp();
  return k;
}

// pair_reduced by the lanes of one warp.  The chain of one pair is float64
// instructions (66 cycles each, however many lanes are active), about 500 of them
// when every lane runs pair_reduced; here the entries of each small vector or
// matrix sit in different lanes and one instruction forms them all: about 140
// (interior features) to 180.  Divisions and square roots are taken in one go
// each: with the Gram matrix M of the c'_k off c, scaled by |c|^2 (M_ij = |c|^2
// c'_i.c'_j - (c.c'_i)(c.c'_j), D = det M),
//   q_1 = (|c|^2 c'_1 - (c.c'_1) c) r2,                        r2 = (|c|^2 M_11)^-1/2,
//   q_2 = (|c|^2 c'_2 - (c.c'_2) c - |c|^2 (q_1.c'_2) q_1) M_11 r3,
//                                                             r3 = (|c|^2 M_11 D)^-1/2,
//   q_1.c'_1 = M_11 r2,  q_1.c'_2 = M_12 r2,  q_2.c'_2 = D r3,
// so that four reciprocal square roots (those of |v|^2 and |c|^2 too) need nothing
// but dot products, and 2 log(d / dhat) = log(|v|^2 / dhat^2).
// The workspace afterwards holds what the lift needs (C[0] = c, Q = c^, q_1, q_2
// and vh); lane l < 15 returns the entry (i, j), i <= j, of the reduced Hessian.
__device__ __forceinline__ double pair_reduced_warp(int type, const double* __restrict__ s,
                                                    const int V[4], double dhat, double kappa,
                                                    int lane, PairWarp& w, int& k, double& gfac,
                                                    int& ri, int& rj) {
  constexpr unsigned full = 0xffffffffu;
  if (lane < 12) {
    const int v = lane < 3 ? V[0] : lane < 6 ? V[1] : lane < 9 ? V[2] : V[3];
    w.X[lane / 3][lane % 3] = s[3 * (size_t)v + lane % 3];
  }
  __syncwarp();
  k = pair_features_warp(type, lane, w);
  const bool odd = lane & 1;
  const int i4 = lane & 3;
  if (lane < 9) {
    const double* cr = w.C[lane / 3];
    const int dd = lane % 3;
    w.W[lane / 3][dd] =
        fma(cr[3], w.X[3][dd], fma(cr[2], w.X[2][dd], fma(cr[1], w.X[1][dd], cr[0] * w.X[0][dd])));
  } else if (lane < 12) {
    w.W[lane - 9][3] = 0.0;
  }
  __syncwarp();
  double g = 0.0;
  if (lane < 10) {      // v.v, E1.E1, E1.E2, E2.E2;  c.c, c.c1, c.c2, c1.c1, c1.c2, c2.c2
    const int a = lane < 4 ? (0x2110 >> (4 * lane)) & 3 : (0x211000 >> (4 * (lane - 4))) & 3;
    const int b = lane < 4 ? (0x2210 >> (4 * lane)) & 3 : (0x221210 >> (4 * (lane - 4))) & 3;
    const double(*base)[4] = lane < 4 ? w.W : w.C;
    g = dot4(base[a], base[b]);
  }
  const double d2 = __shfl_sync(full, g, 0), cn2 = __shfl_sync(full, g, 4),
               a1 = __shfl_sync(full, g, 5), a2 = __shfl_sync(full, g, 6);
  const double e00 = k > 0 ? __shfl_sync(full, g, 1) : 1.0;
  const double e01 = k > 1 ? __shfl_sync(full, g, 2) : 0.0;
  const double e11 = k > 1 ? __shfl_sync(full, g, 3) : 1.0;
  // M: entries 1.1, 1.2, 2.2 in lanes 7, 8, 9
  const double mm = fma(-(lane == 9 ? a2 : a1), lane == 7 ? a1 : a2, cn2 * g);
  const double M00 = k > 0 ? __shfl_sync(full, mm, 7) : 1.0;
  const double M01 = k > 1 ? __shfl_sync(full, mm, 8) : 0.0;
  const double M11 = k > 1 ? __shfl_sync(full, mm, 9) : 1.0;
  const double DD = fma(M00, M11, -(M01 * M01));
  const double cM = cn2 * M00;
  // 1 / det(E^T E) and |v|^2 / dhat^2; the reciprocal square roots
  const double qt = (odd ? d2 : 1.0) / (odd ? dhat * dhat : fma(e00, e11, -(e01 * e01)));
  const double id = __shfl_sync(full, qt, 0), L2 = log(__shfl_sync(full, qt, 1));
  const double rr = rsqrt(i4 == 0 ? d2 : i4 == 1 ? cn2 : i4 == 2 ? cM : cM * DD);
  const double inv_d = __shfl_sync(full, rr, 0), icn = __shfl_sync(full, rr, 1),
               r2 = __shfl_sync(full, rr, 2), r3 = __shfl_sync(full, rr, 3);
  double d = d2 * inv_d;
  d = fma(fma(-d, d, d2), 0.5 * inv_d, d);
  const double u = d - dhat, q = u * inv_d;
  gfac = kappa * (-u * (L2 + q));
  const double K1 = gfac * inv_d, K2 = kappa * fma(q, q, -fma(4.0, q, L2)) * cn2;
  const double q01 = M01 * r2;                                   // (0 unless k = 2)
  // c^; lanes 0 .. 3 q_1, lanes 4 .. 7 q_2
  const double t = fma(cn2, w.C[lane & 4 ? 2 : 1][i4], -((lane & 4 ? a2 : a1) * w.C[0][i4]));
  const double q1 = t * r2;
  const double q1i = __shfl_sync(full, q1, i4);
  const double q2 = fma(-cn2 * q01, q1i, t) * (M00 * r3);
  if (lane < 4) {
    w.Q[0][lane] = w.C[0][lane] * icn;
    w.Q[1][lane] = k > 0 ? q1 : 0.0;
  } else if (lane < 8) {
    w.Q[2][i4] = k > 1 ? q2 : 0.0;
  }
  const int fa = lane >> 1;
  double f = 0.0;
  if (fa < 3) {
    const double ch = (odd ? a2 : a1) * icn;
    f = fma(ch, w.W[0][fa], cn2 * icn * w.W[1 + odd][fa]);
  } else if (fa == 3) {
    f = (odd ? q01 : M00 * r2) * d;
  } else if (odd) {
    f = DD * r3 * d;
  }
  f = (odd ? k > 1 : k > 0) ? f : 0.0;
  if (lane < 10) w.F[fa][odd] = f;
  else if (lane < 13) w.vh[lane - 10] = w.W[0][lane - 10] * inv_d;
  // (E^T E)^-1 F'^T: the two entries of row fa sit in neighbouring lanes
  const double fo = __shfl_xor_sync(full, f, 1);
  if (lane < 10) w.T[fa][odd] = fma((odd ? e00 : e11) * id, f, -(e01 * id) * fo);
  __syncwarp();
  const int l15 = lane < 15 ? lane : 14;
  ri = (int)(0x433222111100000ull >> (4 * l15)) & 7;
  rj = (int)(0x443432432143210ull >> (4 * l15)) & 7;
  const double vv = rj < 3 ? w.vh[ri] * w.vh[rj] : 0.0;
  double h = -fma(w.F[ri][0], w.T[rj][0], w.F[ri][1] * w.T[rj][1]);
  if (rj < 3) h = fma(cn2, (ri == rj ? 1.0 : 0.0) - vv, h);
  h = fma(K1, h, K2 * vv);
  return rj < 3 + k ? h : 0.0;
}

// Plane rotation (c, s, t = s / c) of a cyclic Jacobi step that annihilates
// apq.  float32: the textbook formulas.  float64: t to float32 accuracy only
// (about 1e-7 of apq stays, which the next sweep removes; the diagonal is
// updated by the full products), c by one third-order step from the float32
// reciprocal square root, so c^2 + s^2 = 1 to rounding: about 14 float64
// instructions instead of about 90 for the divisions and square roots.
__device__ __forceinline__ void jacobi_rotation(float app, float aqq, float apq, float& c, float& s,
                                                float& t) {
  const float th = (aqq - app) / (2.f * apq);
  t = (th >= 0.f ? 1.f : -1.f) / (fabsf(th) + sqrtf(th * th + 1.f));
  c = 1.f / sqrtf(t * t + 1.f);
  s = t * c;
}
__device__ __forceinline__ void jacobi_rotation(double app, double aqq, double apq, double& c,
                                                double& s, double& t) {
  // a difference and an entry outside the float32 range are scaled alike
  double dif = aqq - app, two = 2.0 * apq;
  const double big = fmax(fabs(dif), fabs(two));
  if (!(big < 1e30 && big > 1e-20)) {
    dif /= big;
    two /= big;
  }
  const float th = (float)dif / (float)two;
  const float tf = (th >= 0.f ? 1.f : -1.f) / (fabsf(th) + sqrtf(fmaf(th, th, 1.f)));
  t = (double)tf;
  const double u = fma(t, t, 1.0);
  const double r0 = (double)rsqrtf((float)u);
  const double e = fma(-u * r0, r0, 1.0);
  c = fma(r0 * e, fma(0.375, e, 0.5), r0);
  s = t * c;
}

// ---------------------------------------------------------------------------
// Edge-edge mollifier (optional; IPC's treatment of nearly parallel edges):
// with c = |e_a x e_b|^2 and eps = 1e-3 |E_a|^2 |E_b|^2 at rest, the EE term
// becomes kappa m(c) b(d), m(c) = (2 - c/eps) c/eps for c < eps, else 1.
// ---------------------------------------------------------------------------
#define FSIM_MOLLIFIER_EPS_SCALE 1e-3

struct EdgeCross {
  double ea[3], eb[3];   // a1 - a0, b1 - b0
  double aa, bb, ab;     // ea.ea, eb.eb, ea.eb
  double c;              // |ea x eb|^2
};

__device__ __forceinline__ void edge_cross(const double X[4][3], EdgeCross& e) {
  for (int d = 0; d < 3; ++d) {
    e.ea[d] = X[1][d] - X[0][d];
    e.eb[d] = X[3][d] - X[2][d];
  }
  const double w0 = e.ea[1] * e.eb[2] - e.ea[2] * e.eb[1];
  const double w1 = e.ea[2] * e.eb[0] - e.ea[0] * e.eb[2];
  const double w2 = e.ea[0] * e.eb[1] - e.ea[1] * e.eb[0];
  e.c = w0 * w0 + w1 * w1 + w2 * w2;
  e.aa = dot3(e.ea, e.ea);
  e.bb = dot3(e.eb, e.eb);
  e.ab = dot3(e.ea, e.eb);
}

__device__ __forceinline__ double mollifier_value(double c, double eps) {
  if (!(c < eps)) return 1.0;
  const double q = c / eps;
  return (2.0 - q) * q;
}

// d c / d X[I][al] (vertices a0, a1, b0, b1)
__device__ __forceinline__ double edge_cross_grad(const EdgeCross& e, int I, int al) {
  const double ga = 2.0 * (e.ea[al] * e.bb - e.ab * e.eb[al]);
  const double gb = 2.0 * (e.eb[al] * e.aa - e.ab * e.ea[al]);
  const double g = (I < 2) ? ga : gb;
  return (I == 0 || I == 2) ? -g : g;
}

// d^2 c / d X[I][al] d X[J][be]
__device__ __forceinline__ double edge_cross_hess(const EdgeCross& e, int I, int al, int J, int be) {
  const double dl = (al == be) ? 1.0 : 0.0;
  const int ei = I >> 1, ej = J >> 1;     // 0: edge a, 1: edge b
  double h;
  if (ei == 0 && ej == 0) h = 2.0 * e.bb * dl - 2.0 * e.eb[al] * e.eb[be];
  else if (ei == 1 && ej == 1) h = 2.0 * e.aa * dl - 2.0 * e.ea[al] * e.ea[be];
  else if (ei == 0) h = 4.0 * e.ea[al] * e.eb[be] - 2.0 * e.eb[al] * e.ea[be] - 2.0 * e.ab * dl;
  else h = 4.0 * e.ea[be] * e.eb[al] - 2.0 * e.eb[be] * e.ea[al] - 2.0 * e.ab * dl;
  const double si = (I == 0 || I == 2) ? -1.0 : 1.0, sj = (J == 0 || J == 2) ? -1.0 : 1.0;
  return si * sj * h;
}

}  // namespace fsim
