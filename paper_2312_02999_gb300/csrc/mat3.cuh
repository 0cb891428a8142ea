// Small fixed-size linear algebra for the per-tet local step (device).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace fsim {

template <typename T>
struct M3 {
  T m[3][3];
};

template <typename T>
__device__ __forceinline__ T sqrt_t(T v);
template <>
__device__ __forceinline__ double sqrt_t<double>(double v) { return sqrt(v); }
template <>
__device__ __forceinline__ float sqrt_t<float>(float v) { return sqrtf(v); }

// a / b and 1 / sqrt(v): exact float64 operations; in float32 the fast
// hardware forms (a few ulp), which the float32 polar rotation can use
// because the mixed local step refines its rotation in double-float
// arithmetic afterwards
template <typename T>
__device__ __forceinline__ T fdiv_t(T a, T b);
template <>
__device__ __forceinline__ double fdiv_t<double>(double a, double b) { return a / b; }
template <>
__device__ __forceinline__ float fdiv_t<float>(float a, float b) { return __fdividef(a, b); }
template <typename T>
__device__ __forceinline__ T rsqrt_t(T v);
template <>
__device__ __forceinline__ double rsqrt_t<double>(double v) { return 1.0 / sqrt(v); }
template <>
__device__ __forceinline__ float rsqrt_t<float>(float v) { return rsqrtf(v); }

template <typename T>
__device__ __forceinline__ void matmul(const T A[3][3], const T B[3][3], T C[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i][j] = A[i][0] * B[0][j] + A[i][1] * B[1][j] + A[i][2] * B[2][j];
}

// C = A^T B
template <typename T>
__device__ __forceinline__ void matmul_tn(const T A[3][3], const T B[3][3], T C[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i][j] = A[0][i] * B[0][j] + A[1][i] * B[1][j] + A[2][i] * B[2][j];
}

// C = A B^T
template <typename T>
__device__ __forceinline__ void matmul_nt(const T A[3][3], const T B[3][3], T C[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) C[i][j] = A[i][0] * B[j][0] + A[i][1] * B[j][1] + A[i][2] * B[j][2];
}

template <typename T>
__device__ __forceinline__ T det3(const T A[3][3]) {
  return A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) -
         A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0]) +
         A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]);
}

// Rotation factor of the polar decomposition of M (closest rotation), by a
// one-sided (Hestenes) Jacobi SVD: plane rotations from the right
// orthogonalise the columns of M, M V = U diag(sigma) with V in SO(3).  The
// column with the smallest sigma is flipped when det M < 0, so that U is a
// rotation and R = U V^T maximises tr(R^T M) over SO(3).
template <typename T, int SWEEPS>
__device__ void polar_rotation(const T M[3][3], T R[3][3]) {
  T B[3][3], V[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      B[i][j] = M[i][j];
      V[i][j] = (i == j) ? T(1) : T(0);
    }
  const T tiny = sizeof(T) == 8 ? T(1e-300) : T(1e-30);
  const T eps = sizeof(T) == 8 ? T(1e-15) : T(1e-7);
#pragma unroll 1
  for (int sw = 0; sw < SWEEPS; ++sw) {
    T off = T(0);
#pragma unroll
    for (int pair = 0; pair < 3; ++pair) {
      const int p = pair == 2 ? 1 : 0;
      const int q = pair == 0 ? 1 : 2;
      T a = B[0][p] * B[0][p] + B[1][p] * B[1][p] + B[2][p] * B[2][p];
      T b = B[0][q] * B[0][q] + B[1][q] * B[1][q] + B[2][q] * B[2][q];
      T g = B[0][p] * B[0][q] + B[1][p] * B[1][q] + B[2][p] * B[2][q];
      T ag = fabs(g);
      if (ag > eps * sqrt_t(a * b) && ag > tiny) {
        off += ag;
        T zeta = fdiv_t(b - a, T(2) * g);
        T t = fdiv_t(zeta >= T(0) ? T(1) : T(-1), fabs(zeta) + sqrt_t(T(1) + zeta * zeta));
        T c = rsqrt_t(T(1) + t * t);
        T s = c * t;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          T bp = B[i][p], bq = B[i][q];
          B[i][p] = c * bp - s * bq;
          B[i][q] = s * bp + c * bq;
          T vp = V[i][p], vq = V[i][q];
          V[i][p] = c * vp - s * vq;
          V[i][q] = s * vp + c * vq;
        }
      }
    }
    if (off == T(0)) break;
  }
  T sig[3];
#pragma unroll
  for (int j = 0; j < 3; ++j) sig[j] = sqrt_t(B[0][j] * B[0][j] + B[1][j] * B[1][j] + B[2][j] * B[2][j]);
  int kmin = 0;
  if (sig[1] < sig[kmin]) kmin = 1;
  if (sig[2] < sig[kmin]) kmin = 2;
  // columns ka < kb are the two others; selects instead of indexing with
  // kmin keep every array in registers
  const T sa = kmin == 0 ? sig[1] : sig[0];
  const T sb = kmin == 2 ? sig[1] : sig[2];
  T a[3], b[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T ba = kmin == 0 ? B[i][1] : B[i][0];
    const T bb = kmin == 2 ? B[i][1] : B[i][2];
    a[i] = sa > tiny ? fdiv_t(ba, sa) : T(0);
    b[i] = sb > tiny ? fdiv_t(bb, sb) : T(0);
  }
  if (!(sa > tiny)) { a[0] = 1; a[1] = 0; a[2] = 0; }
  if (!(sb > tiny)) {  // any unit vector orthogonal to a
    T px = fabs(a[0]) < T(0.9) ? T(1) : T(0), py = fabs(a[0]) < T(0.9) ? T(0) : T(1), pz = T(0);
    T cx = a[1] * pz - a[2] * py, cy = a[2] * px - a[0] * pz, cz = a[0] * py - a[1] * px;
    T nn = sqrt_t(cx * cx + cy * cy + cz * cz);
    b[0] = cx / nn; b[1] = cy / nn; b[2] = cz / nn;
  }
  // the third column completes a right-handed frame in the orientation of
  // (ka, kb, kmin) inside V's frame: u_kmin = s * (u_ka x u_kb), where s is
  // the sign that makes det U = +1 for the cyclic order of the indices
  // (s = -1 only for (ka, kb, kmin) = (0, 2, 1))
  const T orient = kmin == 1 ? T(-1) : T(1);
  T c[3];
  c[0] = orient * (a[1] * b[2] - a[2] * b[1]);
  c[1] = orient * (a[2] * b[0] - a[0] * b[2]);
  c[2] = orient * (a[0] * b[1] - a[1] * b[0]);
  T U[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    U[i][0] = kmin == 0 ? c[i] : a[i];
    U[i][1] = kmin == 1 ? c[i] : (kmin == 0 ? a[i] : b[i]);
    U[i][2] = kmin == 2 ? c[i] : b[i];
  }
  // R = U V^T (V is a product of plane rotations, det V = +1)
  matmul_nt(U, V, R);
}

// Rotation factor of M by the Newton iteration X <- (X + X^-T) / 2 for the
// orthogonal polar factor (Higham 1986), X0 = M, with the Frobenius-norm scaling
// in the first step.  It needs det M > 0 and a moderate condition: false (R
// undefined) when det M is below 0.05 of the determinant of a rotation of
// the same Frobenius norm, or when it has not converged in 8 steps; the
// caller then takes polar_rotation.  Stretches of 0.5 to 2 converge in 4
// steps of about 45 float32 operations, where the Jacobi SVD takes about 900.
// The step that moves X by less than 1.6e-4 leaves an error near 1e-8, so it
// is the last one; the result is orthogonal and closest to M to a few float32
// roundings, like polar_rotation<float>.
__device__ __forceinline__ bool polar_rotation_newton(const float M[3][3], float R[3][3]) {
  float X[3][3];
  float n2 = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      X[i][j] = M[i][j];
      n2 += M[i][j] * M[i][j];
    }
  float det = det3(X);
  // the range of n2 keeps the squares and cubes below far from the ends of float32
  if (!(n2 > 1e-6f && n2 < 1e6f && det > 0.f && 27.f * det * det > 2.5e-3f * n2 * n2 * n2))
    return false;
  bool done = false;
#pragma unroll 1
  for (int it = 0; it < 8 && !done; ++it) {
    float C[3][3];      // cofactors: X^-T = C / det
    C[0][0] = X[1][1] * X[2][2] - X[1][2] * X[2][1];
    C[0][1] = X[1][2] * X[2][0] - X[1][0] * X[2][2];
    C[0][2] = X[1][0] * X[2][1] - X[1][1] * X[2][0];
    C[1][0] = X[0][2] * X[2][1] - X[0][1] * X[2][2];
    C[1][1] = X[0][0] * X[2][2] - X[0][2] * X[2][0];
    C[1][2] = X[0][1] * X[2][0] - X[0][0] * X[2][1];
    C[2][0] = X[0][1] * X[1][2] - X[0][2] * X[1][1];
    C[2][1] = X[0][2] * X[1][0] - X[0][0] * X[1][2];
    C[2][2] = X[0][0] * X[1][1] - X[0][1] * X[1][0];
    det = X[0][0] * C[0][0] + X[0][1] * C[0][1] + X[0][2] * C[0][2];
    float a = 0.5f, b = __fdividef(0.5f, det);
    if (it == 0) {      // scale by g, g^2 = |X^-1| / |X|
      float c2 = 0.f;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) c2 += C[i][j] * C[i][j];
      const float q = sqrtf(__fdividef(c2, n2 * det * det));
      const float g = sqrtf(q);
      a *= g;
      b = __fdividef(b, g);
    }
    float d2 = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const float v = a * X[i][j] + b * C[i][j];
        const float d = v - X[i][j];
        d2 += d * d;
        X[i][j] = v;
      }
    done = d2 < 2.5e-8f;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) R[i][j] = X[i][j];
  return done;
}

}  // namespace fsim
