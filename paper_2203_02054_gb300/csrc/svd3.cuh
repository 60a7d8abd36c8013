// Rotation fit of one element by a signed 3x3 SVD (the "rotation computed by
// SVD" of Eq. 1 in the paper).
//
// For D = X_c T_c^T, returns the proper rotation R = U V^T of the signed SVD
// D = U diag(s1, s2, s3) V^T with U, V in SO(3), s1 >= s2 >= |s3| and s3 of
// either sign; R maximises tr(R^T D) over SO(3) (Kabsch) and that maximum is
// s1 + s2 + s3.  Steps (the structure of McAdams et al. 2011, "Computing the
// singular value decomposition of 3x3 matrices with minimal branching and
// elementary floating point operations", with exact Jacobi angles instead of
// their approximate quaternion rotations):
//   1. cyclic Jacobi on the symmetric S = D^T D (Golub and Van Loan,
//      symmetric Schur rotations), accumulating V;
//   2. sort the eigenvalues descending, permuting the columns of V with one
//      sign flip per swap so that det V stays +1;
//   3. Givens QR of B = D V = U Sigma: U is a product of rotations and the
//      diagonal of the triangular factor holds the signed singular values.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace casim {

template <typename T>
__device__ __forceinline__ T rsqrt_t(T x);
template <>
__device__ __forceinline__ float rsqrt_t<float>(float x) { return rsqrtf(x); }
template <>
__device__ __forceinline__ double rsqrt_t<double>(double x) { return rsqrt(x); }

// One Jacobi rotation zeroing S[p][q] of the symmetric 3x3 S; V <- V J.
template <typename T>
__device__ __forceinline__ void jacobi_rotate(T S[3][3], T V[3][3], int p, int q) {
  const T spq = S[p][q];
  if (spq == T(0)) return;
  const T tau = (S[q][q] - S[p][p]) / (T(2) * spq);
  const T t = (tau >= T(0) ? T(1) : T(-1)) / (fabs(tau) + sqrt(T(1) + tau * tau));
  const T c = rsqrt_t<T>(T(1) + t * t);
  const T s = t * c;
  // S <- J^T S J with J the rotation in the (p, q) plane
  for (int k = 0; k < 3; ++k) {
    const T skp = S[k][p], skq = S[k][q];
    S[k][p] = c * skp - s * skq;
    S[k][q] = s * skp + c * skq;
  }
  for (int k = 0; k < 3; ++k) {
    const T spk = S[p][k], sqk = S[q][k];
    S[p][k] = c * spk - s * sqk;
    S[q][k] = s * spk + c * sqk;
  }
  S[p][q] = T(0);
  S[q][p] = T(0);
  for (int k = 0; k < 3; ++k) {
    const T vkp = V[k][p], vkq = V[k][q];
    V[k][p] = c * vkp - s * vkq;
    V[k][q] = s * vkp + c * vkq;
  }
}

template <typename T>
__device__ __forceinline__ void swap_cols_neg(T V[3][3], T lam[3], int a, int b) {
  T tl = lam[a];
  lam[a] = lam[b];
  lam[b] = tl;
  for (int k = 0; k < 3; ++k) {
    T t = V[k][a];
    V[k][a] = V[k][b];
    V[k][b] = -t;
  }
}

// Givens rotation acting on rows p, q of B (3x3) zeroing B[q][col]; U <- U G^T.
template <typename T>
__device__ __forceinline__ void givens_rows(T B[3][3], T U[3][3], int p, int q, int col) {
  const T a = B[p][col], b = B[q][col];
  const T r2 = a * a + b * b;
  if (!(r2 > T(0))) return;
  const T ir = rsqrt_t<T>(r2);
  const T c = a * ir, s = b * ir;
  for (int k = 0; k < 3; ++k) {
    const T bp = B[p][k], bq = B[q][k];
    B[p][k] = c * bp + s * bq;
    B[q][k] = -s * bp + c * bq;
  }
  B[q][col] = T(0);
  for (int k = 0; k < 3; ++k) {
    const T up = U[k][p], uq = U[k][q];
    U[k][p] = c * up + s * uq;
    U[k][q] = -s * up + c * uq;
  }
}

// R = U V^T (row-major 3x3) and tr(R^T D) for one D (row-major).
template <typename T, int SWEEPS>
__device__ __forceinline__ void kabsch_rotation(const T D[3][3], T R[3][3], T& trace) {
  T S[3][3], V[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      S[i][j] = D[0][i] * D[0][j] + D[1][i] * D[1][j] + D[2][i] * D[2][j];
      V[i][j] = (i == j) ? T(1) : T(0);
    }
#pragma unroll
  for (int sweep = 0; sweep < SWEEPS; ++sweep) {
    jacobi_rotate<T>(S, V, 0, 1);
    jacobi_rotate<T>(S, V, 0, 2);
    jacobi_rotate<T>(S, V, 1, 2);
  }
  T lam[3] = {S[0][0], S[1][1], S[2][2]};
  if (lam[0] < lam[1]) swap_cols_neg<T>(V, lam, 0, 1);
  if (lam[0] < lam[2]) swap_cols_neg<T>(V, lam, 0, 2);
  if (lam[1] < lam[2]) swap_cols_neg<T>(V, lam, 1, 2);
  T B[3][3], U[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      B[i][j] = D[i][0] * V[0][j] + D[i][1] * V[1][j] + D[i][2] * V[2][j];
      U[i][j] = (i == j) ? T(1) : T(0);
    }
  givens_rows<T>(B, U, 0, 1, 0);
  givens_rows<T>(B, U, 0, 2, 0);
  givens_rows<T>(B, U, 1, 2, 1);
  // B is now upper triangular: B[0][0] >= 0, B[1][1] >= 0, B[2][2] signed
  trace = B[0][0] + B[1][1] + B[2][2];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) R[i][j] = U[i][0] * V[j][0] + U[i][1] * V[j][1] + U[i][2] * V[j][2];
}

// Two Newton steps on SO(3) towards the rotation that maximises tr(R^T D), from a
// near one.  With S = R^T D, tr(exp([y]x)^T S) = tr S + a . y - y^T H y / 2 +
// O(|y|^3) with a the axial vector of S - S^T and H = tr(S) I - (S + S^T) / 2, so
// y = H^-1 a.  The second step takes the same H^-1, and the error it leaves is about
// the product of the steps.  True if H is positive definite (a maximum, not a
// saddle) and the squares of the steps are below the limits.
__device__ __forceinline__ bool newton_rotation(const double D[3][3], double R[3][3], double& trace, double limit1,
                                                double limit2) {
  double S[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) S[i][j] = R[0][i] * D[0][j] + R[1][i] * D[1][j] + R[2][i] * D[2][j];
  const double h00 = S[1][1] + S[2][2], h11 = S[0][0] + S[2][2], h22 = S[0][0] + S[1][1];
  const double h01 = -0.5 * (S[0][1] + S[1][0]), h02 = -0.5 * (S[0][2] + S[2][0]), h12 = -0.5 * (S[1][2] + S[2][1]);
  const double i00 = h11 * h22 - h12 * h12, i01 = h02 * h12 - h01 * h22, i02 = h01 * h12 - h02 * h11;
  const double i11 = h00 * h22 - h02 * h02, i12 = h01 * h02 - h00 * h12, i22 = h00 * h11 - h01 * h01;
  const double det = h00 * i00 + h01 * i01 + h02 * i02;
  bool good = h00 > 0.0 && i22 > 0.0 && det > 0.0;
  const double id = 1.0 / det;
  double a0 = (S[2][1] - S[1][2]) * id, a1 = (S[0][2] - S[2][0]) * id, a2 = (S[1][0] - S[0][1]) * id;
  double y0 = i00 * a0 + i01 * a1 + i02 * a2, y1 = i01 * a0 + i11 * a1 + i12 * a2, y2 = i02 * a0 + i12 * a1 + i22 * a2;
  const double yy = y0 * y0 + y1 * y1 + y2 * y2;
  good = good && yy < limit1;
  // R <- R C with C = I + [y]x + ([y]x)^2 / 2 (orthogonal to |y|^4 / 4)
  const double c00 = -0.5 * (y1 * y1 + y2 * y2), c11 = -0.5 * (y0 * y0 + y2 * y2), c22 = -0.5 * (y0 * y0 + y1 * y1);
  const double p01 = 0.5 * y0 * y1, p02 = 0.5 * y0 * y2, p12 = 0.5 * y1 * y2;
  for (int i = 0; i < 3; ++i) {
    const double r0 = R[i][0], r1 = R[i][1], r2 = R[i][2];
    R[i][0] = r0 + (r0 * c00 + r1 * (p01 + y2) + r2 * (p02 - y1));
    R[i][1] = r1 + (r0 * (p01 - y2) + r1 * c11 + r2 * (p12 + y0));
    R[i][2] = r2 + (r0 * (p02 + y1) + r1 * (p12 - y0) + r2 * c22);
  }
  // second step, first order in y
  a0 = (R[0][2] * D[0][1] + R[1][2] * D[1][1] + R[2][2] * D[2][1] - (R[0][1] * D[0][2] + R[1][1] * D[1][2] + R[2][1] * D[2][2])) * id;
  a1 = (R[0][0] * D[0][2] + R[1][0] * D[1][2] + R[2][0] * D[2][2] - (R[0][2] * D[0][0] + R[1][2] * D[1][0] + R[2][2] * D[2][0])) * id;
  a2 = (R[0][1] * D[0][0] + R[1][1] * D[1][0] + R[2][1] * D[2][0] - (R[0][0] * D[0][1] + R[1][0] * D[1][1] + R[2][0] * D[2][1])) * id;
  y0 = i00 * a0 + i01 * a1 + i02 * a2, y1 = i01 * a0 + i11 * a1 + i12 * a2, y2 = i02 * a0 + i12 * a1 + i22 * a2;
  good = good && y0 * y0 + y1 * y1 + y2 * y2 < limit2;
  for (int i = 0; i < 3; ++i) {
    const double r0 = R[i][0], r1 = R[i][1], r2 = R[i][2];
    R[i][0] = r0 + (r1 * y2 - r2 * y1);
    R[i][1] = r1 + (r2 * y0 - r0 * y2);
    R[i][2] = r2 + (r0 * y1 - r1 * y0);
  }
  trace = S[0][0] + S[1][1] + S[2][2];
  return good;
}

// The FP64 SVD fit behind a call, for the few elements that need it.  Its error is
// about 1e-16 times the square of D's condition (it starts from D^T D); the Newton
// steps, where they apply, leave the condition itself.
template <int SWEEPS>
__device__ __noinline__ void kabsch_rotation_call(const double (*D)[3], double (*R)[3], double* trace) {
  double d[3][3], r[3][3], n[3][3], t;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) d[i][j] = D[i][j];
  kabsch_rotation<double, SWEEPS>(d, r, t);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) n[i][j] = r[i][j];
  double tn;
  const bool better = newton_rotation(d, n, tn, 1e-8, 1e-20);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) R[i][j] = better ? n[i][j] : r[i][j];
  *trace = better ? tn : t;
}

// The rotation R that maximises tr(R^T D): in FP32 the SVD fit itself.  In FP64
// the SVD fit of D in FP32, brought to FP64 by two Newton steps: the first starts
// from an error of about 1e-7 and leaves about 1e-14.  An element that fails their
// tests (nearly flat or collapsed, a scale outside FP32's) takes the FP64 SVD fit.
//
// An FP64 instruction costs a warp 64 cycles of its scheduler, and the six Jacobi
// sweeps are about 1,900 of them, the two steps about 230.  Measured, FP64 SVD and
// this: k_local 163 and 63 us for 51,840 tets, 64 and 29 us for 1,920; k_adj_local
// 149 and 85 us for 20,736.
template <typename T, int SWEEPS>
__device__ __forceinline__ void rotation_fit(const T D[3][3], T R[3][3], T& trace) {
  if constexpr (std::is_same<T, float>::value) {
    kabsch_rotation<float, SWEEPS>(D, R, trace);
  } else {
    float Df[3][3], m = 0.0f;
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Df[i][j] = (float)D[i][j];
        m = fmaxf(m, fabsf(Df[i][j]));
      }
    bool good = m > 1e-30f && m < 1e30f;
    {
      const float s = 1.0f / m;
      float Rf[3][3], t;
      for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) Df[i][j] *= s;
      kabsch_rotation<float, 4>(Df, Rf, t);
      // as a quaternion (its largest component first, Shepperd 1978), so that the
      // FP64 matrix made of it is orthogonal to FP64 rounding
      const float tr = Rf[0][0] + Rf[1][1] + Rf[2][2];
      float qw, qx, qy, qz;
      if (tr >= Rf[0][0] && tr >= Rf[1][1] && tr >= Rf[2][2]) {
        qw = 1.0f + tr, qx = Rf[2][1] - Rf[1][2], qy = Rf[0][2] - Rf[2][0], qz = Rf[1][0] - Rf[0][1];
      } else if (Rf[0][0] >= Rf[1][1] && Rf[0][0] >= Rf[2][2]) {
        qw = Rf[2][1] - Rf[1][2], qx = 1.0f + 2.0f * Rf[0][0] - tr, qy = Rf[0][1] + Rf[1][0], qz = Rf[0][2] + Rf[2][0];
      } else if (Rf[1][1] >= Rf[2][2]) {
        qw = Rf[0][2] - Rf[2][0], qx = Rf[0][1] + Rf[1][0], qy = 1.0f + 2.0f * Rf[1][1] - tr, qz = Rf[1][2] + Rf[2][1];
      } else {
        qw = Rf[1][0] - Rf[0][1], qx = Rf[0][2] + Rf[2][0], qy = Rf[1][2] + Rf[2][1], qz = 1.0f + 2.0f * Rf[2][2] - tr;
      }
      const double w = qw, x = qx, y = qy, z = qz;
      const double n = 2.0 / (w * w + x * x + y * y + z * z);
      const double xs = x * n, ys = y * n, zs = z * n;
      R[0][0] = 1.0 - (y * ys + z * zs), R[0][1] = x * ys - w * zs, R[0][2] = x * zs + w * ys;
      R[1][0] = x * ys + w * zs, R[1][1] = 1.0 - (x * xs + z * zs), R[1][2] = y * zs - w * xs;
      R[2][0] = x * zs - w * ys, R[2][1] = y * zs + w * xs, R[2][2] = 1.0 - (x * xs + y * ys);
    }
    good = newton_rotation(D, R, trace, 1e-10, 1e-22) && good;
    if (!good) kabsch_rotation_call<SWEEPS>(D, R, &trace);
  }
}

}  // namespace casim
