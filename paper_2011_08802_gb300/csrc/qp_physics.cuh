// Quadrature-point physics of the multivariant finite-strain phase-field
// model: local energy density, its gradient and its exact 15x15 Hessian with
// respect to z = (F_iJ row-major, eta_1..eta_6).
//
// Model (Sec. 2.1-2.3, Sec. 3.1): eta_0 = 1 - sum eta_k; F^t = sum_i eta_i U_i
// (Eq. LinMix); F^e = F (F^t)^-1, C^e = F^eT F^e, H^e = 1/2 log C^e and
// F_el = 1/2 det(F^t) H^e . L(eta) H^e with L = sum_i eta_i L_i
// (Eq. elasticEn); chemical sum eta_i F_i^0; local part of the double
// obstacle sum_{i<j} 4 gamma_ij/(pi ell_ij) eta_i eta_j (Eq. IntEnergy);
// backward-Euler dissipation sum (eta_i - eta_i,n)^2/(2 m_i tau) (Sec. 2.3);
// penalty sum 1/2 eps <eta_i>_-^2 (Eq. PenPot). The gradient part of the
// interface energy is a constant quadratic form handled by the element
// kernels.
//
// Derivatives. With A = (F^t)^-1, M = F^e = F A and E = C^e = M^T M, the elastic
// energy is J_t g(M), g = 1/2 h:L:h, h = 1/2 log E, J_t = det F^t. Every
// direction moves M along a rank-one matrix l A_c^T (A_c: column c of A): F_pc
// along l = e_p, an entry (i, c) of F^t along l = -M e_i, so with q = Q^T M^T l
// and a_c = Q^T A_c (Q: eigenvectors of E) the rotated change of E is
// a_c q^T + q a_c^T. The second derivative along two such directions is
// q^T R_cc' q' with six 3x3 matrices R_cc' per Gauss point (the spectral second
// derivative of g contracted with a_c and a_c', plus the stress term
// (A 2S A)_cc' diag(1/lambda), because l . l' = q^T Lambda^-1 q'). The
// order parameters enter only through the six entries of the symmetric F^t:
// rows and columns of the Hessian are formed for those six entries and turned
// into the eta_hat_k by the constant matrix of dU_k = U_k - U_0.
// The point physics is bound by the FP64 pipe (about 2 multiply-adds per clock
// and SM), so what counts is the number of FP64 instructions; FP32 ones are
// nearly free. The eigenvectors start from FP32 Jacobi rotations of the
// deviator of E and two FP64 corrections by small rotations follow
// (quadratic convergence from 1e-7); the rotation is held as a quaternion, so it
// is orthonormal to rounding without a Gram-Schmidt pass. The divided
// differences of log use the series of 2 atanh((a-b)/(a+b)) when a and b are
// close, which needs one reciprocal and no logarithm. Measured against the form
// with one direction per unknown, a Jacobi eigensolve in FP64 and a 120-entry
// array of the Hessian: linearisation with residual of 80x72x56 elements 37.8 ->
// 23.6 ms (stack per thread 5.9 -> 1.6 KB), residual of 97x65x50 10.1 -> 7.0 ms
// (5.4 ms with the nodal gradient energy and shared differences in the gather).
//
// The matrix logarithm's derivatives are the Daleckii-Krein formulas: in the
// eigenbasis Dlog[X]_ab = f1(l_a,l_b) X_ab and
// D2log[X,Y]_ab = sum_c f2(l_a,l_c,l_b) (X_ac Y_cb + Y_ac X_cb), with f1, f2
// the first and second divided differences of log, exact for repeated
// eigenvalues because no difference quotient of nearly equal values is formed.
//
// Pade modes (Sec. 2.4, Eqs. pade11, pade22, pade33). The paper's (m,m)
// approximant of H^e is the primary matrix function h = 1/2 r_m(C^e), r_m the
// [m/m] Pade approximant of log about 1. The m-point Gauss-Legendre rule on
// log x = int_0^1 (x - 1)/(1 + s (x - 1)) ds is that approximant (Dieci,
// Morini and Papini, 1996): r_m(x) = sum_k w_k (x - 1) p_k(x)^-1 with
// p_k(x) = 1 + s_k (x - 1). The same spectral route then applies with
// divided differences that are products of the reciprocals 1/p_k, free of
// cancellation for any eigenvalue spread:
// r_m[a,b] = sum_k w_k / (p_k(a) p_k(b)),
// r_m[a,b,c] = -sum_k w_k s_k / (p_k(a) p_k(b) p_k(c)).
#pragma once

#include <type_traits>

#include "fixed_point.cuh"

#ifdef __CUDACC__
#define PFM_HD __host__ __device__ __forceinline__
#define PFM_HD_BIG __host__ __device__
#define PFM_HD_COLD static __host__ __device__ __noinline__
#else
#define PFM_HD_BIG inline
#define PFM_HD_COLD static inline
#include <cmath>
#define PFM_HD inline
using std::sqrt;
using std::log;
using std::log1p;
using std::fabs;
#endif

namespace pfm {

#ifdef __CUDACC__
// keep the C math functions visible next to the double-float overloads below
using ::fabs;
using ::log;
using ::log1p;
using ::sqrt;

// ---------------------------------------------------------------------------
// Double-float number hi + lo (two FP32 values, |lo| <= ulp(hi)/2): about 48
// significant bits from FP32 adds, multiplies and fused multiply-adds only
// (Dekker 1971; Knuth's TwoSum), so the point physics can run on the FP32
// pipes. Division, square root and the logarithms go through FP64 (a handful
// per Gauss point). The _rn intrinsics keep the compiler from contracting or
// reassociating the error-free transformations.
struct df64 {
  float hi, lo;
  df64() = default;
  __device__ __forceinline__ df64(double x) {
    hi = __double2float_rn(x);
    lo = __double2float_rn(x - double(hi));
  }
  __device__ __forceinline__ explicit operator double() const { return double(hi) + double(lo); }
  __device__ __forceinline__ static df64 make(float h, float l) {
    df64 r;
    r.hi = h;
    r.lo = l;
    return r;
  }
};

__device__ __forceinline__ df64 df64_fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return df64::make(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ df64 operator+(df64 a, df64 b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  return df64_fast_two_sum(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ df64 operator-(df64 a) { return df64::make(-a.hi, -a.lo); }
__device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }
__device__ __forceinline__ df64 operator*(df64 a, df64 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df64_fast_two_sum(p, e);
}
__device__ __forceinline__ df64 operator/(df64 a, df64 b) { return df64(double(a) / double(b)); }
__device__ __forceinline__ df64& operator+=(df64& a, df64 b) { return a = a + b; }
__device__ __forceinline__ df64& operator-=(df64& a, df64 b) { return a = a - b; }
__device__ __forceinline__ df64& operator*=(df64& a, df64 b) { return a = a * b; }
__device__ __forceinline__ df64& operator/=(df64& a, df64 b) { return a = a / b; }
__device__ __forceinline__ bool operator<(df64 a, df64 b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
__device__ __forceinline__ bool operator>(df64 a, df64 b) { return b < a; }
__device__ __forceinline__ bool operator<=(df64 a, df64 b) { return !(b < a); }
__device__ __forceinline__ bool operator>=(df64 a, df64 b) { return !(a < b); }
__device__ __forceinline__ bool operator==(df64 a, df64 b) { return a.hi == b.hi && a.lo == b.lo; }
__device__ __forceinline__ bool operator!=(df64 a, df64 b) { return !(a == b); }
__device__ __forceinline__ df64 fabs(df64 a) { return a.hi < 0.f ? -a : a; }
__device__ __forceinline__ df64 sqrt(df64 a) { return df64(::sqrt(double(a))); }
__device__ __forceinline__ df64 log(df64 a) { return df64(::log(double(a))); }
__device__ __forceinline__ df64 log1p(df64 a) { return df64(::log1p(double(a))); }
__device__ __forceinline__ df64 shx(df64 v, int m) {
  return df64::make(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
}
#endif

// Number of martensite variants N, fixed at compile time: 6 for the CuAlNi
// data of Sec. 5.1 (the default build), 12 for a NiTi-type monoclinic set
// (15 unknowns per node, the footnote of Sec. 5.4); the library is built once
// per value (libpfm.so, libpfm_nv12.so).
#ifndef PFM_NV
#define PFM_NV 6
#endif
constexpr int NV = PFM_NV;
constexpr int NPH = NV + 1;           // phases: austenite + N variants
constexpr int NZ = 9 + NV;            // local unknowns at a point: F (9) + eta_hat (N)
constexpr int NH = NZ * (NZ + 1) / 2; // packed upper triangle of the NZ x NZ Hessian (120 for N = 6)
// entries stored per Gauss point: NH rounded up to a multiple of 8, so that
// 16-byte vectors of binary16, FP32 or FP64 entries tile it (120 and 232)
constexpr int NHP = (NH + 7) / 8 * 8;

// Physical parameters, passed by value to kernels (constant bank).
struct DevParams {
  double U0[6];             // transformation stretch U_0 (Voigt slots 00, 11, 22, 12, 02, 01)
  double dU[NV][6];         // U_k - U_0, the derivative of F^t with respect to eta_hat_k
  int dU1[NV][6], dU0[NV][6], dUe;  // and as limbs relative to 2^dUe (fixed_point.cuh; FX_NONE: not available)
  double Lv[NPH][6][6];     // stiffness L_i in Voigt form (engineering shear)
  double inv_mtau[NPH];     // 1 / (m_i tau)
  // chemical and obstacle energy in the condensed unknowns (eta_0 = 1 - sum eta_hat):
  // W0 + sum_k lin_k eta_hat_k + 1/2 sum_kl Cc_kl eta_hat_k eta_hat_l
  double W0, lin[NV], Cc[NV][NV];
  double G[NV][NV];         // gradient-energy matrix in eta_hat (per direction)
  double eps_eta;           // penalty parameter
  int same_L;               // 1 when every phase has the same stiffness (then L(eta) = L, as sum eta = 1)
  int cubic;                // 1 when that stiffness is cubic in the frame of the data:
  double cub_lambda, cub_mu, cub_delta;  // L = lambda I x I + 2 mu I_sym + delta sum_n e_n^4
  int hencky;               // 0: exact log; m = 1, 2, 3: Pade (m,m) (Gauss-Legendre form below)
  double pade_s[3], pade_w[3];  // m-point Gauss-Legendre nodes and weights on [0, 1]
};

// Packed index of (r, c), r <= c, in the row-major upper triangle.
PFM_HD int hidx(int r, int c) { return r * NZ - (r * (r - 1)) / 2 + (c - r); }

template <typename T> struct Tol;
template <> struct Tol<double> {
  static constexpr float f2_gap = 2e-2f;     // relative spread up to which f2 of three values uses its series
  static constexpr double jacobi_off = 1e-17;
};
#ifdef __CUDACC__
template <> struct Tol<df64> {
  static constexpr float f2_gap = 2e-2f;
  static constexpr double jacobi_off = 1e-14;  // the double-float resolution
};
#endif
template <> struct Tol<float> {
  static constexpr float f2_gap = 1e-1f;
  static constexpr float jacobi_off = 1e-8f;
};

template <typename T> PFM_HD float to_f32(T a) { return float(a); }
#ifdef __CUDACC__
template <> PFM_HD float to_f32<df64>(df64 a) { return a.hi; }
#endif

// ---------------------------------------------------------------------------
// 3x3 helpers (full storage)

template <typename T>
PFM_HD void mm3(const T a[3][3], const T b[3][3], T c[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) c[i][k] = a[i][0] * b[0][k] + a[i][1] * b[1][k] + a[i][2] * b[2][k];
}

// c = a^T b
template <typename T>
PFM_HD void mtm3(const T a[3][3], const T b[3][3], T c[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) c[i][k] = a[0][i] * b[0][k] + a[1][i] * b[1][k] + a[2][i] * b[2][k];
}

// c = Q^T a Q (rotate a symmetric matrix into the basis of Q's columns)
template <typename T>
PFM_HD void rot_in(const T Q[3][3], const T a[3][3], T c[3][3]) {
  T t[3][3];
  mm3(a, Q, t);
  mtm3(Q, t, c);
}

// Inverse (packed) and determinant of a packed symmetric 3x3 matrix.
template <typename T>
PFM_HD T inv_sym6(const T a[6], T r[6]) {
  const T c00 = a[1] * a[2] - a[3] * a[3];
  const T c01 = a[3] * a[4] - a[5] * a[2];
  const T c02 = a[5] * a[3] - a[1] * a[4];
  const T det = a[0] * c00 + a[5] * c01 + a[4] * c02;
  const T id = T(1) / det;
  r[0] = c00 * id;
  r[5] = c01 * id;
  r[4] = c02 * id;
  r[1] = (a[0] * a[2] - a[4] * a[4]) * id;
  r[3] = (a[5] * a[4] - a[0] * a[3]) * id;
  r[2] = (a[0] * a[1] - a[5] * a[5]) * id;
  return det;
}

// Packed symmetric 3x3 storage (00, 11, 22, 12, 02, 01), the Voigt order.
PFM_HD int sym_i(int v) { return v < 3 ? v : (v == 3 ? 1 : 0); }
PFM_HD int sym_j(int v) { return v < 3 ? v : (v == 5 ? 1 : 2); }
template <typename T>
PFM_HD T symget(const T* X, int a, int b) {
  if (a == b) return X[a];
  const int s = a + b;  // (1,2) -> 3, (0,2) -> 2, (0,1) -> 1
  return X[s == 3 ? 3 : (s == 2 ? 4 : 5)];
}
// Voigt slot (00, 11, 22, 12, 02, 01) of the symmetric pair (a, c).
PFM_HD int voigt_slot(int a, int c) { return a == c ? a : 6 - a - c; }

// ---------------------------------------------------------------------------
// Symmetric 3x3 eigen-decomposition by cyclic Jacobi rotations:
// a = Q diag(lam) Q^T, Q orthonormal (columns are eigenvectors).

template <typename T>
PFM_HD void jacobi_eig3(T a[3][3], T lam[3], T Q[3][3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) Q[i][j] = (i == j) ? T(1) : T(0);
  for (int sweep = 0; sweep < 16; ++sweep) {
    T off = fabs(a[0][1]) + fabs(a[0][2]) + fabs(a[1][2]);
    T dia = fabs(a[0][0]) + fabs(a[1][1]) + fabs(a[2][2]);
    if (off <= Tol<T>::jacobi_off * dia) break;
#pragma unroll
    for (int pq = 0; pq < 3; ++pq) {
      const int p = (pq == 2) ? 1 : 0;
      const int q = (pq == 0) ? 1 : 2;
      const int r = 3 - p - q;
      T apq = a[p][q];
      if (fabs(apq) <= Tol<T>::jacobi_off * (fabs(a[p][p]) + fabs(a[q][q]))) {
        a[p][q] = a[q][p] = T(0);
        continue;
      }
      // rotation angle phi with cot(2 phi) = theta zeroes a_pq; t = tan(phi)
      T theta = (a[q][q] - a[p][p]) / (T(2) * apq);
      T t = T(1) / (fabs(theta) + sqrt(theta * theta + T(1)));
      if (theta < T(0)) t = -t;
      T c = T(1) / sqrt(t * t + T(1));
      T s = t * c;
      T tau = s / (T(1) + c);
      a[p][p] -= t * apq;
      a[q][q] += t * apq;
      a[p][q] = a[q][p] = T(0);
      T arp = a[r][p], arq = a[r][q];
      a[r][p] = a[p][r] = arp - s * (arq + tau * arp);
      a[r][q] = a[q][r] = arq + s * (arp - tau * arq);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        T qkp = Q[k][p], qkq = Q[k][q];
        Q[k][p] = qkp - s * (qkq + tau * qkp);
        Q[k][q] = qkq + s * (qkp - tau * qkq);
      }
    }
  }
  lam[0] = a[0][0]; lam[1] = a[1][1]; lam[2] = a[2][2];
}


// Rotation matrix of a quaternion (w, x, y, z) of any length.
template <typename T>
PFM_HD void quat_rot(const T q[4], T R[3][3]) {
  const T s = T(2) / (q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
  const T xs = q[1] * s, ys = q[2] * s, zs = q[3] * s;
  const T wx = q[0] * xs, wy = q[0] * ys, wz = q[0] * zs;
  const T xx = q[1] * xs, xy = q[1] * ys, xz = q[1] * zs;
  const T yy = q[2] * ys, yz = q[2] * zs, zz = q[3] * zs;
  R[0][0] = T(1) - (yy + zz);
  R[0][1] = xy - wz;
  R[0][2] = xz + wy;
  R[1][0] = xy + wz;
  R[1][1] = T(1) - (xx + zz);
  R[1][2] = yz - wx;
  R[2][0] = xz - wy;
  R[2][1] = yz + wx;
  R[2][2] = T(1) - (xx + yy);
}

// q <- q (1, x, y, z) (Hamilton product): R(q) <- R(q) R(1, x, y, z)
template <typename T>
PFM_HD void quat_mul_unit(T q[4], T x, T y, T z) {
  const T w = q[0], a = q[1], b = q[2], c = q[3];
  q[0] = w - (a * x + b * y + c * z);
  q[1] = a + (w * x + b * z - c * y);
  q[2] = b + (w * y + c * x - a * z);
  q[3] = c + (w * z + a * y - b * x);
}

// Cyclic Jacobi on the packed symmetric matrix a (FP32): on return a is
// diagonal to rounding and q the quaternion of the rotation Q with
// a_in = Q diag(a) Q^T. A rotation by the angle phi in the plane (p, r) that
// keeps axis n multiplies the quaternion by (1, -+ tan(phi/2) e_n).
PFM_HD void jacobi_quat(float a[6], float q[4]) {
  q[0] = 1.f;
  q[1] = q[2] = q[3] = 0.f;
  for (int sweep = 0; sweep < 16; ++sweep) {
    const float off = fabsf(a[3]) + fabsf(a[4]) + fabsf(a[5]);
    const float dia = fabsf(a[0]) + fabsf(a[1]) + fabsf(a[2]);
    if (off <= Tol<float>::jacobi_off * dia) break;
#pragma unroll
    for (int n = 2; n >= 0; --n) {  // planes (0,1), (0,2), (1,2)
      const int p = n == 0 ? 1 : 0, r = n == 2 ? 1 : 2;
      const float apr = a[3 + n];
      if (fabsf(apr) <= Tol<float>::jacobi_off * (fabsf(a[p]) + fabsf(a[r]))) {
        a[3 + n] = 0.f;
        continue;
      }
      const float theta = (a[r] - a[p]) / (2.f * apr);
      float t = 1.f / (fabsf(theta) + sqrtf(theta * theta + 1.f));
      if (theta < 0.f) t = -t;
      const float c = 1.f / sqrtf(t * t + 1.f);
      const float sn = t * c;
      const float tau = sn / (1.f + c);
      a[p] -= t * apr;
      a[r] += t * apr;
      a[3 + n] = 0.f;
      // the entries that couple axis n to p and r are the slots 3 + r and 3 + p
      const float anp = a[3 + r], anr = a[3 + p];
      a[3 + r] = anp - sn * (anr + tau * anp);
      a[3 + p] = anr + sn * (anp - tau * anr);
      const float v = n == 1 ? tau : -tau;
      const float w = q[0], x = q[1], y = q[2], z = q[3];
      if (n == 0) {
        q[0] = w - x * v; q[1] = x + w * v; q[2] = y + z * v; q[3] = z - y * v;
      } else if (n == 1) {
        q[0] = w - y * v; q[1] = x - z * v; q[2] = y + w * v; q[3] = z + x * v;
      } else {
        q[0] = w - z * v; q[1] = x + y * v; q[2] = y - x * v; q[3] = z + w * v;
      }
    }
  }
}

// b = R^T X R (packed)
template <typename T>
PFM_HD void rot_sym6(const T R[3][3], const T X[6], T b[6]) {
  T t[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      t[i][j] = symget(X, i, 0) * R[0][j] + symget(X, i, 1) * R[1][j] + symget(X, i, 2) * R[2][j];
#pragma unroll
  for (int v = 0; v < 6; ++v) {
    const int i = sym_i(v), j = sym_j(v);
    b[v] = R[0][i] * t[0][j] + R[1][i] * t[1][j] + R[2][i] * t[2][j];
  }
}

// Where FP32 angles are not good enough: Jacobi rotations with exact angles on
// R^T A R (on A, R = I, where that is not finite), R <- the eigenvectors of A. Rare,
// and out of line so that it takes no registers from the common path.
PFM_HD_COLD void eig_finish_jacobi(const double A[6], double lam[3], double R[3][3]) {
  double b[6];
  rot_sym6(R, A, b);
  if (!(fabs(b[0]) + fabs(b[1]) + fabs(b[2]) + fabs(b[3]) + fabs(b[4]) + fabs(b[5]) < HUGE_VAL)) {
    for (int v = 0; v < 6; ++v) b[v] = A[v];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) R[i][j] = i == j ? 1.0 : 0.0;
  }
  double a[3][3] = {{b[0], b[5], b[4]}, {b[5], b[1], b[3]}, {b[4], b[3], b[2]}};
  double Q1[3][3], Q[3][3];
  jacobi_eig3(a, lam, Q1);
  mm3(R, Q1, Q);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) R[i][j] = Q[i][j];
}

// Eigen-decomposition E = Q diag(m + d) Q^T of the packed symmetric matrix E.
// Usually m is the mean of E's diagonal and d belongs to the deviator, so that neither
// the distances of the eigenvalues from 1, (m - 1) + d, nor their differences carry
// the rounding of numbers near 1; the eigenvalues are m + d, not 1 + ((m - 1) + d), so
// that small ones (strong compression) do not carry it either. Where the deviator is
// large against the smallest eigenvalue (more than twice that: stretches apart by a
// factor of about 2 or more) the small ones would carry the deviator's rounding: then
// E itself is rotated and m is 0.
PFM_HD bool eig_wide(const float a[3], float m) {
  const float dev = 0.5f * (fabsf(a[0]) + fabsf(a[1]) + fabsf(a[2]));  // NaN and infinite numbers count as wide
  return !(dev <= 2.f * fminf(m + fminf(a[0], fminf(a[1], a[2])), 1e37f));
}
PFM_HD void eig_sym6(const float E[6], float& m, float x[3], float Q[3][3]) {
  m = (E[0] + E[1] + E[2]) * (1.f / 3.f);
  float a[6] = {E[0] - m, E[1] - m, E[2] - m, E[3], E[4], E[5]}, q[4];
  jacobi_quat(a, q);
  if (eig_wide(a, m)) {
    m = 0.f;
#pragma unroll
    for (int v = 0; v < 6; ++v) a[v] = E[v];
    jacobi_quat(a, q);
  }
  quat_rot(q, Q);
#pragma unroll
  for (int i = 0; i < 3; ++i) x[i] = a[i];
}
// FP64: eigenvectors from FP32 Jacobi, then twice b = R^T X R and the
// simultaneous small rotation tan(phi/2) = b_pr / (2 (b_rr - b_pp)) in the three
// planes, its angles in FP32 (the error left after the first correction is the
// square of the angles, about 1e-13 of the deviator, and nothing after the
// second). Angles above 1e-3 in the first correction mean nearly equal
// eigenvalues, where Jacobi with exact angles takes over, as it does for wide ones.
PFM_HD void eig_sym6(const double E[6], double& m, double x[3], double Q[3][3]) {
  m = (E[0] + E[1] + E[2]) * (1.0 / 3.0);
  const double X[6] = {E[0] - m, E[1] - m, E[2] - m, E[3], E[4], E[5]};
  float a[6], qf[4];
#pragma unroll
  for (int v = 0; v < 6; ++v) a[v] = float(X[v]);
  jacobi_quat(a, qf);
  const bool wide = eig_wide(a, float(m));
  double q[4] = {double(qf[0]), double(qf[1]), double(qf[2]), double(qf[3])};
  double b[6];
#pragma unroll
  for (int pass = 0; pass < 2; ++pass) {
    quat_rot(q, Q);
    rot_sym6(Q, X, b);
    float tau[3];  // tau[n]: the plane that keeps axis n
    const float num[3] = {float(b[3]), float(b[4]), float(b[5])};
    const float den[3] = {float(b[2] - b[1]), float(b[2] - b[0]), float(b[1] - b[0])};
    bool rough = wide;
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      tau[n] = num[n] == 0.f ? 0.f : 0.5f * num[n] / den[n];
      rough = rough || !(fabsf(tau[n]) <= 1e-3f);
    }
    if (pass == 0 && rough) {
      double A[6];
#pragma unroll
      for (int v = 0; v < 6; ++v) A[v] = wide ? E[v] : X[v];
      if (wide) m = 0.0;
      eig_finish_jacobi(A, x, Q);
      return;
    }
    quat_mul_unit(q, double(-tau[0]), double(tau[1]), double(-tau[2]));
  }
  quat_rot(q, Q);
#pragma unroll
  for (int i = 0; i < 3; ++i) x[i] = b[i];
}

#ifdef __CUDACC__
// Double-float version of the FP64 eigen-decomposition: FP32 Jacobi seed,
// re-orthonormalisation and the finishing sweeps in double-float.
__device__ __forceinline__ void eig_sym6(const df64 E[6], df64& m, df64 x[3], df64 Q[3][3]) {
  df64 a[3][3] = {{E[0], E[5], E[4]}, {E[5], E[1], E[3]}, {E[4], E[3], E[2]}};
  float af[3][3], lf[3], Qf[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) af[i][j] = a[i][j].hi;
  jacobi_eig3(af, lf, Qf);
  df64 Q0[3][3], b[3][3], Q1[3][3];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) Q0[i][j] = df64(double(Qf[i][j]));
  for (int c = 0; c < 3; ++c) {
    for (int pc = 0; pc < c; ++pc) {
      df64 d = Q0[0][c] * Q0[0][pc] + Q0[1][c] * Q0[1][pc] + Q0[2][c] * Q0[2][pc];
      for (int i = 0; i < 3; ++i) Q0[i][c] -= d * Q0[i][pc];
    }
    df64 inrm = df64(1.0 / ::sqrt(double(Q0[0][c] * Q0[0][c] + Q0[1][c] * Q0[1][c] + Q0[2][c] * Q0[2][c])));
    for (int i = 0; i < 3; ++i) Q0[i][c] *= inrm;
  }
  rot_in(Q0, a, b);
  jacobi_eig3(b, x, Q1);
  m = df64(0.0);  // the rotated matrix is E itself
  mm3(Q0, Q1, Q);
}
#endif

// First divided difference f1 = (log a - log b)/(a - b) of log and, with PAIR,
// the second ones f2(a,a,b) and f2(a,b,b) (d = a - b, ia = 1/a, ib = 1/b). With
// z = (a - b)/(a + b): f1 = 2/(a+b) sum_n z^2n/(2n+1) and
// f2(a,a,b), f2(a,b,b) = -1/(2ab) +- 2/(a+b)^2 sum_{n>=1} 2n/(2n+1) z^(2n-1)
// (their mean is (1/a - 1/b)/(2(a-b)); the odd part of the series is the rest).
// Seven terms give 1e-18 for |z| <= 1/16, that is a/b within 13 per cent;
// wider pairs take the quotients, which lose nothing there.
template <bool PAIR, typename T>
PFM_HD T dd_log(T a, T b, T d, T ia, T ib, T* faab, T* fabb) {
  const T r = T(1) / (a + b);
  const T z = d * r;
  if (fabsf(to_f32(z)) <= 0.0625f) {
    const T y = z * z;
    const T r2 = r + r;
    T p = T(1.0 / 13.0);
    p = p * y + T(1.0 / 11.0);
    p = p * y + T(1.0 / 9.0);
    p = p * y + T(1.0 / 7.0);
    p = p * y + T(1.0 / 5.0);
    p = p * y + T(1.0 / 3.0);
    p = p * y + T(1);
    if (PAIR) {
      T c = T(14.0 / 15.0);
      c = c * y + T(12.0 / 13.0);
      c = c * y + T(10.0 / 11.0);
      c = c * y + T(8.0 / 9.0);
      c = c * y + T(6.0 / 7.0);
      c = c * y + T(4.0 / 5.0);
      c = c * y + T(2.0 / 3.0);
      const T odd = r2 * r * z * c;
      const T even = T(-0.5) * ia * ib;
      *faab = even + odd;
      *fabb = even - odd;
    }
    return r2 * p;
  }
  const T f1 = d < T(0) ? log1p(-d / a) / -d : log1p(d / b) / d;
  if (PAIR) {
    const T id = T(1) / d;
    *faab = (ia - f1) * id;
    *fabb = (f1 - ib) * id;
  }
  return f1;
}

// Second divided difference of log at three values l = m0 + d from their first ones
// (f12 = f[l1,l2] and so on). Narrow spread (the whole spread below
// Tol::f2_gap of the mean m): f^(2+j)(m)/(2+j)! h_j(x - m) summed over j, for log
// (1/m^2) sum_j (-1)^(j+1) h_j(u)/(j+2), u = (x - m)/m, with the complete
// homogeneous symmetric polynomials h_j; the u sum to zero, so
// h_j = -e2 h_(j-2) + e3 h_(j-3). Otherwise the quotient over the largest gap.
template <typename T>
PFM_HD T dd2_log(T m0, const T x[3], T f12, T f02, T f01) {
  const float g01 = fabsf(to_f32(x[0] - x[1])), g02 = fabsf(to_f32(x[0] - x[2])), g12 = fabsf(to_f32(x[1] - x[2]));
  const float gap = fmaxf(g01, fmaxf(g02, g12));
  const T m = (x[0] + x[1] + x[2]) * T(1.0 / 3.0), ml = m0 + m;
  if (gap < Tol<T>::f2_gap * fminf(fabsf(to_f32(ml)), 1e38f)) {  // beyond FP32: the quotient
    const T im = T(1) / ml;
    const T u0 = (x[0] - m) * im, u1 = (x[1] - m) * im, u2 = (x[2] - m) * im;
    const T ne2 = u0 * u0 + u1 * (u0 + u1);  // -e2 = u0^2 + u0 u1 + u1^2
    const T e3 = u0 * u1 * u2;
    const T h4 = ne2 * ne2, h5 = T(2) * ne2 * e3;
    const T h6 = ne2 * h4 + e3 * e3, h7 = ne2 * h5 + e3 * h4, h8 = ne2 * h6 + e3 * h5;
    const T s = T(-0.5) - T(0.25) * ne2 + T(0.2) * e3 - T(1.0 / 6.0) * h4 + T(1.0 / 7.0) * h5 - T(0.125) * h6 +
                T(1.0 / 9.0) * h7 - T(0.1) * h8;
    return s * im * im;
  }
  if (g02 >= g01 && g02 >= g12) return (f01 - f12) / (x[0] - x[2]);
  if (g01 >= g12) return (f02 - f12) / (x[0] - x[1]);
  return (f01 - f02) / (x[1] - x[2]);
}

// Kinematics of one Gauss point: A = (F^t)^-1 and J_t, M = F^e = F A, the
// eigen-decomposition of C^e = M^T M = Q diag(lam) Q^T, the Hencky strain h at the
// eigenvalues (halved log, or the Pade approximant) and the divided differences
// of the function: f1 in the Voigt slots and, with F2, f2d[a] = f2(a,a,a),
// f2p[n] = {f2(p,p,r), f2(p,r,r)} for the pair (p, r), p < r, without n, and
// f2t = f2(0,1,2).
template <typename T>
struct Kinematics {
  T A[6], Jt, M[3][3], lam[3], Q[3][3], h[3], f1[6];
  T f2d[3], f2p[3][2], f2t;
};
template <bool F2, typename T>
PFM_HD void kinematics(const DevParams& P, const T Fin[9], const T eh[NV], Kinematics<T>& kin) {
  // transformation stretch F^t = U_0 + sum eta_hat_k dU_k, its inverse and determinant
  {
    T Ft[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      T s = eh[0] * T(P.dU[0][v]);
#pragma unroll
      for (int k = 1; k < NV; ++k) s += eh[k] * T(P.dU[k][v]);
      Ft[v] = T(P.U0[v]) + s;  // one rounding near 1
    }
    kin.Jt = inv_sym6(Ft, kin.A);
  }
  T (&M)[3][3] = kin.M;
  const T* A = kin.A;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      M[i][j] = Fin[3 * i] * symget(A, 0, j) + Fin[3 * i + 1] * symget(A, 1, j) + Fin[3 * i + 2] * symget(A, 2, j);
  T m, d[3];
  T (&lam)[3] = kin.lam;
  {
    T E[6];  // C^e = M^T M
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      const int i = sym_i(v), j = sym_j(v);
      E[v] = M[0][i] * M[0][j] + M[1][i] * M[1][j] + M[2][i] * M[2][j];
    }
    eig_sym6(E, m, d, kin.Q);
#pragma unroll
    for (int a = 0; a < 3; ++a) lam[a] = m + d[a];
  }
  T (&h)[3] = kin.h;
  T (&f1)[6] = kin.f1;
  T (&f2d)[3] = kin.f2d;
  T (&f2p)[3][2] = kin.f2p;
  T& f2t = kin.f2t;
  f2t = T(0);
  if (P.hencky == 0) {
#pragma unroll
    for (int a = 0; a < 3; ++a) f1[a] = T(1) / lam[a];
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const int p = n == 0 ? 1 : 0, r = n == 2 ? 1 : 2;
      f1[3 + n] = dd_log<F2>(lam[p], lam[r], d[p] - d[r], f1[p], f1[r], &f2p[n][0], &f2p[n][1]);
    }
    // log at one eigenvalue, the others through the divided differences
    const T x0 = (m - T(1)) + d[0];
    const T l0 = x0 * dd_log<false>(lam[0], T(1), x0, T(0), T(0), (T*)nullptr, (T*)nullptr);
    h[0] = T(0.5) * l0;
    h[1] = T(0.5) * (l0 + (d[1] - d[0]) * f1[5]);
    h[2] = T(0.5) * (l0 + (d[2] - d[0]) * f1[4]);
    if (F2) {
#pragma unroll
      for (int a = 0; a < 3; ++a) f2d[a] = T(-0.5) * f1[a] * f1[a];
      f2t = dd2_log(m, d, f1[3], f1[4], f1[5]);
    }
  } else {
    T x[3];  // lam - 1
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      x[a] = (m - T(1)) + d[a];
      h[a] = f2d[a] = f2p[a][0] = f2p[a][1] = T(0);
    }
#pragma unroll
    for (int v = 0; v < 6; ++v) f1[v] = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k < P.hencky) {
        const T sk = T(P.pade_s[k]), wk = T(P.pade_w[k]);
        T rp[3];  // 1 / p_k(lam_a)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          rp[a] = T(1) / (T(1) + sk * x[a]);
          h[a] += T(0.5) * wk * x[a] * rp[a];
        }
#pragma unroll
        for (int v = 0; v < 6; ++v) f1[v] += wk * rp[sym_i(v)] * rp[sym_j(v)];
        if (F2) {
          const T ws = wk * sk;
#pragma unroll
          for (int a = 0; a < 3; ++a) f2d[a] -= ws * rp[a] * rp[a] * rp[a];
#pragma unroll
          for (int n = 0; n < 3; ++n) {
            const int p = n == 0 ? 1 : 0, r = n == 2 ? 1 : 2;
            const T wpr = ws * rp[p] * rp[r];
            f2p[n][0] -= wpr * rp[p];
            f2p[n][1] -= wpr * rp[r];
          }
          f2t -= ws * rp[0] * rp[1] * rp[2];
        }
      }
    }
  }
}

// The order-parameter columns of the Hessian (stiffness shared by all phases) from
// FU and K in fixed point (fixed_point.cuh): FU dU_k and dU_p K dU_q were 666 of
// about 4100 FP64 operations per point with six variants (1548 with twelve) in a
// kernel bound by the FP64 pipe; as integer operations in rolled loops they run
// beside the rest (linearisation call on 80x72x56 elements 28.8 -> 25.5 ms).
// The loops stay rolled: with the whole chain from Mb unrolled in fixed point the
// kernel was bound by instruction fetch. False (nothing done) when a number is not
// finite or far from 1.
template <typename Emit>
PFM_HD bool eta_fx(const DevParams& P, const double (&FU)[9][6], const double (&K)[21], const double eh[NV], double eta0,
                   const Emit& emit) {
  auto hm6 = [](int I, int J) { return I <= J ? I * 6 - (I * (I - 1)) / 2 + (J - I) : J * 6 - (J * (J - 1)) / 2 + (I - J); };
  unsigned tF = 0, tK = 0;
  auto top = [](unsigned& t, double v) {
    const unsigned x = fx_top(v);
    t = x > t ? x : t;
  };
#pragma unroll
  for (int r = 0; r < 9; ++r)
#pragma unroll
    for (int v = 0; v < 6; ++v) top(tF, FU[r][v]);
#pragma unroll
  for (int v = 0; v < 21; ++v) top(tK, K[v]);
  bool ok = P.dUe != FX_NONE;
  const int EF = fx_block_exponent(tF, 400, ok), EK = fx_block_exponent(tK, 400, ok);
  if (!ok) return false;
  const int Ed = P.dUe;
  {
    Fx F[9][6];
#pragma unroll
    for (int r = 0; r < 9; ++r)
#pragma unroll
      for (int v = 0; v < 6; ++v) F[r][v] = fx_of(FU[r][v], EF);
#pragma unroll 1
    for (int k = 0; k < NV; ++k) {
      Fx d[6];
#pragma unroll
      for (int v = 0; v < 6; ++v) d[v] = Fx{P.dU1[k][v], P.dU0[k][v]};
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        int64_t s1 = 0, s0 = 0;
#pragma unroll
        for (int v = 0; v < 6; ++v) fx_mad(s1, s0, F[r][v], d[v]);
        emit(hidx(r, 9 + k), fx_value(s1, s0, 1027 + EF + Ed));
      }
    }
  }
  Fx Kx[21];
#pragma unroll
  for (int v = 0; v < 21; ++v) Kx[v] = fx_of(K[v], EK);
  const double dd0 = P.inv_mtau[0] + (eta0 < 0.0 ? P.eps_eta : 0.0);
#pragma unroll 1
  for (int q = 0; q < NV; ++q) {
    Fx t[6];
    int Et = EK + Ed;
    {
      int64_t u[6];
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        int64_t s1 = 0, s0 = 0;
#pragma unroll
        for (int x = 0; x < 6; ++x) fx_mad(s1, s0, Kx[hm6(v, x)], Fx{P.dU1[q][x], P.dU0[q][x]});
        u[v] = fx_sum(s1, s0);
      }
      Et += fx_normalise(u, t);
    }
#pragma unroll 1
    for (int p = 0; p <= q; ++p) {
      int64_t s1 = 0, s0 = 0;
#pragma unroll
      for (int v = 0; v < 6; ++v) fx_mad(s1, s0, t[v], Fx{P.dU1[p][v], P.dU0[p][v]});
      double loc = dd0 + P.Cc[p][q];
      if (p == q) loc += P.inv_mtau[p + 1] + (eh[p] < 0.0 ? P.eps_eta : 0.0);
      emit(hidx(9 + p, 9 + q), fx_value(s1, s0, 1027 + Et + Ed) + loc);
    }
  }
  return true;
}

// ---------------------------------------------------------------------------
// Local energy density with gradient and (optionally) packed Hessian.
//
// Fin: F row-major; eh, ehn: eta_1..eta_6 at t_{n+1} and t_n.
// Outputs: *W, g[15] = dW/dz; with Emit::want every entry of the packed Hessian
// d^2W/dz^2 is handed once to emit(index, value) when it is final (no order), so no
// array of the whole Hessian is kept.
template <typename T>
struct NoHess {
  static constexpr bool want = false;
  PFM_HD void operator()(int, T) const {}
};
template <typename T>
struct HessArray {
  static constexpr bool want = true;
  T* Hp;
  PFM_HD void operator()(int i, T v) const { Hp[i] = v; }
};

template <typename T, typename Emit>
PFM_HD void qp_point(const DevParams& P, const T Fin[9], const T eh[NV], const T ehn[NV], T* W, T g[NZ],
                     const Emit& emit) {
  Kinematics<T> kin;
  kinematics<Emit::want>(P, Fin, eh, kin);
  const T (&A)[6] = kin.A;
  const T Jt = kin.Jt;
  const T (&M)[3][3] = kin.M;
  const T (&lam)[3] = kin.lam;
  const T (&Q)[3][3] = kin.Q;
  const T (&h)[3] = kin.h;
  const T (&f1)[6] = kin.f1;
  const T (&f2d)[3] = kin.f2d;
  const T (&f2p)[3][2] = kin.f2p;
  const T f2t = kin.f2t;

  // products of the rows of Q: w[n][v] = Q_na Q_nb for the slot v = (a, b)
  T w[3][6];
#pragma unroll
  for (int n = 0; n < 3; ++n)
#pragma unroll
    for (int v = 0; v < 6; ++v) w[n][v] = Q[n][sym_i(v)] * Q[n][sym_j(v)];

  // rotated stress-like T~ = Q^T (L(eta):h) Q, times J_t
  T TJ[6];
  T hv[6];             // general stiffness: lab-frame Hencky strain (Voigt, engineering shear)
  T hLh[NPH];          // and h : L_i : h
  if (P.cubic) {
    // lambda I x I + 2 mu I_sym is the same in every basis; delta sum_n e_n^4
    // becomes delta sum_n w_n w_n^T
    const T tr = h[0] + h[1] + h[2];
    const T lt = T(P.cub_lambda) * tr;
    T c[3];
#pragma unroll
    for (int n = 0; n < 3; ++n) c[n] = T(P.cub_delta) * (w[n][0] * h[0] + w[n][1] * h[1] + w[n][2] * h[2]);
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      T t = c[0] * w[0][v] + c[1] * w[1][v] + c[2] * w[2][v];
      if (v < 3) t += lt + T(2.0 * P.cub_mu) * h[v];
      TJ[v] = Jt * t;
    }
  } else {
    T hm[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      const int i = sym_i(v), j = sym_j(v);
      hm[v] = Q[i][0] * h[0] * Q[j][0] + Q[i][1] * h[1] * Q[j][1] + Q[i][2] * h[2] * Q[j][2];
      hv[v] = v < 3 ? hm[v] : T(2) * hm[v];
    }
    T Tv[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
    T se = eh[0];
#pragma unroll
    for (int k = 1; k < NV; ++k) se += eh[k];
    const T eta0 = T(1) - se;
    const int np = P.same_L ? 1 : NPH;
    for (int p = 0; p < np; ++p) {
      const T ep = P.same_L ? T(1) : (p == 0 ? eta0 : eh[p - 1]);
      T s = T(0);
#pragma unroll
      for (int I = 0; I < 6; ++I) {
        T li = T(0);
#pragma unroll
        for (int J = 0; J < 6; ++J) li += T(P.Lv[p][I][J]) * hv[J];
        Tv[I] += ep * li;
        s += hv[I] * li;
      }
      hLh[p] = s;
    }
    T Tt[6];
    rot_sym6(Q, Tv, Tt);
#pragma unroll
    for (int v = 0; v < 6; ++v) TJ[v] = Jt * Tt[v];
  }
  const T cW = T(0.5) * (h[0] * TJ[0] + h[1] * TJ[1] + h[2] * TJ[2]);  // elastic energy 1/2 J_t h:L:h

  // twice the rotated stress S~ = dW_el/dE = 1/2 J_t f1 o T~, and the rotated
  // columns of A and rows of M
  T S2[6], Aq[3][3], Mq[3][3];
#pragma unroll
  for (int v = 0; v < 6; ++v) S2[v] = f1[v] * TJ[v];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Aq[c][a] = symget(A, c, 0) * Q[0][a] + symget(A, c, 1) * Q[1][a] + symget(A, c, 2) * Q[2][a];
      Mq[c][a] = M[c][0] * Q[0][a] + M[c][1] * Q[1][a] + M[c][2] * Q[2][a];
    }
  // dW_el/dF = 2 M S A = (M Q) 2S~ (A Q)^T
  T Pf[3][3];
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    T n[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      n[a] = Mq[p][0] * symget(S2, 0, a) + Mq[p][1] * symget(S2, 1, a) + Mq[p][2] * symget(S2, 2, a);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      Pf[p][c] = n[0] * Aq[c][0] + n[1] * Aq[c][1] + n[2] * Aq[c][2];
      g[3 * p + c] = Pf[p][c];
    }
  }
  // dW_el/dF^t = cW A - Zs with Zs the symmetric part of 2 E S A = M^T dW_el/dF
  T Zs[6];
#pragma unroll
  for (int v = 0; v < 6; ++v) {
    const int i = sym_i(v), j = sym_j(v);
    T z = M[0][i] * Pf[0][j] + M[1][i] * Pf[1][j] + M[2][i] * Pf[2][j];
    if (v >= 3) z = T(0.5) * (z + (M[0][j] * Pf[0][i] + M[1][j] * Pf[1][i] + M[2][j] * Pf[2][i]));
    Zs[v] = z;
  }
  T gU[6];
#pragma unroll
  for (int v = 0; v < 6; ++v) {
    const T t = cW * A[v] - Zs[v];
    gU[v] = v < 3 ? t : t + t;
  }
  // order parameters: elastic part along dU_k, chemical and obstacle energy,
  // dissipation and penalty (eta_0 = 1 - sum eta_hat, Sec. 3.1)
  T se = eh[0], d0 = ehn[0] - eh[0];
#pragma unroll
  for (int k = 1; k < NV; ++k) {
    se += eh[k];
    d0 += ehn[k] - eh[k];
  }
  const T eta0 = T(1) - se;
  const T neg0 = eta0 < T(0) ? eta0 : T(0);
  T Wloc = cW + T(P.W0);
  const T g0 = T(P.inv_mtau[0]) * d0 + T(P.eps_eta) * neg0;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    T qk = T(0);
#pragma unroll
    for (int l = 0; l < NV; ++l) qk += T(P.Cc[k][l]) * eh[l];
    const T d = eh[k] - ehn[k];
    const T neg = eh[k] < T(0) ? eh[k] : T(0);
    const T dis = T(P.inv_mtau[k + 1]) * d, pen = T(P.eps_eta) * neg;
    Wloc += eh[k] * (T(P.lin[k]) + T(0.5) * qk) + T(0.5) * (dis * d + pen * neg);
    T gk = T(P.lin[k]) + qk;
#pragma unroll
    for (int v = 0; v < 6; ++v) gk += gU[v] * T(P.dU[k][v]);
    g[9 + k] = gk + ((dis + pen) - g0);  // the penalty, by far the largest, last
  }
  Wloc += T(0.5) * (T(P.inv_mtau[0]) * d0 * d0 + T(P.eps_eta) * neg0 * neg0);
  if (!P.same_L) {
#pragma unroll
    for (int k = 0; k < NV; ++k) g[9 + k] += T(0.5) * Jt * (hLh[k + 1] - hLh[0]);
  }
  *W = Wloc;
  if (!Emit::want) return;

  // ---------------------------------------------------------------------
  // Spectral second derivative: J_t (Dh[X]:L~:Dh[Y] + h''-part) as a symmetric
  // form Mb in the Voigt slots of X~, the diagonal slots holding half of X~_aa
  // (X~ = a q^T + q a^T has 2 a_a q_a there)
  T Mb[21];  // packed upper triangle, hm6(I, J)
  auto hm6 = [](int I, int J) { return I <= J ? I * 6 - (I * (I - 1)) / 2 + (J - I) : J * 6 - (J * (J - 1)) / 2 + (I - J); };
  {
    T fJ[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) fJ[v] = Jt * f1[v];
    if (P.cubic) {
      T dw[3][6];
#pragma unroll
      for (int n = 0; n < 3; ++n)
#pragma unroll
        for (int v = 0; v < 6; ++v) dw[n][v] = T(P.cub_delta) * w[n][v];
#pragma unroll
      for (int I = 0; I < 6; ++I)
#pragma unroll
        for (int J = I; J < 6; ++J) {
          T v = dw[0][I] * w[0][J] + dw[1][I] * w[1][J] + dw[2][I] * w[2][J];
          if (I < 3 && J < 3) v += T(P.cub_lambda);
          if (I == J) v += I < 3 ? T(2.0 * P.cub_mu) : T(P.cub_mu);
          Mb[hm6(I, J)] = fJ[I] * f1[J] * v;
        }
    } else {
      T Nv[6][6];  // v(Q X~ Q^T) = Nv v(X~), engineering shear
      for (int I = 0; I < 6; ++I) {
        const int i = sym_i(I), j = sym_j(I);
        const T cI = (I < 3) ? T(1) : T(2);
        for (int B = 0; B < 6; ++B) {
          const int a = sym_i(B), b = sym_j(B);
          Nv[I][B] = (B < 3) ? cI * Q[i][a] * Q[j][a] : cI * T(0.5) * (Q[i][a] * Q[j][b] + Q[i][b] * Q[j][a]);
        }
      }
      T LN[6][6];
      for (int I = 0; I < 6; ++I) {
        T Le[6];  // row I of L(eta)
        for (int J = 0; J < 6; ++J) {
          T l = T(P.Lv[0][I][J]);
          if (!P.same_L) {
            l = eta0 * l;
            for (int k = 0; k < NV; ++k) l += eh[k] * T(P.Lv[k + 1][I][J]);
          }
          Le[J] = l;
        }
        for (int B = 0; B < 6; ++B) {
          T s = T(0);
          for (int J = 0; J < 6; ++J) s += Le[J] * Nv[J][B];
          LN[I][B] = s;
        }
      }
#pragma unroll
      for (int I = 0; I < 6; ++I)
#pragma unroll
        for (int J = I; J < 6; ++J) {
          T s = T(0);
          for (int K = 0; K < 6; ++K) s += Nv[K][I] * LN[K][J];
          Mb[hm6(I, J)] = fJ[I] * f1[J] * s;
        }
    }
    // sum over a, b, c of f2(a,b,c) T~_ab into the slots (a,c), (b,c)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Mb[hm6(a, a)] += f2d[a] * (T(4) * TJ[a]);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (c == a) continue;
        const int n = 3 - a - c, sl = 3 + n;
        Mb[hm6(sl, sl)] += (a < c ? f2p[n][0] : f2p[n][1]) * TJ[a];
      }
    }
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      const int p = n == 0 ? 1 : 0, r = n == 2 ? 1 : 2, sl = 3 + n;
      const T t2 = T(2) * TJ[sl];
      Mb[hm6(p, sl)] += f2p[n][0] * t2;
      Mb[hm6(r, sl)] += f2p[n][1] * t2;
      Mb[hm6(3 + r, 3 + p)] += f2t * TJ[sl];  // slots (p, n) and (r, n)
    }
  }
  // left vectors of the directions in the eigenbasis: Mq[p] (F_p.) and
  // Uq[i] = -Lambda Q^T e_i (entry (i, .) of F^t)
  T Uq[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int a = 0; a < 3; ++a) Uq[i][a] = -(lam[a] * Q[i][a]);
  T il[3];  // 1 / lambda
#pragma unroll
  for (int a = 0; a < 3; ++a) il[a] = P.hencky == 0 ? f1[a] : T(1) / lam[a];
  T FU[9][6], K[21];
#pragma unroll
  for (int r = 0; r < 9; ++r)
#pragma unroll
    for (int v = 0; v < 6; ++v) FU[r][v] = T(0);
#pragma unroll
  for (int v = 0; v < 21; ++v) K[v] = T(0);
#pragma unroll
  for (int c2 = 0; c2 < 3; ++c2) {
    T Y[6][3];  // Mb N_c2: change of slot v along (column c2, left vector e_b)
#pragma unroll
    for (int v = 0; v < 6; ++v)
#pragma unroll
      for (int b = 0; b < 3; ++b)
        Y[v][b] = Mb[hm6(v, voigt_slot(b, 0))] * Aq[c2][0] + Mb[hm6(v, voigt_slot(b, 1))] * Aq[c2][1] +
                  Mb[hm6(v, voigt_slot(b, 2))] * Aq[c2][2];
    T sa[3];  // 2S~ a_c2
#pragma unroll
    for (int a = 0; a < 3; ++a)
      sa[a] = symget(S2, a, 0) * Aq[c2][0] + symget(S2, a, 1) * Aq[c2][1] + symget(S2, a, 2) * Aq[c2][2];
#pragma unroll
    for (int c = 0; c <= c2; ++c) {
      T R[3][3];
      const T asa = Aq[c][0] * sa[0] + Aq[c][1] * sa[1] + Aq[c][2] * sa[2];
#pragma unroll
      for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          if (c == c2 && b < e) {
            R[e][b] = R[b][e];
            continue;
          }
          T s = Aq[c][0] * Y[voigt_slot(e, 0)][b] + Aq[c][1] * Y[voigt_slot(e, 1)][b] + Aq[c][2] * Y[voigt_slot(e, 2)][b];
          if (e == b) s += asa * il[e];
          R[e][b] = s;
        }
      T Zf[3][3], Zu[3][3];  // left vectors times R
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          Zf[p][b] = Mq[p][0] * R[0][b] + Mq[p][1] * R[1][b] + Mq[p][2] * R[2][b];
          Zu[p][b] = Uq[p][0] * R[0][b] + Uq[p][1] * R[1][b] + Uq[p][2] * R[2][b];
        }
      // acc += x . y, as three multiply-adds into acc
      auto dot_to = [](T& acc, const T* x, const T* y) {
        acc += x[0] * y[0];
        acc += x[1] * y[1];
        acc += x[2] * y[2];
      };
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          // F_pc with F_rc2 (final)
          if (c < c2 || p <= r) {
            const int i = 3 * p + c, j = 3 * r + c2;
            emit(i <= j ? hidx(i, j) : hidx(j, i), Zf[p][0] * Mq[r][0] + Zf[p][1] * Mq[r][1] + Zf[p][2] * Mq[r][2]);
          }
          // F_pc with F^t_(r, c2), and F_pc2 with F^t_(r, c)
          dot_to(FU[3 * p + c][voigt_slot(r, c2)], Zf[p], Uq[r]);
          if (c < c2) dot_to(FU[3 * p + c2][voigt_slot(r, c)], Zu[r], Mq[p]);
          // F^t_(p, c) with F^t_(r, c2); a pair within one slot counts twice
          if (c < c2 || p <= r) {
            const int v = voigt_slot(p, c), x = voigt_slot(r, c2);
            dot_to(K[hm6(v, x)], Zu[p], Uq[r]);
            if (v == x && !(p == r && c == c2)) dot_to(K[hm6(v, x)], Zu[p], Uq[r]);
          }
        }
    }
  }
  // second derivatives of F^e along F and F^t, and of J_t: tr(A dU) P - A dU P^T
  T At[6];
#pragma unroll
  for (int v = 0; v < 6; ++v) At[v] = v < 3 ? A[v] : A[v] + A[v];
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int v = 0; v < 6; ++v) {
        const int i = sym_i(v), j = sym_j(v);
        T& fu = FU[3 * p + c][v];
        fu += At[v] * Pf[p][c];
        fu -= symget(A, c, i) * Pf[p][j];
        if (v >= 3) fu -= symget(A, c, j) * Pf[p][i];
      }
  // K += 2 tr(Z' dU A dU') - tr(A dU) tr(Z' dU') - tr(Z' dU) tr(A dU'), Z' = Zs - cW/2 A
  {
    T Z[6], Z2[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      Z[v] = Zs[v] - T(0.5) * cW * A[v];
      Z2[v] = Z[v] + Z[v];
    }
#pragma unroll
    for (int v = 0; v < 6; ++v)
#pragma unroll
      for (int x = v; x < 6; ++x) {
        const int i = sym_i(v), j = sym_j(v), k = sym_i(x), l = sym_j(x);
        T& kk = K[hm6(v, x)];
        // tr(2 Z E A E') over the entries (i,j), (j,i) of E and (k,l), (l,k) of E'
        kk += symget(Z2, l, i) * symget(A, j, k);
        if (x >= 3) kk += symget(Z2, k, i) * symget(A, j, l);
        if (v >= 3) {
          kk += symget(Z2, l, j) * symget(A, i, k);
          if (x >= 3) kk += symget(Z2, k, j) * symget(A, i, l);
        }
        kk -= At[v] * (x < 3 ? Z[x] : Z2[x]);
        kk -= (v < 3 ? Z[v] : Z2[v]) * At[x];
      }
  }
  // per-phase stiffness: (dL_k h) along the directions, LX[k][v] for F^t
  T LX[NV][6];
  if (!P.same_L) {
    for (int k = 0; k < NV; ++k) {
      T lv[6], lr[6];
      for (int I = 0; I < 6; ++I) {
        T s = T(0);
        for (int J = 0; J < 6; ++J) s += (T(P.Lv[k + 1][I][J]) - T(P.Lv[0][I][J])) * hv[J];
        lv[I] = s;
      }
      rot_sym6(Q, lv, lr);
      for (int v = 0; v < 6; ++v) lr[v] = Jt * f1[v] * lr[v];
      for (int v = 0; v < 6; ++v) LX[k][v] = T(0);
      for (int c = 0; c < 3; ++c) {
        T t[3];
        for (int a = 0; a < 3; ++a)
          t[a] = symget(lr, a, 0) * Aq[c][0] + symget(lr, a, 1) * Aq[c][1] + symget(lr, a, 2) * Aq[c][2];
        for (int p = 0; p < 3; ++p) {
          T fk = t[0] * Mq[p][0] + t[1] * Mq[p][1] + t[2] * Mq[p][2];
          for (int v = 0; v < 6; ++v) fk += FU[3 * p + c][v] * T(P.dU[k][v]);
          emit(hidx(3 * p + c, 9 + k), fk);
          LX[k][voigt_slot(p, c)] += t[0] * Uq[p][0] + t[1] * Uq[p][1] + t[2] * Uq[p][2];
        }
      }
    }
  } else {
    if constexpr (std::is_same<T, double>::value) {
      if (eta_fx(P, FU, K, eh, eta0, emit)) return;
    }
#pragma unroll 1
    for (int k = 0; k < NV; ++k) {
      T d[6];
#pragma unroll
      for (int v = 0; v < 6; ++v) d[v] = T(P.dU[k][v]);
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        T s = FU[r][0] * d[0];
#pragma unroll
        for (int v = 1; v < 6; ++v) s += FU[r][v] * d[v];
        emit(hidx(r, 9 + k), s);
      }
    }
  }
  // eta-eta: K along the dU_k, and the local terms
  // Cc_kl + d_0 + delta_kl d_k, d_i = 1/(m_i tau) + eps [eta_i < 0]
  const T dd0 = T(P.inv_mtau[0]) + (eta0 < T(0) ? T(P.eps_eta) : T(0));
#pragma unroll 1
  for (int q = 0; q < NV; ++q) {
    T t[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      T s = K[hm6(v, 0)] * T(P.dU[q][0]);
#pragma unroll
      for (int x = 1; x < 6; ++x) s += K[hm6(v, x)] * T(P.dU[q][x]);
      t[v] = s;
    }
    for (int p = 0; p <= q; ++p) {
      T s = T(P.Cc[p][q]);
#pragma unroll
      for (int v = 0; v < 6; ++v) s += t[v] * T(P.dU[p][v]);
      T loc = dd0;
      if (p == q) loc += T(P.inv_mtau[p + 1]) + (eh[p] < T(0) ? T(P.eps_eta) : T(0));
      if (!P.same_L) {
        T ap = T(0), aq = T(0);  // tr(A dU_p), tr(A dU_q)
        for (int v = 0; v < 6; ++v) {
          ap += At[v] * T(P.dU[p][v]);
          aq += At[v] * T(P.dU[q][v]);
          s += LX[p][v] * T(P.dU[q][v]) + LX[q][v] * T(P.dU[p][v]);
        }
        s += T(0.5) * Jt * (ap * (hLh[q + 1] - hLh[0]) + aq * (hLh[p + 1] - hLh[0]));
      }
      emit(hidx(9 + p, 9 + q), s + loc);
    }
  }
}

// Parts of the elastic energy that belong to the cubic constants
// theta = (C11, C12, C44) of a stiffness shared by all phases (the energy is
// linear in them): E[k] = the energy density at unit theta_k with the others 0,
// and D[k] = its derivative along a direction of the unknowns with the gradient
// dF (row-major) of the displacements and the change dUt (Voigt entries) of F^t.
// One set of kinematics serves the three parts. In the eigenbasis the unit
// stiffnesses give the stresses sum_n c_n w_n w_n^T-wise for C11 (c = w h), the
// trace minus that for C12, and 2 h minus twice that for C44.
template <typename T>
PFM_HD void qp_cubic_parts(const DevParams& P, const T Fin[9], const T eh[NV], const T dF[9], const T dUt[6], T E[3],
                           T D[3]) {
  Kinematics<T> kin;
  kinematics<false>(P, Fin, eh, kin);
  const T (&Q)[3][3] = kin.Q;
  const T (&h)[3] = kin.h;
  T cu[6];  // Voigt slots of sum_n (w_n . h) w_n
#pragma unroll
  for (int v = 0; v < 6; ++v) cu[v] = T(0);
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    T w[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) w[v] = Q[n][sym_i(v)] * Q[n][sym_j(v)];
    const T c = w[0] * h[0] + w[1] * h[1] + w[2] * h[2];
#pragma unroll
    for (int v = 0; v < 6; ++v) cu[v] += c * w[v];
  }
  const T tr = h[0] + h[1] + h[2];
  T Aq[3][3], Mq[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Aq[c][a] = symget(kin.A, c, 0) * Q[0][a] + symget(kin.A, c, 1) * Q[1][a] + symget(kin.A, c, 2) * Q[2][a];
      Mq[c][a] = kin.M[c][0] * Q[0][a] + kin.M[c][1] * Q[1][a] + kin.M[c][2] * Q[2][a];
    }
  T trAdU = T(0);  // tr(A dF^t)
#pragma unroll
  for (int v = 0; v < 6; ++v) trAdU += (v < 3 ? kin.A[v] : kin.A[v] + kin.A[v]) * dUt[v];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T TJ[6], S2[6];
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      T t = k == 0 ? cu[v] : (k == 1 ? -cu[v] : T(-2) * cu[v]);
      if (v < 3) {
        if (k == 1) t += tr;
        if (k == 2) t += T(2) * h[v];
      }
      TJ[v] = kin.Jt * t;
      S2[v] = kin.f1[v] * TJ[v];
    }
    const T cW = T(0.5) * (h[0] * TJ[0] + h[1] * TJ[1] + h[2] * TJ[2]);
    T Pf[3][3];
    T d = T(0);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      T n[3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
        n[a] = Mq[p][0] * symget(S2, 0, a) + Mq[p][1] * symget(S2, 1, a) + Mq[p][2] * symget(S2, 2, a);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        Pf[p][c] = n[0] * Aq[c][0] + n[1] * Aq[c][1] + n[2] * Aq[c][2];
        d += Pf[p][c] * dF[3 * p + c];
      }
    }
    // along F^t: cW A - sym(M^T Pf)
    d += cW * trAdU;
#pragma unroll
    for (int v = 0; v < 6; ++v) {
      const int i = sym_i(v), j = sym_j(v);
      T z = kin.M[0][i] * Pf[0][j] + kin.M[1][i] * Pf[1][j] + kin.M[2][i] * Pf[2][j];
      if (v >= 3) z += kin.M[0][j] * Pf[0][i] + kin.M[1][j] * Pf[1][i] + kin.M[2][j] * Pf[2][i];
      d -= z * dUt[v];
    }
    E[k] = cW;
    D[k] = d;
  }
}

// qp_point with the packed Hessian (if wanted) in an array.
template <typename T, bool WANT_HESS>
PFM_HD_BIG void qp_local(const DevParams& P, const T Fin[9], const T eh[NV], const T ehn[NV], T* W, T g[NZ], T* Hp) {
  if constexpr (WANT_HESS)
    qp_point<T>(P, Fin, eh, ehn, W, g, HessArray<T>{Hp});
  else
    qp_point<T>(P, Fin, eh, ehn, W, g, NoHess<T>{});
}

}  // namespace pfm
