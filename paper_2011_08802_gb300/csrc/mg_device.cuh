// Building blocks of the multigrid kernels (the transfers also compile for
// the host, where a test checks them against the oracle), shared by the
// single-problem kernels (mg_kernels.cu) and the batched kernels (batch.cu):
// integer-exact 1-D interpolation between structured grids on the same box,
// state injection, prolongation and restriction at one node, the Chebyshev
// smoothing updates at one node and the power-iteration start vector.
//
// Grid transfer in 1-D: fine node i sits at coarse coordinate i*nc/nf; with
// i*nc = I0*nf + rem, its interpolation weights are (1 - rem/nf) on coarse
// node I0 and rem/nf on I0+1. All index arithmetic is integer, so P and
// R = P^T use identical weights on nested (nf = 2 nc) and non-nested grids.
#pragma once

#include <cfloat>
#include <cstdint>

#include "common.cuh"

namespace pfm {

struct Interp1 {
  int i0;
  double t;  // weight of i0+1
};

__host__ __device__ __forceinline__ Interp1 interp1(int i, int nf, int nc) {
  // coarse coordinate of fine node i: i*nc/nf
  long long num = (long long)i * nc;
  int I0 = int(num / nf);
  long long rem = num - (long long)I0 * nf;
  if (I0 >= nc) { I0 = nc - 1; rem = nf; }
  return {I0, double(rem) / double(nf)};
}

// The 8 trilinear weights of the point with per-axis local coordinates t, and
// the value of a nodal field X (rows of sy, planes of sz nodes; X at the first
// corner) there. Formed once per node and used for every field; points with
// weight 0 are not read (they may lie outside the grid).
__host__ __device__ __forceinline__ void trilinear_weights(const double t[3], double w[8]) {
  const double u[3] = {1.0 - t[0], 1.0 - t[1], 1.0 - t[2]};
#pragma unroll
  for (int c = 0; c < 8; ++c)
    w[c] = ((c & 1) ? t[0] : u[0]) * (((c >> 1) & 1) ? t[1] : u[1]) * ((c >> 2) ? t[2] : u[2]);
}
template <typename T>
__host__ __device__ __forceinline__ double trilinear(const T* X, int64_t sy, int64_t sz, const double w[8]) {
  double s = 0.0;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    if (w[c] != 0.0) s += w[c] * double(X[(c & 1) + ((c >> 1) & 1) * sy + (c >> 2) * sz]);
  return s;
}

// Coarse node idx: the fine Q1 field evaluated at its position, all fields.
__host__ __device__ __forceinline__ void inject_node(const Grid& f, const Grid& c, const double* __restrict__ Uf,
                                            double* __restrict__ Uc, int64_t idx) {
  const int64_t nnc = c.nn();
  const int64_t nnf = f.nn();
  int I = int(idx % (c.nx + 1));
  int J = int((idx / (c.nx + 1)) % (c.ny + 1));
  int K = int(idx / (int64_t(c.nx + 1) * (c.ny + 1)));
  // fine coordinate of coarse node: I*nf/nc
  int i0[3];
  double t[3];
  const int Ic[3] = {I, J, K}, nfv[3] = {f.nx, f.ny, f.nz}, ncv[3] = {c.nx, c.ny, c.nz};
  for (int d = 0; d < 3; ++d) {
    Interp1 p = interp1(Ic[d], ncv[d], nfv[d]);  // coarse node in fine coordinates
    i0[d] = p.i0;
    t[d] = p.t;
  }
  double w[8];
  trilinear_weights(t, w);
  const int64_t sy = f.nx + 1, sz = int64_t(f.nx + 1) * (f.ny + 1);
  const double* X = Uf + i0[0] + i0[1] * sy + i0[2] * sz;
  for (int fld = 0; fld < NF; ++fld) Uc[fld * nnc + idx] = trilinear(X + fld * nnf, sy, sz, w);
}

// Fine node idx: xf += P xc at its free DOFs.
template <typename T>
__host__ __device__ __forceinline__ void prolong_node(const Grid& f, const Grid& c, const T* __restrict__ xc,
                                             const dmask_t* __restrict__ mf, T* __restrict__ xf, int64_t idx) {
  const int64_t nnf = f.nn();
  const int64_t nnc = c.nn();
  int i = int(idx % (f.nx + 1));
  int j = int((idx / (f.nx + 1)) % (f.ny + 1));
  int k = int(idx / (int64_t(f.nx + 1) * (f.ny + 1)));
  Interp1 px = interp1(i, f.nx, c.nx), py = interp1(j, f.ny, c.ny), pz = interp1(k, f.nz, c.nz);
  const double t[3] = {px.t, py.t, pz.t};
  double w[8];
  trilinear_weights(t, w);
  const int64_t sy = c.nx + 1, sz = int64_t(c.nx + 1) * (c.ny + 1);
  const T* X = xc + px.i0 + py.i0 * sy + pz.i0 * sz;
  const dmask_t dm = mf[idx];
  for (int fld = 0; fld < NF; ++fld) {
    if ((dm >> fld) & 1) continue;
    xf[fld * nnf + idx] += T(trilinear(X + fld * nnc, sy, sz, w));
  }
}

// Coarse node idx: rc = (P^T (rf - y)) there (y null: P^T rf), zero at its
// Dirichlet DOFs. Coarse
// node I collects fine nodes i with |i*nc - I*nf| < nf, weight
// 1 - |i*nc - I*nf|/nf (per axis).
template <typename T>
__host__ __device__ __forceinline__ void restrict_node(const Grid& f, const Grid& c, const T* __restrict__ rf,
                                              const dmask_t* __restrict__ mc, T* __restrict__ rc, int64_t idx,
                                              const T* __restrict__ y = nullptr) {
  const int64_t nnf = f.nn();
  const int64_t nnc = c.nn();
  const int Ic[3] = {int(idx % (c.nx + 1)), int((idx / (c.nx + 1)) % (c.ny + 1)),
                     int(idx / (int64_t(c.nx + 1) * (c.ny + 1)))};
  const int nfv[3] = {f.nx, f.ny, f.nz}, ncv[3] = {c.nx, c.ny, c.nz};
  int lo[3], hi[3];
  for (int d = 0; d < 3; ++d) {
    long long center = (long long)Ic[d] * nfv[d];  // in units of 1/(nf*nc) ... i*nc vs I*nf
    // i*nc > I*nf - nf  and  i*nc < I*nf + nf
    long long a = center - nfv[d];
    long long b = center + nfv[d];
    int l = int(a >= 0 ? a / ncv[d] + 1 : 0);
    int h = int(b % ncv[d] == 0 ? b / ncv[d] - 1 : b / ncv[d]);
    if (l < 0) l = 0;
    if (h > nfv[d]) h = nfv[d];
    lo[d] = l;
    hi[d] = h;
  }
  const dmask_t dm = mc[idx];
  double acc[NF];
  for (int fld = 0; fld < NF; ++fld) acc[fld] = 0.0;
  auto weight = [&](int d, int i) {
    return 1.0 - fabs(double((long long)i * ncv[d] - (long long)Ic[d] * nfv[d])) / nfv[d];
  };
  // the x weights once per node (an FP64 division each): at most 4 fine nodes
  // when nf <= 2 nc, the hierarchy's case
  constexpr int WX = 4;
  double wxa[WX];
#pragma unroll
  for (int m = 0; m < WX; ++m) wxa[m] = lo[0] + m <= hi[0] ? weight(0, lo[0] + m) : 0.0;
  for (int k = lo[2]; k <= hi[2]; ++k) {
    const double wz = weight(2, k);
    for (int j = lo[1]; j <= hi[1]; ++j) {
      const double wyz = weight(1, j) * wz;
#pragma unroll 4
      for (int i = lo[0]; i <= hi[0]; ++i) {
        const int m = i - lo[0];
        const double w = (m < WX ? wxa[m & (WX - 1)] : weight(0, i)) * wyz;
        const int64_t fn = i + int64_t(f.nx + 1) * (j + int64_t(f.ny + 1) * k);
        for (int fld = 0; fld < NF; ++fld) acc[fld] += w * double(y ? rf[fld * nnf + fn] - y[fld * nnf + fn] : rf[fld * nnf + fn]);
      }
    }
  }
  for (int fld = 0; fld < NF; ++fld) rc[fld * nnc + idx] = ((dm >> fld) & 1) ? T(0) : T(acc[fld]);
}

// Transfers of FP32 vectors between non-nested grids, one field at a time. The
// weights are fractions with the common denominator N = nf_x nf_y nf_z and
// integer numerators; for N < 2^24 the numerators are FP32 numbers, and the sums
// of numerator x value are formed with a compensated FP32 accumulator (the
// product split by a fused multiply-add, TwoSum, Ogita, Rump and Oishi 2005) and
// divided by N at the end: the accuracy of FP64 sums rounded once to FP32, on
// the FP32 pipes. The FP64 form (weights, products and conversions all on the
// FP64 pipe) took 131 us per restriction and 95 us per prolongation on average
// over the levels of 75^3 elements; this form 36 and 22 us.
struct CSum {
  float s = 0.f, c = 0.f;
  __host__ __device__ __forceinline__ void add(float w, float x) {
#ifdef __CUDA_ARCH__
    const float p = __fmul_rn(w, x);
    const float e = __fmaf_rn(w, x, -p);
    const float t = __fadd_rn(s, p);
    const float bb = __fsub_rn(t, s);
    const float q = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(p, bb));
    c = __fadd_rn(c, __fadd_rn(q, e));
#else
    const float p = w * x;
    const float e = fmaf(w, x, -p);
    const float t = s + p;
    const float bb = t - s;
    const float q = (s - (t - bb)) + (p - bb);
    c += q + e;
#endif
    s = t;
  }
  // (s + c) / n, n an integer: 1/n as an FP32 number and its remainder
  __host__ __device__ __forceinline__ float over(float n) const {
    const float r = 1.f / n;
    const float rl = r * fmaf(-n, r, 1.f);
#ifdef __CUDA_ARCH__
    const float p = __fmul_rn(s, r);
    return __fadd_rn(p, __fmaf_rn(s, rl, __fmaf_rn(c, r, __fmaf_rn(s, r, -p))));
#else
    const float p = s * r;
    return p + fmaf(s, rl, fmaf(c, r, fmaf(s, r, -p)));
#endif
  }
};
// common denominator of the weights, and whether the integer form applies
inline __host__ __device__ int64_t transfer_denominator(const Grid& f) { return int64_t(f.nx) * f.ny * f.nz; }
inline __host__ __device__ bool transfer_integer(const Grid& f) { return transfer_denominator(f) < (int64_t(1) << 24); }

// Fine nodes lo..hi of an axis with a weight at coarse node I: |i nc - I nf| < nf.
inline __host__ __device__ void transfer_support(int I, int nf, int nc, int& lo, int& hi) {
  const int64_t center = int64_t(I) * nf;
  const int64_t a = center - nf, b = center + nf;
  lo = a >= 0 ? int(a / nc) + 1 : 0;
  hi = int((b + nc - 1) / nc) - 1;
  if (hi > nf) hi = nf;
}

// The FP64 sums of one (node, field), for results that are not finite: numerator x
// value overflows in FP32 from values of 2^104 on, and its remainder makes NaN of an
// infinite value. Rare, so out of line and with arguments that a kernel has at hand
// anyway (passing the node indices kept registers for the call and cost a V-cycle on
// 33^3 elements 1.1 per cent).
inline __host__ __device__ __noinline__ float prolong_entry_f64(Grid f, Grid c, const float* xc, int64_t idx) {
  const int64_t nnf = f.nn(), node = idx % nnf;
  const Interp1 px = interp1(int(node % (f.nx + 1)), f.nx, c.nx),
                py = interp1(int((node / (f.nx + 1)) % (f.ny + 1)), f.ny, c.ny),
                pz = interp1(int(node / (int64_t(f.nx + 1) * (f.ny + 1))), f.nz, c.nz);
  const double t[3] = {px.t, py.t, pz.t};
  double w[8];
  trilinear_weights(t, w);
  const int64_t sy = c.nx + 1, sz = int64_t(c.nx + 1) * (c.ny + 1);
  return float(trilinear(xc + (idx / nnf) * c.nn() + px.i0 + py.i0 * sy + pz.i0 * sz, sy, sz, w));
}
inline __host__ __device__ __noinline__ float restrict_entry_f64(Grid f, Grid c, const float* rf, const float* y,
                                                                 int64_t idx) {
  const int64_t nnc = c.nn(), node = idx % nnc, off = (idx / nnc) * f.nn();
  const int Ic[3] = {int(node % (c.nx + 1)), int((node / (c.nx + 1)) % (c.ny + 1)),
                     int(node / (int64_t(c.nx + 1) * (c.ny + 1)))};
  const int nf[3] = {f.nx, f.ny, f.nz}, nc[3] = {c.nx, c.ny, c.nz};
  int lo[3], hi[3];
  for (int d = 0; d < 3; ++d) transfer_support(Ic[d], nf[d], nc[d], lo[d], hi[d]);
  auto weight = [&](int d, int i) {
    return 1.0 - fabs(double(int64_t(i) * nc[d] - int64_t(Ic[d]) * nf[d])) / nf[d];
  };
  double acc = 0.0;
  for (int k = lo[2]; k <= hi[2]; ++k)
    for (int j = lo[1]; j <= hi[1]; ++j)
      for (int i = lo[0]; i <= hi[0]; ++i) {
        const int64_t n = off + i + int64_t(f.nx + 1) * (j + int64_t(f.ny + 1) * k);
        acc += weight(0, i) * weight(1, j) * weight(2, k) * double(y ? rf[n] - y[n] : rf[n]);
      }
  return float(acc);
}
inline __host__ __device__ bool transfer_finite(float v) { return fabsf(v) <= FLT_MAX; }

// (P x)(i, j, k) of the coarse field x.
__host__ __device__ __forceinline__ float prolong_value_int(const Grid& f, const Grid& c, const float* __restrict__ x,
                                                            int i, int j, int k) {
  const int fi[3] = {i, j, k}, nf[3] = {f.nx, f.ny, f.nz}, nc[3] = {c.nx, c.ny, c.nz};
  int i0[3], w[3][2];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int64_t num = int64_t(fi[d]) * nc[d];
    int q = int(num / nf[d]);
    int rem = int(num - int64_t(q) * nf[d]);
    if (q >= nc[d]) {
      q = nc[d] - 1;
      rem = nf[d];
    }
    i0[d] = q;
    w[d][0] = nf[d] - rem;
    w[d][1] = rem;
  }
  const int64_t sy = c.nx + 1, sz = int64_t(c.nx + 1) * (c.ny + 1);
  const float* X = x + i0[0] + i0[1] * sy + i0[2] * sz;
  CSum a;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int a0 = m & 1, a1 = (m >> 1) & 1, a2 = m >> 2;
    const int wt = w[0][a0] * w[1][a1] * w[2][a2];
    if (wt != 0) a.add(float(wt), X[a0 + a1 * sy + a2 * sz]);
  }
  return a.over(float(transfer_denominator(f)));
}

// (P^T (r - y))(I, J, K) of the fine fields r and y (y null: P^T r).
__host__ __device__ __forceinline__ float restrict_value_int(const Grid& f, const Grid& c, const float* __restrict__ r,
                                                             const float* __restrict__ y, int I, int J, int K) {
  const int Ic[3] = {I, J, K}, nf[3] = {f.nx, f.ny, f.nz}, nc[3] = {c.nx, c.ny, c.nz};
  int lo[3], hi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) transfer_support(Ic[d], nf[d], nc[d], lo[d], hi[d]);
  auto weight = [&](int d, int i) {
    const int64_t t = int64_t(i) * nc[d] - int64_t(Ic[d]) * nf[d];
    return nf[d] - int(t < 0 ? -t : t);
  };
  const int64_t sy = f.nx + 1, sz = int64_t(f.nx + 1) * (f.ny + 1);
  CSum a;
  for (int k = lo[2]; k <= hi[2]; ++k) {
    const int wz = weight(2, k);
    for (int j = lo[1]; j <= hi[1]; ++j) {
      const int wyz = weight(1, j) * wz;
      const int64_t row = j * sy + k * sz;
#pragma unroll 4
      for (int i = lo[0]; i <= hi[0]; ++i)
        a.add(float(weight(0, i) * wyz), y ? r[row + i] - y[row + i] : r[row + i]);
    }
  }
  return a.over(float(transfer_denominator(f)));
}

// One (node, field) of the transfers: idx = field * nodes + node.
__host__ __device__ __forceinline__ void prolong_entry_int(const Grid& f, const Grid& c, const float* __restrict__ xc,
                                                           const dmask_t* __restrict__ mf, float* __restrict__ xf,
                                                           int64_t idx) {
  const int64_t nnf = f.nn();
  const int fld = int(idx / nnf);
  const int64_t node = idx - fld * nnf;
  if ((mf[node] >> fld) & 1) return;
  const int nxp = f.nx + 1, nyp = f.ny + 1;
  const int64_t r = node / nxp;
  float v = prolong_value_int(f, c, xc + fld * c.nn(), int(node - r * nxp), int(r % nyp), int(r / nyp));
  if (!transfer_finite(v)) v = prolong_entry_f64(f, c, xc, idx);
  xf[idx] += v;
}
__host__ __device__ __forceinline__ void restrict_entry_int(const Grid& f, const Grid& c, const float* __restrict__ rf,
                                                            const dmask_t* __restrict__ mc, float* __restrict__ rc,
                                                            int64_t idx, const float* __restrict__ y = nullptr) {
  const int64_t nnc = c.nn();
  const int fld = int(idx / nnc);
  const int64_t node = idx - fld * nnc;
  const int nxp = c.nx + 1, nyp = c.ny + 1;
  const int64_t r = node / nxp;
  float v = 0.f;
  if (!((mc[node] >> fld) & 1)) {
    v = restrict_value_int(f, c, rf + fld * f.nn(), y ? y + fld * f.nn() : nullptr, int(node - r * nxp), int(r % nyp),
                           int(r / nyp));
    if (!transfer_finite(v)) v = restrict_entry_f64(f, c, rf, y, idx);
  }
  rc[idx] = v;
}

// Nested grids (nf = 2 nc on every axis), the case of every level of a
// power-of-two hierarchy: fine node i of an axis coincides with coarse node
// i/2 (even i, weight 1) or lies midway between coarse nodes (i-1)/2 and
// (i+1)/2 (odd i, weights 1/2). These are the weights of the general
// transfers above on such grids; being powers of two they are exact in
// binary arithmetic, so the node bodies below form their sums in T (FP32 in
// the FP32 preconditioner) and take the node from its (i, j, k) position.

// One (node, field) of the nested transfers, for one thread each. Prolongation
// averages the coarse values at floor and ceil of half the index on every axis
// (the same one twice at an even index: (a + a) / 2 = a exactly), so lanes at
// odd and even nodes run the same instructions. Values within a factor 8 of the
// largest number overflow in those sums: then only the different ones are added.
template <typename T>
__host__ __device__ __noinline__ T prolong_value_nested_few(const T* X, int64_t sy, int64_t sz, int i, int j, int k) {
  T s = T(0);
  for (int a2 = 0; a2 <= (k & 1); ++a2)
    for (int a1 = 0; a1 <= (j & 1); ++a1)
      for (int a0 = 0; a0 <= (i & 1); ++a0) s += X[(i >> 1) + a0 + ((j >> 1) + a1) * sy + ((k >> 1) + a2) * sz];
  return s * ((i & 1 ? T(0.5) : T(1)) * (j & 1 ? T(0.5) : T(1)) * (k & 1 ? T(0.5) : T(1)));
}
template <typename T>
__host__ __device__ __forceinline__ T prolong_value_nested(const T* __restrict__ X, int64_t sy, int64_t sz, int i, int j,
                                                           int k) {
  const int i0 = i >> 1, i1 = (i + 1) >> 1;
  const int64_t r0 = (j >> 1) * sy, r1 = ((j + 1) >> 1) * sy, p0 = (k >> 1) * sz, p1 = ((k + 1) >> 1) * sz;
  const T a = (X[p0 + r0 + i0] + X[p0 + r0 + i1]) + (X[p0 + r1 + i0] + X[p0 + r1 + i1]);
  const T b = (X[p1 + r0 + i0] + X[p1 + r0 + i1]) + (X[p1 + r1 + i0] + X[p1 + r1 + i1]);
  const T v = T(0.125) * (a + b);
  return v - v == T(0) ? v : prolong_value_nested_few<T>(X, sy, sz, i, j, k);
}
// P^T (r - y) at coarse node (I, J, K) of one field (y null: P^T r).
template <typename T>
__host__ __device__ __forceinline__ T restrict_value_nested(const Grid& f, const T* __restrict__ r,
                                                            const T* __restrict__ y, int I, int J, int K) {
  const int64_t sy = f.nx + 1, sz = int64_t(f.nx + 1) * (f.ny + 1);
  T acc = T(0);
#pragma unroll
  for (int dk = -1; dk <= 1; ++dk) {
    const int k = 2 * K + dk;
    if (k < 0 || k > f.nz) continue;
    T sj = T(0);
#pragma unroll
    for (int dj = -1; dj <= 1; ++dj) {
      const int j = 2 * J + dj;
      if (j < 0 || j > f.ny) continue;
      const int64_t o = j * sy + k * sz + 2 * I;
      auto at = [&](int64_t m) { return y ? r[m] - y[m] : r[m]; };
      T si = at(o);
      if (I > 0) si += T(0.5) * at(o - 1);
      if (2 * I + 1 <= f.nx) si += T(0.5) * at(o + 1);
      sj += (dj ? T(0.5) : T(1)) * si;
    }
    acc += (dk ? T(0.5) : T(1)) * sj;
  }
  return acc;
}

// (node, field) fld of fine node (i, j, k): xf += P xc if it is free; of coarse node
// (I, J, K): rc = P^T (rf - y), zero if prescribed.
template <typename T>
__host__ __device__ __forceinline__ void prolong_entry_nested(const Grid& f, const Grid& c, const T* __restrict__ xc,
                                                              const dmask_t* __restrict__ mf, T* __restrict__ xf,
                                                              int fld, int i, int j, int k) {
  const int64_t node = i + int64_t(f.nx + 1) * (j + int64_t(f.ny + 1) * k);
  if ((mf[node] >> fld) & 1) return;
  xf[fld * f.nn() + node] +=
      prolong_value_nested<T>(xc + fld * c.nn(), c.nx + 1, int64_t(c.nx + 1) * (c.ny + 1), i, j, k);
}
template <typename T>
__host__ __device__ __forceinline__ void restrict_entry_nested(const Grid& f, const Grid& c, const T* __restrict__ rf,
                                                               const T* __restrict__ y, const dmask_t* __restrict__ mc,
                                                               T* __restrict__ rc, int fld, int I, int J, int K) {
  const int64_t node = I + int64_t(c.nx + 1) * (J + int64_t(c.ny + 1) * K), off = fld * f.nn();
  rc[fld * c.nn() + node] =
      ((mc[node] >> fld) & 1) ? T(0) : restrict_value_nested<T>(f, rf + off, y ? y + off : nullptr, I, J, K);
}
// every field of one node
template <typename T>
__host__ __device__ __forceinline__ void prolong_node_nested(const Grid& f, const Grid& c, const T* __restrict__ xc,
                                                    const dmask_t* __restrict__ mf, T* __restrict__ xf, int i,
                                                    int j, int k) {
  for (int fld = 0; fld < NF; ++fld) prolong_entry_nested<T>(f, c, xc, mf, xf, fld, i, j, k);
}
template <typename T>
__host__ __device__ __forceinline__ void restrict_node_nested(const Grid& f, const Grid& c, const T* __restrict__ rf,
                                                     const dmask_t* __restrict__ mc, T* __restrict__ rc, int I,
                                                     int J, int K) {
  for (int fld = 0; fld < NF; ++fld) restrict_entry_nested<T>(f, c, rf, nullptr, mc, rc, fld, I, J, K);
}

inline __host__ __device__ bool nested(const Grid& f, const Grid& c) {
  return f.nx == 2 * c.nx && f.ny == 2 * c.ny && f.nz == 2 * c.nz;
}

// z = D^-1 r at one node, D^-1 packed symmetric.
template <typename T>
__device__ __forceinline__ void dinv_node(int64_t nn, const T* __restrict__ D, const T r[NF], T z[NF], int64_t node) {
#pragma unroll
  for (int f = 0; f < NF; ++f) z[f] = T(0);
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int c = f; c < NF; ++c) {
      const T v = D[bidx(f, c) * nn + node];
      z[f] += v * r[c];
      if (c != f) z[c] += v * r[f];
    }
}

// Chebyshev-accelerated point-block Jacobi at one node (Saad, Iterative
// Methods, Alg. 12.1 applied to D^-1 J), bound by reading D^-1 (NBD entries per
// node) and the vectors. First step: r = b - y (y null: r = b), d = c D^-1 r,
// x = d (zero_x) or x += d. yn (optional): d at prescribed DOFs and 0 elsewhere,
// where the application of J to d starts from; it may be y, whose entries of
// this node have been read by then.
template <typename T>
__device__ __forceinline__ void cheb_first_node(int64_t nn, const T* __restrict__ D, const T* __restrict__ b,
                                                const T* y, T c, bool zero_x, T* __restrict__ r, T* __restrict__ d,
                                                T* __restrict__ x, const dmask_t* __restrict__ mask, T* yn,
                                                int64_t node) {
  T rv[NF], z[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    rv[f] = b[f * nn + node];
    if (y) rv[f] -= y[f * nn + node];
    r[f * nn + node] = rv[f];
  }
  dinv_node<T>(nn, D, rv, z, node);
  const dmask_t dm = yn ? mask[node] : dmask_t(0);
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const T dv = c * z[f];
    d[f * nn + node] = dv;
    x[f * nn + node] = zero_x ? dv : x[f * nn + node] + dv;
    if (yn) yn[f * nn + node] = ((dm >> f) & 1) ? dv : T(0);
  }
}

// Later steps: r -= y; d = a d + c D^-1 r; x += d; yn as above.
template <typename T>
__device__ __forceinline__ void cheb_step_node(int64_t nn, const T* __restrict__ D, const T* y, T a, T c,
                                               T* __restrict__ r, T* __restrict__ d, T* __restrict__ x,
                                               const dmask_t* __restrict__ mask, T* yn, int64_t node) {
  T rv[NF], z[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    rv[f] = r[f * nn + node] - y[f * nn + node];
    r[f * nn + node] = rv[f];
  }
  dinv_node<T>(nn, D, rv, z, node);
  const dmask_t dm = yn ? mask[node] : dmask_t(0);
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const T dv = a * d[f * nn + node] + c * z[f];
    d[f * nn + node] = dv;
    x[f * nn + node] += dv;
    if (yn) yn[f * nn + node] = ((dm >> f) & 1) ? dv : T(0);
  }
}

// Deterministic start value of the power iteration at DOF index i of a level
// with nn nodes: in [-1, 1) from an integer hash of i, zero at Dirichlet DOFs.
__device__ __forceinline__ double power_init_value(int64_t i, int64_t nn, const dmask_t* __restrict__ mask) {
  uint64_t z = uint64_t(i) + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  const double u = double(z >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
  const int f = int(i / nn);
  return ((mask[i % nn] >> f) & 1) ? 0.0 : u;
}

}  // namespace pfm
