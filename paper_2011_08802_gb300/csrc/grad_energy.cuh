// Gradient part of the interface energy (Eq. IntEnergy) as an operator on the
// nodes. Its element contribution, sum_d G int d_d N_a d_d N_b, is constant, and
// the 2-point rule integrates products of trilinear gradients exactly, so
// assembled on the structured grid it is G times the sum over the axes of
// tensor products of the 1-D stiffness and mass matrices:
//   (K x)_i = (n_i x_i - s_i)/h,  (M x)_i = (2 n_i x_i + s_i) h/6,
// s_i = x_(i-1) + x_(i+1) over the neighbours that exist and n_i their number
// of adjacent elements (2 inside, 1 at an end). One node costs 27 values and
// about 35 operations per order parameter; inside the element kernels the same
// term took, for each of the 8 (element, node) pairs of a node, the gradients of
// every order parameter at the Gauss points, the product with G and their
// scatter (about 0.4 of the FP64 operations and 0.6 of the shuffles of an
// application). Only displacements may be prescribed, so no row or column of
// this operator is masked. Used where the element kernel is bound by
// arithmetic (FP64 and double-float applications, residual); the applications
// in FP32 arithmetic keep the term in their element kernel: from the FP32 store
// they are bound by reading it, and from the binary16 store the extra pass cost
// more than it saved (V-cycle on 75^3 elements 4.9 -> 5.2 ms).
// Measured: FP64 application of 61x45x33 elements 982 -> 615 us, double-float of
// 93x77x61 1629 -> 1040 us.
//
// One thread takes GE_Z nodes above one another for one order parameter (two
// planes more than it writes: 1.5 plane passes per node); a block holds 32 such
// columns times all order parameters and exchanges the operator's values through
// shared memory for the product with G. One thread per column for all of them
// needed no exchange but left a chain of NV x 6 planes per thread: 27 us at 33^3
// nodes in FP64 and slower V-cycles on small levels; 14 us in this form.
#pragma once

#include <cstdint>
#include <type_traits>

#include "common.cuh"

namespace pfm {

constexpr int GE_Z = 4;

template <typename TA>
struct GradE {
  TA G[NV][NV];
  TA cx, cy, cz;  // hy hz/(36 hx) and so on
};
template <typename TA>
inline void grad_energy_const(const Grid& g, const DevParams& P, GradE<TA>& c) {
  for (int k = 0; k < NV; ++k)
    for (int l = 0; l < NV; ++l) c.G[k][l] = TA(P.G[k][l]);
  c.cx = TA(g.hy * g.hz / (36.0 * g.hx));
  c.cy = TA(g.hx * g.hz / (36.0 * g.hy));
  c.cz = TA(g.hx * g.hy / (36.0 * g.hz));
}
// (hi, lo) form of the constants for the double-float kernels
struct GradEDf {
  float2 G[NV][NV];
  float2 cx, cy, cz;
};
inline float2 ge_split(double x) {
  const float hi = float(x);
  return make_float2(hi, float(x - double(hi)));
}
inline void grad_energy_const(const Grid& g, const DevParams& P, GradEDf& c) {
  for (int k = 0; k < NV; ++k)
    for (int l = 0; l < NV; ++l) c.G[k][l] = ge_split(P.G[k][l]);
  c.cx = ge_split(g.hy * g.hz / (36.0 * g.hx));
  c.cy = ge_split(g.hx * g.hz / (36.0 * g.hy));
  c.cz = ge_split(g.hx * g.hy / (36.0 * g.hz));
}

// arithmetic of the kernels: FP32, FP64 or double-float
template <typename TA>
struct GeArith {
  using C = GradE<TA>;
  template <typename TV>
  static __device__ __forceinline__ TA load(TV x) { return TA(x); }
  static __device__ __forceinline__ TA constant(TA x) { return x; }
  // n x + s with n = 1, 2 or 4
  static __device__ __forceinline__ TA scaled(float n, TA x, TA s) { return TA(n) * x + s; }
  static __device__ __forceinline__ double out(TA x) { return double(x); }
};
template <>
struct GeArith<df64> {
  using C = GradEDf;
  template <typename TV>
  static __device__ __forceinline__ df64 load(TV x) {
    static_assert(std::is_same<TV, float>::value, "double-float applications take FP32 vectors");
    return df64::make(x, 0.f);
  }
  static __device__ __forceinline__ df64 constant(float2 x) { return df64::make(x.x, x.y); }
  static __device__ __forceinline__ df64 scaled(float n, df64 x, df64 s) { return df64::make(n * x.hi, n * x.lo) + s; }
  static __device__ __forceinline__ double out(df64 x) { return double(x); }
};

// Columns (i, j, chunk of GE_Z planes) of a grid.
__host__ __device__ inline int64_t grad_energy_columns(const Grid& g) {
  return int64_t(g.nx + 1) * (g.ny + 1) * ((g.nz + 1 + GE_Z - 1) / GE_Z);
}

// How the nodal values are written:
//   GE_APPLY  first pass of a tangent application: displacement rows v at
//             prescribed DOFs (identity rows), 0 elsewhere; order-parameter rows
//             the operator's values (the element kernel adds to them)
//   GE_RES    first pass of a residual: displacement rows 0
//   GE_ADD    the operator's values added to the order-parameter rows (after the
//             node pass of the atomic-free forms, which writes every row)
enum { GE_APPLY = 0, GE_RES = 1, GE_ADD = 2 };

constexpr int GE_COLS = 32;  // columns per block; blockDim = (GE_COLS, NV)

template <typename TA>
struct GradESmem {
  TA L[NV][GE_Z][GE_COLS];
};

// The operator's values L and, up to the factor hx hy hz / 216, the mass matrix's
// values M of one field x (at the column's first node) on the GE_Z nodes of the
// column (i, j, k0).
template <typename TA, typename TV>
__device__ __forceinline__ void grad_energy_operator(const Grid& g, const typename GeArith<TA>::C& c, const TV* x, int i,
                                                     int j, int k0, TA L[GE_Z], TA M[GE_Z]) {
  using Ar = GeArith<TA>;
  const int nxp = g.nx + 1;
  const int64_t plane = int64_t(nxp) * (g.ny + 1);
  const TA zero = TA(0.f);
  const bool xm = i > 0, xp = i < g.nx, ym = j > 0, yp = j < g.ny;
  const float ni = (xm ? 1.f : 0.f) + (xp ? 1.f : 0.f), nj = (ym ? 1.f : 0.f) + (yp ? 1.f : 0.f);
  const TA cx = Ar::constant(c.cx), cy = Ar::constant(c.cy), cz = Ar::constant(c.cz);
  TA mm0 = zero, q0 = zero, mm1 = zero, q1 = zero;  // planes k - 1 and k
#pragma unroll
  for (int p = -1; p <= GE_Z; ++p) {
    TA mm2 = zero, q2 = zero;
    const int k = k0 + p;
    if (k >= 0 && k <= g.nz) {
      // row: Mx = 2 n x + s, Kx = n x - s
      const TV* xr = x + p * plane;
      auto row = [&](const TV* a, TA& M, TA& K) {
        const TA s = (xm ? Ar::load(a[-1]) : zero) + (xp ? Ar::load(a[1]) : zero);
        const TA b = Ar::load(a[0]);
        M = Ar::scaled(2.f * ni, b, s);
        K = Ar::scaled(ni, b, -s);
      };
      TA M0, K0, Ma = zero, Ka = zero, Mb = zero, Kb = zero;
      row(xr, M0, K0);
      if (ym) row(xr - nxp, Ma, Ka);
      if (yp) row(xr + nxp, Mb, Kb);
      const TA sM = Ma + Mb, sK = Ka + Kb;
      mm2 = Ar::scaled(2.f * nj, M0, sM);
      q2 = cx * Ar::scaled(2.f * nj, K0, sK) + cy * Ar::scaled(nj, M0, -sM);
    }
    if (p >= 1) {
      const int kz = k0 + p - 1;
      const float n = (kz > 0 ? 1.f : 0.f) + (kz < g.nz ? 1.f : 0.f);
      L[p - 1] = Ar::scaled(2.f * n, q1, q0 + q2) + cz * Ar::scaled(n, mm1, -(mm0 + mm2));
      M[p - 1] = Ar::scaled(2.f * n, mm1, mm0 + mm2);
    }
    mm0 = mm1;
    q0 = q1;
    mm1 = mm2;
    q1 = q2;
  }
}

// Columns t0 .. t0 + 31 of grid g by one block (GE_COLS, NV); every thread of the
// block calls it. Returns this thread's part of x . (operator x) / 2 (the gradient
// energy) when `energy` is set.
template <typename TA, int MODE, typename TV, typename TY>
__device__ __forceinline__ double grad_energy_block(const Grid& g, const typename GeArith<TA>::C& c,
                                                    const dmask_t* __restrict__ mask, const TV* __restrict__ v,
                                                    TY* __restrict__ y, int64_t t0, int64_t ncol, GradESmem<TA>& sm,
                                                    bool energy) {
  using Ar = GeArith<TA>;
  const int col = int(threadIdx.x), l = int(threadIdx.y);
  const int64_t t = t0 + col;
  const bool on = t < ncol;
  const int nxp = g.nx + 1, nyp = g.ny + 1;
  const int64_t tt = on ? t : 0;
  const int i = int(tt % nxp);
  const int64_t r = tt / nxp;
  const int j = int(r % nyp);
  const int k0 = int(r / nyp) * GE_Z;
  const int64_t nn = g.nn(), plane = int64_t(nxp) * nyp;
  const int64_t node0 = i + int64_t(nxp) * (j + int64_t(nyp) * k0);
  const int nk = !on ? 0 : (g.nz + 1 - k0 < GE_Z ? g.nz + 1 - k0 : GE_Z);
  if (on) {
    TA L[GE_Z], M[GE_Z];
    grad_energy_operator<TA>(g, c, v + (3 + l) * nn + node0, i, j, k0, L, M);
#pragma unroll
    for (int z = 0; z < GE_Z; ++z) sm.L[l][z][col] = L[z];
  }
  __syncthreads();
  double en = 0.0;
  for (int z = 0; z < nk; ++z) {
    const int64_t node = node0 + z * plane;
    if constexpr (MODE != GE_ADD) {
      if (l < 3) {  // displacement row l
        const int64_t idx = l * nn + node;
        if constexpr (MODE == GE_APPLY)
          y[idx] = ((mask[node] >> l) & 1) ? TY(v[idx]) : TY(0);
        else
          y[idx] = TY(0);
      }
    }
    TA acc = Ar::constant(c.G[l][0]) * sm.L[0][z][col];
#pragma unroll
    for (int m = 1; m < NV; ++m) acc += Ar::constant(c.G[l][m]) * sm.L[m][z][col];
    const int64_t idx = (3 + l) * nn + node;
    if (energy) en += double(v[idx]) * Ar::out(acc);
    if constexpr (MODE == GE_ADD)
      y[idx] += TY(Ar::out(acc));
    else if constexpr (std::is_same<TA, TY>::value)
      y[idx] = acc;
    else
      y[idx] = TY(Ar::out(acc));
  }
  return 0.5 * en;
}

}  // namespace pfm
