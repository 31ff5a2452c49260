// Geometric-multigrid kernels (Sec. 3.4): state injection to coarse levels
// for re-discretisation, trilinear prolongation P and restriction R = P^T
// between nested or non-nested structured grids on the same box, the damped
// point-block Jacobi update, and the dense coarse-level operator with its
// inverse by blocked Gauss-Jordan elimination with partial pivoting.
//
// Grid transfer in 1-D: fine node i sits at coarse coordinate i*nc/nf; with
// i*nc = I0*nf + rem, its interpolation weights are (1 - rem/nf) on coarse
// node I0 and rem/nf on I0+1. All index arithmetic is integer, so P and
// R = P^T use identical weights on nested (nf = 2 nc) and non-nested grids.
#include <algorithm>
#include <type_traits>

#include "coarse_inverse.cuh"
#include "common.cuh"
#include "mg_device.cuh"

namespace pfm {
namespace {

inline unsigned grid_for(int64_t threads, int block) {
  int64_t b = (threads + block - 1) / block;
  return unsigned(b > 0 ? b : 1);
}

// Coarse state = fine Q1 field evaluated at coarse node positions.
__global__ void k_inject_state(Grid f, Grid c, const double* __restrict__ Uf, double* __restrict__ Uc) {
  const int64_t nnc = c.nn();
  for (int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; idx < nnc;
       idx += int64_t(gridDim.x) * blockDim.x)
    inject_node(f, c, Uf, Uc, idx);
}

// Coarse Dirichlet bits = bits of the nearest fine node.
__global__ void k_coarse_mask(Grid f, Grid c, const dmask_t* __restrict__ mf, dmask_t* __restrict__ mc) {
  const int64_t nnc = c.nn();
  for (int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; idx < nnc;
       idx += int64_t(gridDim.x) * blockDim.x) {
    int I = int(idx % (c.nx + 1));
    int J = int((idx / (c.nx + 1)) % (c.ny + 1));
    int K = int(idx / (int64_t(c.nx + 1) * (c.ny + 1)));
    auto nearest = [](int Ic, int nc, int nf) { return int((2LL * Ic * nf + nc) / (2LL * nc)); };
    int i = nearest(I, c.nx, f.nx), j = nearest(J, c.ny, f.ny), k = nearest(K, c.nz, f.nz);
    mc[idx] = mf[i + int64_t(f.nx + 1) * (j + int64_t(f.ny + 1) * k)];
  }
}

// xf += P xc at free fine DOFs.
template <typename T>
__global__ void k_prolong_add(Grid f, Grid c, const T* __restrict__ xc, const dmask_t* __restrict__ mf,
                              T* __restrict__ xf) {
  const int64_t nnf = f.nn();
  for (int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; idx < nnf;
       idx += int64_t(gridDim.x) * blockDim.x)
    prolong_node<T>(f, c, xc, mf, xf, idx);
}

// FP32 vectors between non-nested grids: one thread per (node, field).
__global__ void __launch_bounds__(128) k_prolong_add_int(Grid f, Grid c, const float* __restrict__ xc,
                                                         const dmask_t* __restrict__ mf, float* __restrict__ xf) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx < NF * f.nn()) prolong_entry_int(f, c, xc, mf, xf, idx);
}
__global__ void __launch_bounds__(128) k_restrict_int(Grid f, Grid c, const float* __restrict__ rf,
                                                      const float* __restrict__ y, const dmask_t* __restrict__ mc,
                                                      float* __restrict__ rc) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx < NF * c.nn()) restrict_entry_int(f, c, rf, mc, rc, idx, y);
}

// Nested grids: one thread per (node, field), i and j over a 32 x 4 thread block,
// k and the field over the grid's z dimension (no index division but one by NF
// per block). One thread per node with the fields in a loop took 0.20 ms per
// prolongation and 0.11 ms per restriction (FP32, 129^3 nodes), bound by its
// serial chains of loads; on average over the levels of 128^3 elements 48.5 and 28.5 us,
// now 32.4 and (with the difference r - y formed here) 19.3 us.
template <typename T>
__global__ void __launch_bounds__(128) k_prolong_add_nested(Grid f, Grid c, const T* __restrict__ xc,
                                                            const dmask_t* __restrict__ mf, T* __restrict__ xf) {
  const int i = int(blockIdx.x * 32 + threadIdx.x), j = int(blockIdx.y * 4 + threadIdx.y);
  if (i > f.nx || j > f.ny) return;
  prolong_entry_nested<T>(f, c, xc, mf, xf, int(blockIdx.z) % NF, i, j, int(blockIdx.z) / NF);
}

template <typename T>
__global__ void __launch_bounds__(128) k_restrict_nested(Grid f, Grid c, const T* __restrict__ rf,
                                                         const T* __restrict__ y, const dmask_t* __restrict__ mc,
                                                         T* __restrict__ rc) {
  const int I = int(blockIdx.x * 32 + threadIdx.x), J = int(blockIdx.y * 4 + threadIdx.y);
  if (I > c.nx || J > c.ny) return;
  restrict_entry_nested<T>(f, c, rf, y, mc, rc, int(blockIdx.z) % NF, I, J, int(blockIdx.z) / NF);
}

// rc = P^T (rf - y), zero at coarse Dirichlet DOFs.
template <typename T>
__global__ void k_restrict(Grid f, Grid c, const T* __restrict__ rf, const T* __restrict__ y,
                           const dmask_t* __restrict__ mc, T* __restrict__ rc) {
  const int64_t nnc = c.nn();
  for (int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; idx < nnc;
       idx += int64_t(gridDim.x) * blockDim.x)
    restrict_node<T>(f, c, rf, mc, rc, idx, y);
}

// x += omega D^-1 (b - y) per node (y == nullptr: y = 0).
template <typename T>
__global__ void k_smooth(int64_t nn, const T* __restrict__ D, const T* __restrict__ b,
                         const T* __restrict__ y, T omega, T* __restrict__ x) {
  for (int64_t node = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; node < nn;
       node += int64_t(gridDim.x) * blockDim.x) {
    T r[NF], z[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) r[f] = b[f * nn + node] - (y ? y[f * nn + node] : T(0));
    dinv_node<T>(nn, D, r, z, node);
#pragma unroll
    for (int f = 0; f < NF; ++f) x[f * nn + node] += omega * z[f];
  }
}

// dst = D^-1 src per node.
template <typename T>
__global__ void k_dinv(int64_t nn, const T* __restrict__ D, const T* __restrict__ src, T* __restrict__ dst) {
  for (int64_t node = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; node < nn;
       node += int64_t(gridDim.x) * blockDim.x) {
    T r[NF], z[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) r[f] = src[f * nn + node];
    dinv_node<T>(nn, D, r, z, node);
#pragma unroll
    for (int f = 0; f < NF; ++f) dst[f * nn + node] = z[f];
  }
}

template <typename T>
__global__ void k_sub(int64_t n, const T* __restrict__ b, const T* __restrict__ y, T* __restrict__ r) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    r[i] = b[i] - y[i];
}

// Dense coarse operator K (row-major, leading dimension ld) from the stored
// point Hessians: entry (l, m) of an element's matrix, l = f*8 + a, is
// sum_q w (Bz^T H_q Bz + Bg^T G Bg). One CTA per (element, row field): the
// element's Hessians and the shape functions at the Gauss points are staged in
// shared memory once and every thread forms entries of the 8 rows of that
// field. Bound by the latency of the FP64 pipe on the few CTAs that a coarsest
// level has (64 elements, 72 x 72 entries each); one thread per whole row, as
// an earlier form had it, took 628 us for that level, this form 75 us.
// color < 0: every element, added with atomics; color = 0..7: only the elements
// with (ei & 1) + 2 (ej & 1) + 4 (ek & 1) == color, which share no node, added
// without atomics (eight launches in colour order give a fixed summation order).
template <typename T>
__global__ void __launch_bounds__(192) k_coarse_assemble(Grid g, DevParams P, const T* __restrict__ H,
                                                         double* __restrict__ K, int ld, int color) {
  __shared__ double Hs[8][NH];
  __shared__ double Ns[8][8], dNs[3][8][8];  // [local node][Gauss point]
  const int64_t e = blockIdx.x;
  const int fl = int(blockIdx.y);
  const int64_t ei = e % g.nx, ej = (e / g.nx) % g.ny, ek = e / (int64_t(g.nx) * g.ny);
  if (color >= 0 && int((ei & 1) + 2 * (ej & 1) + 4 * (ek & 1)) != color) return;
  const int64_t nn = g.nn();
  const double w = g.w();
  for (int i = threadIdx.x; i < 8 * NH; i += blockDim.x)
    Hs[i / NH][i % NH] = double(H[hstore_offset<T>(e >> 2, i % NH, int(e & 3) * 8 + i / NH)]);
  if (threadIdx.x < 64) {
    const double ih[3] = {1.0 / g.hx, 1.0 / g.hy, 1.0 / g.hz};
    const int a = int(threadIdx.x) >> 3, q = int(threadIdx.x) & 7;
    double phi[3], dphi[3];
    for (int d = 0; d < 3; ++d) {
      const int ad = (a >> d) & 1, qd = (q >> d) & 1;
      phi[d] = (ad == qd) ? GB : GA;
      dphi[d] = (ad ? 1.0 : -1.0) * ih[d];
    }
    Ns[a][q] = phi[0] * phi[1] * phi[2];
    dNs[0][a][q] = dphi[0] * phi[1] * phi[2];
    dNs[1][a][q] = phi[0] * dphi[1] * phi[2];
    dNs[2][a][q] = phi[0] * phi[1] * dphi[2];
  }
  __syncthreads();
  auto node_of = [&](int a) {
    return (ei + (a & 1)) + int64_t(g.nx + 1) * ((ej + ((a >> 1) & 1)) + int64_t(g.ny + 1) * (ek + (a >> 2)));
  };
  for (int i = threadIdx.x; i < 8 * NED; i += blockDim.x) {
    const int al = i / NED, m = i % NED;
    const int fm = m / 8, am = m % 8;
    double s = 0.0;
    for (int q = 0; q < 8; ++q) {
      // z-rows touched by DOF (f, a): u_i -> 3i+J (dN_J); eta_k -> 9+k (N)
      const double* Hq = Hs[q];
      if (fl < 3 && fm < 3) {
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
          for (int y = 0; y < 3; ++y) {
            const int rl = 3 * fl + x, rm = 3 * fm + y;
            s += dNs[x][al][q] * dNs[y][am][q] * Hq[rl < rm ? hidx(rl, rm) : hidx(rm, rl)];
          }
      } else if (fl < 3) {
#pragma unroll
        for (int x = 0; x < 3; ++x) s += dNs[x][al][q] * Ns[am][q] * Hq[hidx(3 * fl + x, 9 + fm - 3)];
      } else if (fm < 3) {
#pragma unroll
        for (int y = 0; y < 3; ++y) s += Ns[al][q] * dNs[y][am][q] * Hq[hidx(3 * fm + y, 9 + fl - 3)];
      } else {
        const int rl = 9 + fl - 3, rm = 9 + fm - 3;
        s += Ns[al][q] * Ns[am][q] * Hq[rl < rm ? hidx(rl, rm) : hidx(rm, rl)];
        s += (dNs[0][al][q] * dNs[0][am][q] + dNs[1][al][q] * dNs[1][am][q] + dNs[2][al][q] * dNs[2][am][q]) *
             P.G[fl - 3][fm - 3];
      }
    }
    double* out = K + (fl * nn + node_of(al)) * ld + (fm * nn + node_of(am));
    if (color >= 0)
      *out += w * s;
    else
      atomicAdd(out, w * s);
  }
}

// Dirichlet rows/columns -> identity.
__global__ void k_coarse_bc(int n, int64_t nn, const dmask_t* __restrict__ mask, double* __restrict__ K,
                            int ld) {
  const int64_t tid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (tid >= int64_t(n) * n) return;
  const int r = int(tid / n), c = int(tid % n);
  const bool dr = (mask[r % nn] >> (r / nn)) & 1;
  const bool dc = (mask[c % nn] >> (c / nn)) & 1;
  if (dr || dc) K[int64_t(r) * ld + c] = (r == c) ? 1.0 : 0.0;
}

// Blocked Gauss-Jordan inverse (coarse_inverse.cuh): panel by one cluster,
// update of the other columns, and the final row/column permutation.
__global__ void __launch_bounds__(GJ_MAX_THREADS) k_gj_panel(double* __restrict__ M, int n, int k0, int R,
                                                             int* __restrict__ used, int* __restrict__ piv,
                                                             double* __restrict__ W, int* singular) {
  gj_panel(M, n, k0, R, used, piv, W, singular, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(GJ_UPD) k_gj_update(double* __restrict__ M, int n, int k0, const int* __restrict__ used,
                                                  const double* __restrict__ W) {
  gj_update_tile(M, n, k0, used, W, int(blockIdx.y) * GJ_TILE, int(blockIdx.x) * GJ_TILE);
}

// Ainv[k][piv[j]] = M[piv[k]][j]
__global__ void k_gj_extract(const double* __restrict__ M, int n, const int* __restrict__ piv,
                             double* __restrict__ Ainv) {
  const int k = blockIdx.x;
  const double* src = M + int64_t(piv[k]) * n;
  for (int j = threadIdx.x; j < n; j += blockDim.x) Ainv[int64_t(k) * n + piv[j]] = src[j];
}

// x = Ainv b (Ainv dense n x n, row-major).
template <typename T>
__global__ void k_coarse_solve(int n, const double* __restrict__ Ainv, const T* __restrict__ b,
                               T* __restrict__ x) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= n) return;
  const double* row = Ainv + int64_t(warp) * n;
  double s = 0.0;
  for (int c = lane; c < n; c += 32) s += row[c] * double(b[c]);
  for (int m = 16; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
  if (lane == 0) x[warp] = T(s);
}

// Chebyshev-accelerated point-block Jacobi, first and later steps (mg_device.cuh).
// 64 registers (4 CTAs of 256 threads per SM) let a node's 45 + 36 loads be in
// flight together. Against the compiler's own choice (32 registers): V-cycle from
// the binary16 store on 75^3 elements 3.14 against 3.31 ms, FP64 Newton solve on 32^3
// 2 per cent less, but 38.2 against 35.1 us per step on average over the levels
// of 128^3 elements (bound by HBM there, about 470 bytes per node). In FP64 with twelve
// variants a node's blocks are 960 bytes and 64 registers spill: 128 registers there, a
// V-cycle on 24^3 elements 4100 -> 4058 us, on 36^3 10.09 -> 10.06 ms.
template <typename T>
constexpr int cheb_minb() {
  return NV > 6 && sizeof(T) == 8 ? 2 : 4;
}
template <typename T>
__global__ void __launch_bounds__(256, (cheb_minb<T>())) k_cheb_first(int64_t nn, const T* __restrict__ D, const T* __restrict__ b, const T* y, T c, bool zero_x,
                             T* __restrict__ r, T* __restrict__ d, T* __restrict__ x, const dmask_t* __restrict__ mask,
                             T* yn) {
  for (int64_t node = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; node < nn;
       node += int64_t(gridDim.x) * blockDim.x)
    cheb_first_node<T>(nn, D, b, y, c, zero_x, r, d, x, mask, yn, node);
}

template <typename T>
__global__ void __launch_bounds__(256, (cheb_minb<T>())) k_cheb_step(int64_t nn, const T* __restrict__ D, const T* y, T a, T c, T* __restrict__ r,
                            T* __restrict__ d, T* __restrict__ x, const dmask_t* __restrict__ mask, T* yn) {
  for (int64_t node = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; node < nn;
       node += int64_t(gridDim.x) * blockDim.x)
    cheb_step_node<T>(nn, D, y, a, c, r, d, x, mask, yn, node);
}

// Deterministic start vector of the power iteration (power_init_value).
template <typename T>
__global__ void k_power_init(int64_t nn, const dmask_t* __restrict__ mask, T* __restrict__ x) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < NF * nn; i += int64_t(gridDim.x) * blockDim.x)
    x[i] = T(power_init_value(i, nn, mask));
}

// xa = a / sqrt(*dot), xb = b / sqrt(*dot)
template <typename T>
__global__ void k_scale2_inv_sqrt(int64_t n, const T* a, const T* b, const double* __restrict__ dot, T* xa, T* xb) {
  __shared__ T s;  // one FP64 square root and division per block, not per thread
  if (threadIdx.x == 0) s = T(1.0 / sqrt(*dot));
  __syncthreads();
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    xa[i] = a[i] * s;
    xb[i] = b[i] * s;
  }
}

// One Lanczos three-term step with the smoother's blocks: u -= alpha q +
// sqrt(beta2prev) qp, w = D^-1 u, and the block's part of u . w (FP64). One pass
// over the nodes and one launch for what took three (the vectors of a coarse
// level take a few microseconds each, so the launches count).
template <typename T>
__global__ void __launch_bounds__(256) k_lanczos_step(int64_t nn, const T* __restrict__ D, T* __restrict__ u,
                                                      const T* __restrict__ q, const T* __restrict__ qp,
                                                      const double* __restrict__ alpha,
                                                      const double* __restrict__ beta2prev, T* __restrict__ w,
                                                      double* __restrict__ partial) {
  __shared__ T ab[2];  // one FP64 square root per block, not per thread
  if (threadIdx.x == 0) {
    ab[0] = T(*alpha);
    ab[1] = beta2prev ? T(sqrt(*beta2prev)) : T(0);
  }
  __syncthreads();
  const T a = ab[0], b = ab[1];
  double acc = 0.0;
  for (int64_t node = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; node < nn;
       node += int64_t(gridDim.x) * blockDim.x) {
    T r[NF], z[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const int64_t i = f * nn + node;
      r[f] = u[i] - (a * q[i] + (beta2prev ? b * qp[i] : T(0)));
      u[i] = r[f];
    }
    dinv_node<T>(nn, D, r, z, node);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      w[f * nn + node] = z[f];
      acc += double(r[f]) * double(z[f]);
    }
  }
  __shared__ double red[8];
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int m = 0; m < 8; ++m) t += red[m];
    partial[blockIdx.x] = t;
  }
}

}  // namespace

template <typename T>
void launch_lanczos_step(int64_t nn, const T* D, T* u, const T* q, const T* qp, const double* alpha,
                         const double* beta2prev, T* w, double* partial, double* out, cudaStream_t s) {
  // at most 1024 partials, as many as fit the dot products' work array
  const int nb = int(std::min<int64_t>((nn + 255) / 256, 1024));
  k_lanczos_step<T><<<nb, 256, 0, s>>>(nn, D, u, q, qp, alpha, beta2prev, w, partial);
  count_launches(1);
  launch_sum_partials(nb, partial, out, s);
}

template <typename T>
void launch_cheb_first(int64_t nn, const T* D, const T* b, const T* y, T c, bool zero_x, T* r, T* d, T* x,
                       const dmask_t* mask, T* yn, cudaStream_t s) {
  k_cheb_first<T><<<grid_for(nn, 256), 256, 0, s>>>(nn, D, b, y, c, zero_x, r, d, x, mask, yn);
  count_launches(1);
}

template <typename T>
void launch_cheb_step(int64_t nn, const T* D, const T* y, T a, T c, T* r, T* d, T* x, const dmask_t* mask, T* yn,
                      cudaStream_t s) {
  k_cheb_step<T><<<grid_for(nn, 256), 256, 0, s>>>(nn, D, y, a, c, r, d, x, mask, yn);
  count_launches(1);
}

template <typename T>
void launch_dinv(int64_t nn, const T* D, const T* src, T* dst, cudaStream_t s) {
  k_dinv<T><<<grid_for(nn, 256), 256, 0, s>>>(nn, D, src, dst);
  count_launches(1);
}

template <typename T>
void launch_power_init(int64_t nn, const dmask_t* mask, T* x, cudaStream_t s) {
  k_power_init<T><<<grid_for(NF * nn, 256), 256, 0, s>>>(nn, mask, x);
  count_launches(1);
}

template <typename T>
void launch_scale2_inv_sqrt(int64_t n, const T* a, const T* b, const double* dot, T* xa, T* xb, cudaStream_t s) {
  k_scale2_inv_sqrt<T><<<grid_for(n, 256), 256, 0, s>>>(n, a, b, dot, xa, xb);
  count_launches(1);
}

void launch_inject_state(const Grid& fine, const Grid& coarse, const double* Uf, double* Uc,
                         cudaStream_t s) {
  k_inject_state<<<grid_for(coarse.nn(), 128), 128, 0, s>>>(fine, coarse, Uf, Uc);
  count_launches(1);
}

void launch_coarse_mask(const Grid& fine, const Grid& coarse, const dmask_t* mf, dmask_t* mc,
                        cudaStream_t s) {
  k_coarse_mask<<<grid_for(coarse.nn(), 128), 128, 0, s>>>(fine, coarse, mf, mc);
  count_launches(1);
}

// y and z node counts within the grid-dimension limit of a 3-D launch
inline bool grid3_ok(const Grid& g) { return (g.ny + 4) / 4 <= 65535 && (int64_t(g.nz) + 1) * NF <= 65535; }
inline dim3 grid3(const Grid& g) {
  return dim3(unsigned((g.nx + 1 + 31) / 32), unsigned((g.ny + 1 + 3) / 4), unsigned((g.nz + 1) * NF));
}

template <typename T>
void launch_prolong_add(const Grid& fine, const Grid& coarse, const T* xc, const dmask_t* mf, T* xf,
                        cudaStream_t s) {
  if (nested(fine, coarse) && grid3_ok(fine)) {
    k_prolong_add_nested<T><<<grid3(fine), dim3(32, 4), 0, s>>>(fine, coarse, xc, mf, xf);
    count_launches(1);
    return;
  }
  if constexpr (std::is_same<T, float>::value) {
    if (transfer_integer(fine)) {
      k_prolong_add_int<<<grid_for(NF * fine.nn(), 128), 128, 0, s>>>(fine, coarse, xc, mf, xf);
      count_launches(1);
      return;
    }
  }
  k_prolong_add<T><<<grid_for(fine.nn(), 256), 256, 0, s>>>(fine, coarse, xc, mf, xf);
  count_launches(1);
}

template <typename T>
void launch_restrict(const Grid& fine, const Grid& coarse, const T* rf, const T* y, const dmask_t* mc, T* rc,
                     cudaStream_t s) {
  if (nested(fine, coarse) && grid3_ok(coarse)) {
    k_restrict_nested<T><<<grid3(coarse), dim3(32, 4), 0, s>>>(fine, coarse, rf, y, mc, rc);
    count_launches(1);
    return;
  }
  if constexpr (std::is_same<T, float>::value) {
    if (transfer_integer(fine)) {
      k_restrict_int<<<grid_for(NF * coarse.nn(), 128), 128, 0, s>>>(fine, coarse, rf, y, mc, rc);
      count_launches(1);
      return;
    }
  }
  k_restrict<T><<<grid_for(coarse.nn(), 128), 128, 0, s>>>(fine, coarse, rf, y, mc, rc);
  count_launches(1);
}

template <typename T>
void launch_smooth(int64_t nn, const T* D, const T* b, const T* y, T omega, T* x, cudaStream_t s) {
  k_smooth<T><<<grid_for(nn, 256), 256, 0, s>>>(nn, D, b, y, omega, x);
  count_launches(1);
}

template <typename T>
void launch_sub(int64_t n, const T* b, const T* y, T* r, cudaStream_t s) {
  k_sub<T><<<grid_for(n, 256), 256, 0, s>>>(n, b, y, r);
  count_launches(1);
}

template <typename T>
void launch_coarse_assemble(const Grid& g, const DevParams& P, const T* H, const dmask_t* mask,
                            double* K, int ld, cudaStream_t s, bool det) {
  const int n = int(NF * g.nn());
  cudaMemsetAsync(K, 0, sizeof(double) * size_t(n) * ld, s);
  for (int c = det ? 0 : -1; c < (det ? 8 : 0); ++c) {
    k_coarse_assemble<T><<<dim3(unsigned(g.ne()), NF), 192, 0, s>>>(g, P, H, K, ld, c);
    count_launches(1);
  }
  k_coarse_bc<<<grid_for(int64_t(n) * n, 256), 256, 0, s>>>(n, g.nn(), mask, K, ld);
  count_launches(1);
}

// Invert the dense coarse operator M (n x n, overwritten; followed by GJ_NB * n
// doubles of work) into Ainv (n x n). used, piv: n integers of work each.
// One panel and one update per GJ_NB columns. Measured at n = 1125 (the 4^3
// coarsest level): 71 panels of 60 us and 71 updates of 27 us, 6.2 ms; one
// launch per column over the augmented matrix took 15.2 ms.
void launch_coarse_inverse(double* M, int n, double* Ainv, int* used, int* piv, int* singular, cudaStream_t s) {
  double* W = M + int64_t(n) * n;
  cudaMemsetAsync(used, 0, sizeof(int) * n, s);
  cudaMemsetAsync(piv, 0, sizeof(int) * n, s);  // in range also where a singular column leaves it unset
  const GjShape sh = gj_shape(n);
  const unsigned tiles = unsigned((n + GJ_TILE - 1) / GJ_TILE);
  for (int k0 = 0; k0 < n; k0 += GJ_NB) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at = {};
    gj_panel_config(sh, 1, s, &cfg, &at);
    cudaLaunchKernelEx(&cfg, k_gj_panel, M, n, k0, sh.rows, used, piv, W, singular);
    k_gj_update<<<dim3(tiles, tiles), GJ_UPD, 0, s>>>(M, n, k0, used, W);
    count_launches(2);
  }
  k_gj_extract<<<n, 256, 0, s>>>(M, n, piv, Ainv);
  count_launches(1);
}

template <typename T>
void launch_coarse_solve(int n, const double* Ainv, const T* b, T* x, cudaStream_t s) {
  k_coarse_solve<T><<<grid_for(int64_t(n) * 32, 256), 256, 0, s>>>(n, Ainv, b, x);
  count_launches(1);
}

#define PFM_INST(T)                                                                              \
  template void launch_prolong_add<T>(const Grid&, const Grid&, const T*, const dmask_t*, T*,     \
                                      cudaStream_t);                                            \
  template void launch_restrict<T>(const Grid&, const Grid&, const T*, const T*, const dmask_t*, T*, \
                                   cudaStream_t);                                               \
  template void launch_smooth<T>(int64_t, const T*, const T*, const T*, T, T*, cudaStream_t);     \
  template void launch_sub<T>(int64_t, const T*, const T*, T*, cudaStream_t);                     \
  template void launch_coarse_assemble<T>(const Grid&, const DevParams&, const T*, const dmask_t*, \
                                          double*, int, cudaStream_t, bool);                    \
  template void launch_coarse_solve<T>(int, const double*, const T*, T*, cudaStream_t);         \
  template void launch_cheb_first<T>(int64_t, const T*, const T*, const T*, T, bool, T*, T*, T*,   \
                                     const dmask_t*, T*, cudaStream_t);                         \
  template void launch_cheb_step<T>(int64_t, const T*, const T*, T, T, T*, T*, T*, const dmask_t*, T*, \
                                    cudaStream_t);                                              \
  template void launch_dinv<T>(int64_t, const T*, const T*, T*, cudaStream_t);                  \
  template void launch_power_init<T>(int64_t, const dmask_t*, T*, cudaStream_t);                  \
  template void launch_scale2_inv_sqrt<T>(int64_t, const T*, const T*, const double*, T*, T*, cudaStream_t); \
  template void launch_lanczos_step<T>(int64_t, const T*, T*, const T*, const T*, const double*,  \
                                       const double*, T*, double*, double*, cudaStream_t);
PFM_INST(float)
PFM_INST(double)
#undef PFM_INST

}  // namespace pfm
