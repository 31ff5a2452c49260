// Inverse of the dense coarse operator by blocked Gauss-Jordan elimination,
// in place and with partial pivoting, shared by the single-problem kernels
// (mg_kernels.cu) and the batched ones (batch.cu).
//
// Scalar form: eliminating column k with pivot row p solves equation p for
// unknown k, so afterwards row p expresses x_k and column k holds the
// coefficients of b_p. The row permutation stays implicit: once every column
// has had its pivot, x_k = sum_j M[p_k][j] b_{p_j}, i.e.
// Ainv[k][p_j] = M[p_k][j]. Pivots are the largest |entry| of the column over
// the rows not used yet (ties: the lowest row).
//
// Blocked form, GJ_NB columns K = [k0, k0 + nb) per step:
//  * panel: the scalar steps applied to the columns of K only (every row).
//    This leaves T = M[:, K] with T[i] the coefficients that row i takes of the
//    nb pivot rows, and the pivot rows' other columns are saved as W.
//  * update of the other columns J: M[i, J] = (i a pivot row of this panel ? 0
//    : M[i, J]) + sum_j T[i][j] W[j, J].
//
// What bounds it: n^3 FP64 multiply-adds in the updates (0.53e12 per second on
// this chip: 2.7 ms at n = 1125) and, in the panel, one exchange of pivot
// candidates per column. The panel runs on one cluster of up to 8 CTAs with
// one row per thread, the row's nb entries in registers; per column every CTA
// sends its best candidate (value, row and the row scaled by the pivot) to all
// CTAs through distributed shared memory and one cluster barrier follows, so a
// column costs about 4 microseconds of latency and no launch (times at
// launch_coarse_inverse).
#pragma once

#include <cooperative_groups.h>

#include <cstdint>

#include "common.cuh"

namespace pfm {

constexpr int GJ_NB = 16;        // columns per panel
constexpr int GJ_MAX_CLUSTER = 8;  // CTAs per panel (the portable cluster size)
constexpr int GJ_MAX_THREADS = 640;  // rows per CTA: 8 x 640 covers MAX_COARSE_DOFS
constexpr int GJ_TILE = 32;      // update: 32 x 32 entries per CTA of 64 threads

// A CTA's pivot candidate: row (scaled by the pivot, with 1 / pivot in the
// pivot's own column), pivot value, search key and row index (-1: no row left).
struct GjCandidate {
  double row[GJ_NB];
  double pivot;
  unsigned long long key;
  int r, pad;
};

// Search key of an entry: the bits of |v| (non-negative FP64 numbers order as
// their bit patterns, a NaN above everything) plus one; 0 stands for no row.
// Integer compares: an FP64 compare would wait for the FP64 pipe.
__device__ __forceinline__ unsigned long long gj_key(double v) {
  return (static_cast<unsigned long long>(__double_as_longlong(v)) & 0x7fffffffffffffffull) + 1ull;
}

// Largest key of the warp with its index (ties: the lowest index).
__device__ __forceinline__ void gj_best(unsigned long long& key, int& r) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) {
    const unsigned long long ok = __shfl_xor_sync(0xffffffffu, key, m);
    const int orow = __shfl_xor_sync(0xffffffffu, r, m);
    if (ok > key || (ok == key && orow < r)) {
      key = ok;
      r = orow;
    }
  }
}

// Panel step (see above) by one cluster of `csize` CTAs, this CTA of rank
// `rank`; R = rows per CTA (<= blockDim.x). used[row] = 1 + the column the row
// was the pivot of (0: not yet). A column without a non-zero pivot sets
// *singular and ends the step (every CTA takes the same decision).
__device__ __forceinline__ void gj_panel(double* __restrict__ M, int n, int k0, int R, int* __restrict__ used,
                                         int* __restrict__ piv, double* __restrict__ W, int* singular, unsigned rank,
                                         unsigned csize) {
  namespace cg = cooperative_groups;
  __shared__ GjCandidate mail[2][GJ_MAX_CLUSTER];
  __shared__ unsigned long long wkey[GJ_MAX_THREADS / 32];
  __shared__ int wrow[GJ_MAX_THREADS / 32];
  __shared__ int prow[GJ_NB];
  cg::cluster_group cl = cg::this_cluster();
  const int tid = int(threadIdx.x), lane = tid & 31, wid = tid >> 5, nwarp = int(blockDim.x) >> 5;
  const int row = int(rank) * R + tid;
  const bool mine = tid < R && row < n;
  const int nb = n - k0 < GJ_NB ? n - k0 : GJ_NB;
  double* Mr = M + int64_t(row) * n + k0;
  double a[GJ_NB];
#pragma unroll
  for (int c = 0; c < GJ_NB; ++c) a[c] = mine && c < nb ? Mr[c] : 0.0;
  int u = mine ? used[row] : 1;
  cl.sync();  // every CTA of the cluster has started: its mailboxes may be written
#pragma unroll
  for (int j = 0; j < GJ_NB; ++j) {
    if (j >= nb) break;
    // best row of the CTA
    unsigned long long key = u == 0 ? gj_key(a[j]) : 0ull;
    int r = row;
    gj_best(key, r);
    if (lane == 0) {
      wkey[wid] = key;
      wrow[wid] = r;
    }
    __syncthreads();
    unsigned long long bk = lane < nwarp ? wkey[lane] : 0ull;
    int br = lane < nwarp ? wrow[lane] : 0;
    gj_best(bk, br);
    // the warp that holds it sends the candidate to every CTA
    const int owner = bk == 0 ? 0 : br - int(rank) * R;
    if (wid == (owner >> 5)) {
      const int src = owner & 31;
      const double pv = __shfl_sync(0xffffffffu, a[j], src);
      const double ip = 1.0 / pv;
      double val = 1.0;
#pragma unroll
      for (int c = 0; c < GJ_NB; ++c) {
        const double x = __shfl_sync(0xffffffffu, a[c], src);
        if (lane == c && c != j) val = x;
      }
      val *= ip;
      for (unsigned t = 0; t < csize; ++t) {
        GjCandidate* m = cl.map_shared_rank(&mail[j & 1][rank], t);
        if (lane < GJ_NB) m->row[lane] = val;
        if (lane == GJ_NB) m->pivot = pv;
        if (lane == GJ_NB + 1) m->key = bk;
        if (lane == GJ_NB + 2) m->r = br;
      }
    }
    cl.sync();
    // the same choice in every CTA
    unsigned long long mk = lane < int(csize) ? mail[j & 1][lane].key : 0ull;
    int best = lane;
    gj_best(mk, best);
    const GjCandidate& p = mail[j & 1][best];
    if (p.key == 0 || !(fabs(p.pivot) > 0.0)) {
      if (rank == 0 && tid == 0) *singular = 1;
      return;  // no CTA writes another's shared memory after this barrier
    }
    if (tid == 0) prow[j] = p.r;
    if (mine) {
      if (row == p.r) {
#pragma unroll
        for (int c = 0; c < GJ_NB; ++c) a[c] = p.row[c];
        u = k0 + j + 1;
      } else {
        const double f = a[j];
        a[j] = 0.0;
#pragma unroll
        for (int c = 0; c < GJ_NB; ++c) a[c] -= f * p.row[c];
      }
    }
  }
  if (mine) {
#pragma unroll
    for (int c = 0; c < GJ_NB; ++c)
      if (c < nb) Mr[c] = a[c];
    used[row] = u;
  }
  __syncthreads();
  if (rank == 0 && tid < nb) piv[k0 + tid] = prow[tid];
  const int64_t step = int64_t(csize) * blockDim.x;
  for (int j = 0; j < nb; ++j) {
    const double* src = M + int64_t(prow[j]) * n;
    double* dst = W + int64_t(j) * n;
    for (int64_t c = int64_t(rank) * blockDim.x + tid; c < n; c += step)
      if (c < k0 || c >= k0 + nb) dst[c] = src[c];
  }
}

// Update of one 32 x 32 tile (rows r0.., columns c0..) by 64 threads, 4 x 4
// entries each.
__device__ __forceinline__ void gj_update_tile(double* __restrict__ M, int n, int k0, const int* __restrict__ used,
                                               const double* __restrict__ W, int r0, int c0) {
  __shared__ double Ts[GJ_TILE][GJ_NB + 1];
  __shared__ double Ws[GJ_NB][GJ_TILE];
  const int tid = int(threadIdx.x);
  const int nb = n - k0 < GJ_NB ? n - k0 : GJ_NB;
  for (int i = tid; i < GJ_TILE * GJ_NB; i += 64) {
    const int r = i / GJ_NB, k = i % GJ_NB;
    Ts[r][k] = r0 + r < n && k < nb ? M[int64_t(r0 + r) * n + k0 + k] : 0.0;
    const int kw = i / GJ_TILE, c = i % GJ_TILE;
    const int col = c0 + c;
    Ws[kw][c] = col < n && kw < nb && (col < k0 || col >= k0 + nb) ? W[int64_t(kw) * n + col] : 0.0;
  }
  const int tx = tid & 7, ty = tid >> 3;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    const int u = r < n ? used[r] - 1 : -1;
    const bool keep = r < n && !(u >= k0 && u < k0 + nb);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = c0 + tx + 8 * q;
      acc[i][q] = keep && c < n ? M[int64_t(r) * n + c] : 0.0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < GJ_NB; ++k) {
    double t[4], w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      t[i] = Ts[ty + 8 * i][k];
      w[i] = Ws[k][tx + 8 * i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][q] += t[i] * w[q];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    if (r >= n) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = c0 + tx + 8 * q;
      if (c < n && (c < k0 || c >= k0 + nb)) M[int64_t(r) * n + c] = acc[i][q];
    }
  }
}

// CTAs per panel and threads per CTA for the largest order n of a launch: about
// 128 rows per CTA, so that a CTA's FP64 pipe (2 multiply-adds per clock) takes
// about as long for a column as the exchange of candidates does.
struct GjShape {
  int cluster, threads, rows;
};
inline GjShape gj_shape(int n) {
  int c = 1;
  while (c < GJ_MAX_CLUSTER && n > 128 * c) c *= 2;
  const int rows = (n + c - 1) / c;
  return {c, (rows + 31) / 32 * 32, rows};
}
// launch configuration of a panel: one cluster per problem (blockIdx.y)
inline void gj_panel_config(const GjShape& sh, int problems, cudaStream_t s, cudaLaunchConfig_t* cfg,
                            cudaLaunchAttribute* at) {
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = unsigned(sh.cluster);
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg->gridDim = dim3(unsigned(sh.cluster), unsigned(problems));
  cfg->blockDim = dim3(unsigned(sh.threads));
  cfg->stream = s;
  cfg->attrs = at;
  cfg->numAttrs = 1;
}

}  // namespace pfm
