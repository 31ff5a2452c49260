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
// What bounds it: n^3 multiply-adds in the updates (in fixed point on the integer
// pipe; 0.53e12 per second on the FP64 pipe, 2.7 ms at n = 1125) and, in the panel,
// one exchange of pivot candidates per column. The panel runs on one cluster of up to 8 CTAs with
// one row per thread, the row's nb entries in registers; per column every CTA
// sends its best candidate (value, row and the row scaled by the pivot) to all
// CTAs through distributed shared memory and one cluster barrier follows, so a
// column costs about 4 microseconds of latency and no launch (times at
// launch_coarse_inverse).
#pragma once

#include <cooperative_groups.h>

#include <cstdint>

#include "common.cuh"
#include "fixed_point.cuh"

namespace pfm {

constexpr int GJ_NB = 16;        // columns per panel
static_assert(GJ_NB <= FX_TERMS, "the update sums GJ_NB fixed-point products");
constexpr int GJ_MAX_CLUSTER = 8;  // CTAs per panel (the portable cluster size)
constexpr int GJ_MAX_THREADS = 640;  // rows per CTA: 8 x 640 covers MAX_COARSE_DOFS
constexpr int GJ_TILE = 32;      // update: 32 x 32 entries per CTA of GJ_UPD threads
constexpr int GJ_UPD = 128;

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

// Update of one 32 x 32 tile (rows r0.., columns c0..) by 128 threads, 4 x 2
// entries each. The FP64 form is bound by the FP64 pipe (16 multiply-adds per
// entry, 42.6 us per step at n = 1125), so the sum over the nb pivot rows is formed
// in fixed point (fixed_point.cuh): with g_k the exponent of W's row k in the tile,
// T[i][k] 2^(g_k) relative to its largest in row i and W[k][j] 2^(-g_k) relative to
// its largest in column j, 48 integer multiply-adds and one FP64 add per entry
// (26.8 us). Tiles with a non-finite entry or an exponent out of range take
// the FP64 sums.
__device__ __forceinline__ void gj_update_tile(double* __restrict__ M, int n, int k0, const int* __restrict__ used,
                                               const double* __restrict__ W, int r0, int c0) {
  __shared__ uint64_t Ts[GJ_TILE][GJ_NB + 1];  // bits of the numbers, then their limbs
  __shared__ uint64_t Ws[GJ_NB][GJ_TILE];
  __shared__ int gam[GJ_NB], al[GJ_TILE], be[GJ_TILE];
  const int tid = int(threadIdx.x);
  const int nb = n - k0 < GJ_NB ? n - k0 : GJ_NB;
  for (int i = tid; i < GJ_TILE * GJ_NB; i += GJ_UPD) {
    const int r = i / GJ_NB, k = i % GJ_NB;
    Ts[r][k] = fx_bits(r0 + r < n && k < nb ? M[int64_t(r0 + r) * n + k0 + k] : 0.0);
    const int kw = i / GJ_TILE, c = i % GJ_TILE;
    const int col = c0 + c;
    Ws[kw][c] = fx_bits(col < n && kw < nb && (col < k0 || col >= k0 + nb) ? W[int64_t(kw) * n + col] : 0.0);
  }
  const int tx = tid & 15, ty = tid >> 4;
  double acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    const int u = r < n ? used[r] - 1 : -1;
    const bool keep = r < n && !(u >= k0 && u < k0 + nb);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c = c0 + tx + 16 * q;
      acc[i][q] = keep && c < n ? M[int64_t(r) * n + c] : 0.0;
    }
  }
  __syncthreads();
  bool bad = false;
  {  // exponents of the rows of W: eight threads per row
    const int k = tid >> 3;
    unsigned top = 0;
#pragma unroll
    for (int c = 0; c < GJ_TILE / 8; ++c) {
      const unsigned t = fx_top(fx_from_bits(Ws[k][(tid & 7) + 8 * c]));
      top = t > top ? t : top;
    }
#pragma unroll
    for (int m = 1; m <= 4; m <<= 1) {
      const unsigned o = __shfl_xor_sync(0xffffffffu, top, m);
      top = o > top ? o : top;
    }
    const int e = int(top >> 20);
    const int g = e ? e - 1022 : 0;
    bad = e == 0x7ff || g < -FX_RANGE || g > FX_RANGE;
    if ((tid & 7) == 0) gam[k] = g;
  }
  __syncthreads();
  {  // of the rows of T (t < 32) and the columns of W: two threads each
    const int t = tid >> 1;
    const bool row = t < GJ_TILE;
    int x = -4 * FX_RANGE;
#pragma unroll
    for (int h = 0; h < GJ_NB / 2; ++h) {
      const int k = 2 * h + (tid & 1);
      const int e = int(fx_top(fx_from_bits(row ? Ts[t & 31][k] : Ws[k][t & 31])) >> 20);
      const int v = e - 1022 + (row ? gam[k] : -gam[k]);
      if (e && v > x) x = v;
      bad |= e == 0x7ff;
    }
    const int o = __shfl_xor_sync(0xffffffffu, x, 1);
    x = o > x ? o : x;
    if (x == -4 * FX_RANGE)
      x = 0;  // all zero
    else
      bad |= x < -FX_RANGE || x > FX_RANGE;
    if ((tid & 1) == 0) (row ? al : be)[t & 31] = x;
  }
  if (__syncthreads_or(bad)) {
#pragma unroll 1
    for (int k = 0; k < GJ_NB; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 2; ++q)
          acc[i][q] += fx_from_bits(Ts[ty + 8 * i][k]) * fx_from_bits(Ws[k][tx + 16 * q]);
  } else {
    auto limbs = [](uint64_t& x, int k) {
      int x1, x0;
      fx_limbs(fx_from_bits(x), k, x1, x0);
      x = (uint64_t(unsigned(x1)) << 32) | unsigned(x0);
    };
    for (int i = tid; i < GJ_TILE * GJ_NB; i += GJ_UPD) {
      const int r = i / GJ_NB, k = i % GJ_NB;
      limbs(Ts[r][k], 1027 + al[r] - gam[k]);
      const int kw = i / GJ_TILE, c = i % GJ_TILE;
      limbs(Ws[kw][c], 1027 + be[c] + gam[kw]);
    }
    __syncthreads();
    int64_t s1[4][2], s0[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q) s1[i][q] = s0[i][q] = 0;
#pragma unroll 4
    for (int k = 0; k < GJ_NB; ++k) {
      uint64_t t[4], w[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) t[i] = Ts[ty + 8 * i][k];
#pragma unroll
      for (int q = 0; q < 2; ++q) w[q] = Ws[k][tx + 16 * q];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 2; ++q)
          fx_mad(s1[i][q], s0[i][q], int(t[i] >> 32), int(unsigned(t[i])), int(w[q] >> 32), int(unsigned(w[q])));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int q = 0; q < 2; ++q)
        acc[i][q] += fx_value(s1[i][q], s0[i][q], 1027 + al[ty + 8 * i] + be[tx + 16 * q]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i;
    if (r >= n) continue;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c = c0 + tx + 16 * q;
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
