// dense_inverse.cu -- batched Gauss-Jordan elimination with partial pivoting.
//
// It returns log|det|, the sign and (inverse mode) the inverse in the library's dual-row layout
// Binv[c][k] = (A^-1)[k][c]; "det-only" mode restricts the elimination to the rows not yet
// pivoted and the columns to the right, which is LU with partial pivoting (n^3/3 multiply-adds)
// -- both are the "single LU decomposition" of Sec. II.C giving the determinant and the inverse
// together.
//
// Blocking. Pivots are taken a panel of columns at a time; the elementary row operations of the
// block combine into T = I + U P^T, where the columns of U are the swept panel columns minus
// the unit vectors of the pivot rows and P selects the pivot rows. Every other column then takes
// one update
//     A[i][c] += sum_j U[i][j] A_old[p_j][c]
// so each matrix element is read and written once per block. The matrix stays in global memory
// (L2-resident while the CTAs in flight fit). Up to 1024 rows (k_gj_split) the update runs on the
// 16-bit tensor cores as split products; above, where its panel exceeds shared memory, k_gj takes
// it on the FP64 pipe (8 columns a block, one CTA per matrix; k_gj_cluster eight for the inverses of a list).
//
// Pivot choice: largest |value| among unpivoted rows, ties to the lowest row index.
// Pivoting is implicit (no row swaps); the pivot row of column k is p[k] and the final
// storage holds A^-1[k][p[j]] at (p[k], j).
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>

#include "fp64_mma.cuh"
#include "scale_internal.cuh"

namespace cg = cooperative_groups;

namespace scale {

namespace {

constexpr int kThreads = 1024;  // 32 warps: DFMA latency hidden within one CTA

// Pivot search on integer keys: the bit pattern of |x| orders like |x| (and puts NaN above
// every number), so the search runs on the integer pipe instead of FP64 compares.
template <typename TW>
struct AbsKey;
template <>
struct AbsKey<double> {
  using T = unsigned long long;
  __device__ static T of(double x) { return (T)__double_as_longlong(x) & 0x7fffffffffffffffull; }
};
template <>
struct AbsKey<float> {
  using T = unsigned int;
  __device__ static T of(float x) { return (T)__float_as_uint(x) & 0x7fffffffu; }
};
template <typename K>
__device__ __forceinline__ void key_merge(K& k, int& i, K k2, int i2) {
  if (k2 > k || (k2 == k && i2 < i)) {
    k = k2;
    i = i2;
  }
}

// Largest key over the warp (ties to the lowest row); the result is valid on lane 0.
template <typename K>
__device__ __forceinline__ void warp_key_max(K& k, int& i) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const K k2 = __shfl_down_sync(0xffffffffu, k, off);
    const int i2 = __shfl_down_sync(0xffffffffu, i, off);
    key_merge(k, i, k2, i2);
  }
}

// Pivot row of panel column jj: the largest |value| among the rows not yet pivoted, ties to
// the lowest row. Each thread scans its rows, each warp merges its lanes, and warp 0 merges
// the warps' winners; the row (n if none) is returned on thread 0 only.
template <typename TW, int NT>
__device__ __forceinline__ int pivot_search(const TW* panel, int ldp, int jj, int n, const unsigned char* used,
                                            typename AbsKey<TW>::T* red_k, int* red_i) {
  using KeyT = typename AbsKey<TW>::T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  KeyT bk = 0;
  int bi = n;
  for (int i = tid; i < n; i += NT) {
    if (used[i]) continue;
    key_merge(bk, bi, AbsKey<TW>::of(panel[i * ldp + jj]), i);
  }
  warp_key_max(bk, bi);
  if (lane == 0) {
    red_k[warp] = bk;
    red_i[warp] = bi;
  }
  __syncthreads();
  if (warp == 0) {
    bk = lane < NT / 32 ? red_k[lane] : KeyT(0);
    bi = lane < NT / 32 ? red_i[lane] : n;
    warp_key_max(bk, bi);
  }
  return bi;
}

// log|det| = sum_k log|pivot_k| by warp 0: one log per lane at a time, then a warp tree
// (the result is valid on thread 0).
__device__ __forceinline__ double sum_log_pivots(const double* pabs, int n, bool skip) {
  const int lane = threadIdx.x & 31;
  double part = 0.0;
  if (!skip)
    for (int k = lane; k < n; k += 32) part += log(pabs[k]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) part += __shfl_down_sync(0xffffffffu, part, off);
  return part;
}

// Matrices above 1024 rows, and inverses up to kSmallInverse rows. TW: working precision; TOUT:
// inverse output precision; TH threads per CTA (one matrix).
//
// The FP64 pipe of sm_103a issues one warp-wide DFMA per SM sub-partition about every 64
// cycles, so the serial part of a pivot step (search, reciprocal, log) is kept off it: the
// search compares integer keys, one thread takes the reciprocal and shares it, and the logs
// of the pivots are summed by all threads at the end.
template <typename TW, typename TOUT, bool kInverse, int W, int TH = kThreads>
__global__ void __launch_bounds__(TH) k_gj(TW* __restrict__ mats, int n, const int32_t* __restrict__ list,
                                                 TOUT* __restrict__ binv, double* __restrict__ logabs_out,
                                                 int32_t* __restrict__ sign_out, int32_t* __restrict__ status) {
  static_assert((W & (W - 1)) == 0, "the panel width is a power of two");
  extern __shared__ unsigned char smem_raw[];
  using KeyT = typename AbsKey<TW>::T;
  double* pabs = reinterpret_cast<double*>(smem_raw);  // [n] |pivot| of column k (log taken at the end)
  TW* panel = reinterpret_cast<TW*>(pabs + n);         // [n][W]
  TW* prow = panel + (size_t)n * W;              // [W][n]
  TW* colk = prow + (size_t)W * n;               // [n]
  TW* rowp = colk + n;                           // [W]
  int* piv = reinterpret_cast<int*>(rowp + W);   // [n] pivot row of column k
  int* qinv = piv + n;                           // [n] column whose pivot row is r
  unsigned char* used = reinterpret_cast<unsigned char*>(qinv + n);  // [n]
  __shared__ KeyT red_k[TH / 32];
  __shared__ int red_i[TH / 32];
  __shared__ TW s_inv;
  __shared__ int s_p;
  __shared__ int s_singular;

  const int b = list ? list[blockIdx.x] : blockIdx.x;
  if (b < 0) return;
  TW* A = mats + (size_t)b * n * n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  for (int i = tid; i < n; i += TH) used[i] = 0;
  if (tid == 0) s_singular = 0;
  int sgn = 1;  // kept by thread 0
  __syncthreads();

  for (int K0 = 0; K0 < n; K0 += W) {
    const int w = min(W, n - K0);
    // panel <- columns [K0, K0+w)
    for (int q = tid; q < n * W; q += TH) {
      const int i = q / W, j = q % W;
      if (j < w) panel[q] = A[(size_t)i * n + K0 + j];
    }
    __syncthreads();
    for (int jj = 0; jj < w; ++jj) {
      const int k = K0 + jj;
      const int bi = pivot_search<TW, TH>(panel, W, jj, n, used, red_k, red_i);
      if (tid == 0) {
        if (bi >= n || !(fabs(panel[bi * W + jj]) > TW(0))) {
          s_singular = 1;
        } else {
          const TW pv = panel[bi * W + jj];
          s_inv = TW(1) / pv;
          s_p = bi;
          piv[k] = bi;
          used[bi] = 1;
          pabs[k] = fabs((double)pv);
          if (pv < TW(0)) sgn = -sgn;
        }
      }
      __syncthreads();
      if (s_singular) break;
      const int p = s_p;
      const TW inv = s_inv;
      // snapshot the pivot row (panel part) and column jj before updating
      for (int j = tid; j < w; j += TH) rowp[j] = (j == jj) ? inv : panel[p * W + j] * inv;
      for (int i = tid; i < n; i += TH) colk[i] = panel[i * W + jj];
      __syncthreads();
      for (int q = tid; q < n * W; q += TH) {
        const int i = q / W, j = q % W;
        if (j >= w) continue;
        if (i == p) {
          panel[q] = rowp[j];
        } else if (kInverse || !used[i]) {
          const TW f = colk[i];
          const TW base = (j == jj) ? TW(0) : panel[q];
          panel[q] = base - f * rowp[j];
        }
      }
      __syncthreads();
    }
    if (s_singular) break;
    // old pivot rows of the block (all columns outside the panel)
    for (int q = tid; q < w * n; q += TH) {
      const int j = q / n, c = q - j * n;
      prow[j * n + c] = A[(size_t)piv[K0 + j] * n + c];
    }
    __syncthreads();
    // rank-w update of the columns outside the panel: warp per row, lanes over columns,
    // the row's multipliers u_j = U[i][j] in registers
    const int c_lo = kInverse ? 0 : K0 + w;
    for (int i = warp; i < n; i += TH / 32) {
      if (!kInverse && used[i]) continue;
      TW u[W];
#pragma unroll
      for (int j = 0; j < W; ++j) u[j] = (j < w) ? panel[i * W + j] - ((piv[K0 + j] == i) ? TW(1) : TW(0)) : TW(0);
      TW* Ai = A + (size_t)i * n;
      if constexpr (!kInverse) {
        // determinant only: every column from c_lo on lies right of the panel; one column
        // per lane, so a strip wastes at most 31 lanes
        for (int c = c_lo + lane; c < n; c += 32) {
          TW a1 = Ai[c];
#pragma unroll
          for (int j = 0; j < W; ++j)
            if (j < w) a1 += u[j] * prow[j * n + c];
          Ai[c] = a1;
        }
        continue;
      }
      // inverse: every column; two columns per lane in flight while both lie inside the
      // row, then the odd strip alone (no strip runs with its lanes idle); the panel
      // columns are written back from the panel below
      int c = lane;
      for (; c + 32 < n; c += 64) {
        const int c2 = c + 32;
        const bool in1 = !(c >= K0 && c < K0 + w);
        const bool in2 = !(c2 >= K0 && c2 < K0 + w);
        TW a1 = in1 ? Ai[c] : TW(0);
        TW a2 = in2 ? Ai[c2] : TW(0);
#pragma unroll
        for (int j = 0; j < W; ++j) {
          if (j < w) {
            a1 += u[j] * prow[j * n + c];
            a2 += u[j] * prow[j * n + c2];
          }
        }
        if (in1) Ai[c] = a1;
        if (in2) Ai[c2] = a2;
      }
      if (c < n && !(c >= K0 && c < K0 + w)) {
        TW a1 = Ai[c];
#pragma unroll
        for (int j = 0; j < W; ++j)
          if (j < w) a1 += u[j] * prow[j * n + c];
        Ai[c] = a1;
      }
    }
    // write the swept panel back
    for (int q = tid; q < n * W; q += TH) {
      const int i = q / W, j = q % W;
      if (j < w) A[(size_t)i * n + K0 + j] = panel[q];
    }
    __syncthreads();
  }

  const double logdet = warp == 0 ? sum_log_pivots(pabs, n, s_singular != 0) : 0.0;  // on thread 0
  if (tid == 0) {
    int st = 0;
    double la = logdet;
    int sg = sgn;
    if (s_singular) {
      st = SCALE_SAMPLE_SINGULAR;
      la = -INFINITY;
      sg = 0;
    } else {
      // sign of the permutation k -> piv[k]
      for (int k = 0; k < n; ++k) qinv[k] = 0;
      int parity = 0;
      for (int k = 0; k < n; ++k) {
        if (qinv[k]) continue;
        int j = k, len = 0;
        while (!qinv[j]) {
          qinv[j] = 1;
          j = piv[j];
          ++len;
        }
        parity += len - 1;
      }
      if (parity & 1) sg = -sg;
    }
    if (logabs_out) logabs_out[b] = la;
    if (sign_out) sign_out[b] = sg;
    if (status && st) status[b] |= st;
  }
  if (!kInverse) return;
  __syncthreads();
  if (s_singular) {
    if (binv)
      for (int q = tid; q < n * n; q += TH) binv[(size_t)b * n * n + q] = TOUT(0);
    return;
  }
  for (int k = tid; k < n; k += TH) qinv[piv[k]] = k;
  __syncthreads();
  // Binv[s][cf] = A^-1[cf][s] = A_final[piv[cf]][qinv[s]]
  for (int q = tid; q < n * n; q += TH) {
    const int s = q / n, cf = q - s * n;
    binv[(size_t)b * n * n + q] = (TOUT)A[(size_t)piv[cf] * n + qinv[s]];
  }
}

// Inverse mode split over a thread-block cluster of C CTAs per matrix (FP64 working
// precision). The columns are cut into C contiguous ranges of whole W-column blocks; CTA q
// owns its range, and only it reads or writes those columns of A. For each block the owner
// sweeps the W-column panel in its shared memory exactly as k_gj does; after one cluster
// barrier every CTA copies the swept panel and the block's pivot rows from the owner's
// shared memory (distributed shared memory) and applies the rank-W update to its own
// columns. The panel alternates between two buffers, so the owner of the next block can
// sweep while the others still copy: one cluster barrier per block. A singular panel is told by its
// block's number, as the others may read the word when the owner is already at the next block. Every
// element sees the same operations in the same order as in k_gj, so the two kernels give the same bits;
// the cluster version spreads the O(n^3) FP64 update of one matrix over C SMs, which shortens
// the refresh of a large matrix (the serial panel steps stay on one SM): 3 matrices of 1100 rows
// 348 ms by k_gj, 64 here.
template <typename TOUT, int W, int C>
__global__ void __launch_bounds__(kThreads) k_gj_cluster(double* __restrict__ mats, int n,
                                                         const int32_t* __restrict__ list, TOUT* __restrict__ binv,
                                                         double* __restrict__ logabs_out, int32_t* __restrict__ sign_out,
                                                         int32_t* __restrict__ status) {
  extern __shared__ unsigned char smem_raw[];
  cg::cluster_group cluster = cg::this_cluster();
  const int q = (int)cluster.block_rank();
  const int mat = blockIdx.x / C;
  const int b = list ? list[mat] : mat;
  if (b < 0) return;  // the whole cluster shares mat, so it leaves together
  double* A = mats + (size_t)b * n * n;
  const int nblocks = (n + W - 1) / W;
  const int bpc = (nblocks + C - 1) / C;  // blocks per CTA
  const int c_lo = min(n, q * bpc * W), c_hi = min(n, (q + 1) * bpc * W);
  const int ncol = c_hi - c_lo, ldp = bpc * W;
  double* pabs = reinterpret_cast<double*>(smem_raw);    // [n] |pivot| of the columns this CTA owns
  double* panels = pabs + n;                             // [2][n][W]
  double* prow = panels + (size_t)2 * n * W;             // [W][ldp]
  double* colk = prow + (size_t)W * ldp;                 // [n]
  double* rowp = colk + n;                               // [W]
  int* piv = reinterpret_cast<int*>(rowp + W);           // [n]
  int* qinv = piv + n;                                   // [n]
  unsigned char* used = reinterpret_cast<unsigned char*>(qinv + n);  // [n]
  __shared__ unsigned long long red_k[kThreads / 32];
  __shared__ int red_i[kThreads / 32];
  __shared__ double s_inv;
  __shared__ int s_p;
  __shared__ int s_singular;  // block whose panel is singular (INT_MAX: none)
  __shared__ int s_sgn;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < n; i += kThreads) used[i] = 0;
  if (tid == 0) {
    s_singular = INT_MAX;
    s_sgn = 1;
  }
  __syncthreads();
  cluster.sync();  // every CTA of the cluster runs before any reads another's shared memory

  bool singular = false;
  for (int blk = 0; blk < nblocks; ++blk) {
    const int K0 = blk * W, w = min(W, n - K0);
    const int owner = blk / bpc;
    double* panel = panels + (size_t)(blk & 1) * n * W;
    if (q == owner) {
      for (int e = tid; e < n * W; e += kThreads) {
        const int i = e / W, j = e % W;
        if (j < w) panel[e] = A[(size_t)i * n + K0 + j];
      }
      __syncthreads();
      for (int jj = 0; jj < w; ++jj) {
        const int k = K0 + jj;
        const int bi = pivot_search<double, kThreads>(panel, W, jj, n, used, red_k, red_i);
        if (tid == 0) {
          if (bi >= n || !(fabs(panel[bi * W + jj]) > 0.0)) {
            s_singular = blk;
          } else {
            const double pv = panel[bi * W + jj];
            s_inv = 1.0 / pv;
            s_p = bi;
            piv[k] = bi;
            used[bi] = 1;
            pabs[k] = fabs(pv);
            if (pv < 0.0) s_sgn = -s_sgn;
          }
        }
        __syncthreads();
        if (s_singular == blk) break;
        const int p = s_p;
        const double inv = s_inv;
        for (int j = tid; j < w; j += kThreads) rowp[j] = (j == jj) ? inv : panel[p * W + j] * inv;
        for (int i = tid; i < n; i += kThreads) colk[i] = panel[i * W + jj];
        __syncthreads();
        for (int e = tid; e < n * W; e += kThreads) {
          const int i = e / W, j = e % W;
          if (j >= w) continue;
          if (i == p) {
            panel[e] = rowp[j];
          } else {
            const double f = colk[i];
            const double base = (j == jj) ? 0.0 : panel[e];
            panel[e] = base - f * rowp[j];
          }
        }
        __syncthreads();
      }
    }
    cluster.sync();  // the owner's swept panel, pivots and singular flag are visible
    const int* o_sing = cluster.map_shared_rank(&s_singular, owner);
    if (*o_sing <= blk) {
      singular = true;
      break;
    }
    if (q != owner) {
      const double* o_panel = cluster.map_shared_rank(panel, owner);
      const int* o_piv = cluster.map_shared_rank(piv, owner);
      for (int e = tid; e < n * W; e += kThreads)
        if (e % W < w) panel[e] = o_panel[e];
      for (int j = tid; j < w; j += kThreads) piv[K0 + j] = o_piv[K0 + j];
      __syncthreads();
      for (int j = tid; j < w; j += kThreads) used[piv[K0 + j]] = 1;
    }
    // old pivot rows of the block on this CTA's columns (outside the panel)
    for (int e = tid; e < w * ncol; e += kThreads) {
      const int j = e / ncol, cc = e - j * ncol;
      prow[j * ldp + cc] = A[(size_t)piv[K0 + j] * n + c_lo + cc];
    }
    __syncthreads();
    // rank-w update of this CTA's columns outside the panel (the order of k_gj)
    for (int i = warp; i < n; i += kThreads / 32) {
      double u[W];
#pragma unroll
      for (int j = 0; j < W; ++j) u[j] = (j < w) ? panel[i * W + j] - ((piv[K0 + j] == i) ? 1.0 : 0.0) : 0.0;
      double* Ai = A + (size_t)i * n;
      int c = c_lo + lane;
      for (; c + 32 < c_hi; c += 64) {
        const int c2 = c + 32;
        const bool in1 = !(c >= K0 && c < K0 + w);
        const bool in2 = !(c2 >= K0 && c2 < K0 + w);
        double a1 = in1 ? Ai[c] : 0.0;
        double a2 = in2 ? Ai[c2] : 0.0;
#pragma unroll
        for (int j = 0; j < W; ++j) {
          if (j < w) {
            a1 += u[j] * prow[j * ldp + (c - c_lo)];
            a2 += u[j] * prow[j * ldp + (c2 - c_lo)];
          }
        }
        if (in1) Ai[c] = a1;
        if (in2) Ai[c2] = a2;
      }
      if (c < c_hi && !(c >= K0 && c < K0 + w)) {
        double a1 = Ai[c];
#pragma unroll
        for (int j = 0; j < W; ++j)
          if (j < w) a1 += u[j] * prow[j * ldp + (c - c_lo)];
        Ai[c] = a1;
      }
    }
    if (q == owner) {
      for (int e = tid; e < n * W; e += kThreads) {
        const int i = e / W, j = e % W;
        if (j < w) A[(size_t)i * n + K0 + j] = panel[e];
      }
    }
    __syncthreads();
  }
  cluster.sync();  // all pivots and flags final: rank 0 gathers the pivots of every block
  if (q == 0) {
    // each column's pivot from the CTA that owns its block, summed as in k_gj
    if (!singular)
      for (int k = tid; k < n; k += kThreads) pabs[k] = cluster.map_shared_rank(pabs, (k / W) / bpc)[k];
    __syncthreads();
    const double logdet = warp == 0 ? sum_log_pivots(pabs, n, singular) : 0.0;
    if (tid == 0) {
      double la = logdet;
      int sg = 1;
      for (int r = 0; r < C; ++r) sg *= *cluster.map_shared_rank(&s_sgn, r);
      if (singular) {
        la = -INFINITY;
        sg = 0;
        if (status) status[b] |= SCALE_SAMPLE_SINGULAR;
      } else {
        for (int k = 0; k < n; ++k) qinv[k] = 0;
        int parity = 0;
        for (int k = 0; k < n; ++k) {
          if (qinv[k]) continue;
          int j = k, len = 0;
          while (!qinv[j]) {
            qinv[j] = 1;
            j = piv[j];
            ++len;
          }
          parity += len - 1;
        }
        if (parity & 1) sg = -sg;
      }
      if (logabs_out) logabs_out[b] = la;
      if (sign_out) sign_out[b] = sg;
    }
  }
  if (singular) {
    // zero this CTA's share of the rows of Binv
    const int r0 = (int)((long long)n * q / C), r1 = (int)((long long)n * (q + 1) / C);
    for (int e = tid; e < (r1 - r0) * n; e += kThreads) binv[(size_t)b * n * n + (size_t)r0 * n + e] = TOUT(0);
  } else {
    // Binv[s][cf] = A^-1[cf][s] = A_final[piv[cf]][col] with s = piv[col], col in this CTA's range
    for (int e = tid; e < ncol * n; e += kThreads) {
      const int cc = e / n, cf = e - cc * n, col = c_lo + cc;
      binv[(size_t)b * n * n + (size_t)piv[col] * n + cf] = (TOUT)A[(size_t)piv[cf] * n + col];
    }
  }
  cluster.sync();  // rank 0 read the others' pivots and signs
}

template <typename TOUT, int W, int C>
cudaError_t run_gj_cluster(cudaStream_t st, double* mats, int n, int B, const int32_t* list, TOUT* binv, double* la,
                           int32_t* sg, int32_t* status) {
  const int nblocks = (n + W - 1) / W, bpc = (nblocks + C - 1) / C;
  const size_t smem =
      sizeof(double) * ((size_t)n + 2 * n * W + (size_t)W * bpc * W + n + W) + sizeof(int) * 2 * n + n + 16;
  auto kern = k_gj_cluster<TOUT, W, C>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();  // above 1443 rows the panels leave no room
    return cudaErrorNotSupported;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)B * C);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();  // clear; the caller falls back to one CTA per matrix
    return cudaErrorNotSupported;
  }
  return cudaLaunchKernelEx(&cfg, kern, mats, n, list, binv, la, sg, status);
}

template <typename TW, typename TOUT, bool kInverse, int W, int TH = kThreads>
cudaError_t run_gj(cudaStream_t st, TW* mats, int n, int B, const int32_t* list, TOUT* binv, double* la,
                   int32_t* sg, int32_t* status) {
  const size_t smem = sizeof(double) * n + sizeof(TW) * ((size_t)2 * n * W + n + W) + sizeof(int) * 2 * n + n + 16;
  auto kern = k_gj<TW, TOUT, kInverse, W, TH>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<B, TH, smem, st>>>(mats, n, list, binv, la, sg, status);
  return cudaGetLastError();
}

// ---- FP64 elimination with the rank-16 updates on the tensor cores -------------------------
// Gauss-Jordan in blocks of 16 pivots, the products of a block taken as split FP16 products
// (fp64_mma.cuh): of the 16 DFMA per element and block one rounded FP64 addition is left. Pivot
// choices, the panel's elimination and every stored value are FP64.
//
//  (1) Panel: LU with partial pivoting of the block's 16 columns, one thread per row, the row in
//      registers; the inverse's earlier pivot rows take the same steps. Pivot: the largest
//      |value| among the rows without a pivot, ties to the lowest row, by warp reductions on
//      integer keys.
//  (2) X = L11^-1 and (inverse) U11^-1 by warp 0, the column slices of the old pivot rows P by
//      the other warps.
//  (3) The left factor U = -L21 X of the rows without a pivot, -U11^-1 X of the block's pivot rows,
//      as split products (its fragment order is that of (4)'s operand, so it stays in registers);
//      X's unit diagonal is left to an FP64 addition. U is also the block's columns of the matrix
//      after the sweep.
//  (4) A[i][c] += sum_k U[i][k] P[k][c] outside the block, a pivot row starting from zero.
//
// Elements whose split sum could lose digits that an FP64 chain keeps (split_weak) are taken by
// such a chain: in (3) from the panel and X in shared memory, in (4) from U in the warp's registers and
// P in FP64 (the matrix itself without inverse, where no pivot row changes; else a copy in the block
// of Binv that the inverse is going to overwrite). A tile's weak elements are queued, so that 32 of them
// share one chain of 16 multiply-adds per lane: a 16 x 16 Hubbard walker has 3% of them, in 6% of the tiles.
constexpr int kSW = 16;        // pivots per block = k of one mma
constexpr int kSLd = kSW + 2;  // panel row stride in doubles: 16-byte rows without bank conflicts
constexpr int kSTd = kSW + 1;  // row stride of the 16 x 16 blocks
constexpr int kSCols = 256;    // columns whose slices are staged at a time: all of them up to 256 rows
constexpr int kSColsTall = 128;  // beside a panel of more than 512 rows
constexpr int kSplitMaxN = 1024;
constexpr int kSPkMax = 32;    // rows up to which the block of Binv is too small for P
constexpr int kSMs = 152;

struct SplitSmem {
  size_t panel, tri, xs, xf, xe, prow, inv, bf, fexp, pk, piv, qinv, act, used, total;
};
__host__ __device__ inline SplitSmem split_smem(int n, int ch) {
  SplitSmem s{};
  size_t off = sizeof(double) * (size_t)((n + 1) & ~1);  // pabs
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 15) & ~size_t(15);
    return at;
  };
  s.panel = take(sizeof(double) * (size_t)n * kSLd);
  s.tri = take(sizeof(double) * kSW * kSTd);
  s.xs = take(sizeof(double) * kSW * kSTd);
  s.xf = take((size_t)2 * kSplit * 32 * sizeof(uint2));
  s.xe = take(sizeof(int) * kSW);
  s.prow = take(sizeof(double) * kSW);
  s.inv = take(sizeof(double) * kSW);
  s.bf = take((size_t)(ch / 8) * kSplit * 32 * sizeof(uint2));
  s.fexp = take(sizeof(int) * ch);
  s.pk = take(n <= kSPkMax ? sizeof(double) * kSW * n : 0);
  s.piv = take(sizeof(int) * n);
  s.qinv = take(sizeof(int) * n);
  s.act = take(sizeof(int) * n);
  s.used = take(n);
  s.total = off;
  return s;
}

__device__ __forceinline__ uint64_t dbits(double x) { return (uint64_t)__double_as_longlong(x); }

// Slices of the B fragment of one 8-column tile from the lane's values x[q] (row k = 2t + (q & 1)
// + 8 (q >> 1) of the lane's column g); the column's scale to *fe (t == 0).
__device__ __forceinline__ void split_column_tile(const uint64_t (&x)[4], uint2* bf, int* fe) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  int e = max(max(exp_field(x[0]), exp_field(x[1])), max(exp_field(x[2]), exp_field(x[3])));
  int nz = ((x[0] | x[1] | x[2] | x[3]) << 1) != 0;
#pragma unroll
  for (int off = 1; off < 4; off <<= 1) {
    e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
    nz |= __shfl_xor_sync(0xffffffffu, nz, off);
  }
  if (t == 0) fe[g] = split_scale(e, nz != 0);
  uint32_t s0[kSplit], s1[kSplit];
  split_pair(split_fixed(x[0], e), split_fixed(x[1], e), s0);
  split_pair(split_fixed(x[2], e), split_fixed(x[3], e), s1);
#pragma unroll
  for (int l = 0; l < kSplit; ++l) bf[l * 32 + lane] = make_uint2(s0[l], s1[l]);
}

// Slices of the A fragment of 16 rows from the lane's values v[q][0..1] (row g + 8 (q & 1), columns
// 2t, 2t + 1 at q < 2 and 2t + 8, 2t + 9 at q >= 2); the scales of the lane's two rows come back in ex.
__device__ __forceinline__ void split_row_tile(const double (&v)[4][2], uint32_t (&a)[kSplit][4], int (&ex)[2]) {
  int em[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint64_t x0 = dbits(v[h][0]), x1 = dbits(v[h][1]), x2 = dbits(v[2 + h][0]), x3 = dbits(v[2 + h][1]);
    int e = max(max(exp_field(x0), exp_field(x1)), max(exp_field(x2), exp_field(x3)));
    int nz = ((x0 | x1 | x2 | x3) << 1) != 0;
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
      nz |= __shfl_xor_sync(0xffffffffu, nz, off);
    }
    em[h] = e;
    ex[h] = split_scale(e, nz != 0);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t s[kSplit];
    split_pair(split_fixed(dbits(v[q][0]), em[q & 1]), split_fixed(dbits(v[q][1]), em[q & 1]), s);
#pragma unroll
    for (int l = 0; l < kSplit; ++l) a[l][q] = s[l];
  }
}

// One matrix by a cluster of C CTAs of TH threads, R TH >= n, R rows of the panel per thread. The
// column blocks are dealt out to the CTAs in turn; every CTA takes the panel, (2) and (3) itself,
// with the same bits, and updates its own columns, with no exchange but through the matrix. Two
// cluster barriers a block: the updates of a block before the next one's panel loads, and the panel loads
// (before the first block the scan of the rows' exponents too) before any store to the matrix, as the
// owner of the block's columns stores them swept. The second is split: CTAs arrive with their panel in
// registers and wait after the pivot steps, which hide it.
template <typename TOUT, bool kInverse, int TH, int R, int C>
__device__ void gj_split_one(unsigned char* smem_raw, double* __restrict__ mats, int n, int ch, int b,
                             TOUT* __restrict__ binv, double* __restrict__ logabs_out, int32_t* __restrict__ sign_out,
                             int32_t* __restrict__ status) {
  constexpr int NW = TH / 32;
  const SplitSmem S = split_smem(n, ch);
  double* pabs = reinterpret_cast<double*>(smem_raw);            // [n] |pivot| of column k
  double* panel = reinterpret_cast<double*>(smem_raw + S.panel);  // [n][kSLd], row r = matrix row act[r]
  double* tri = reinterpret_cast<double*>(smem_raw + S.tri);      // [16][kSTd] L11 below, U11 on and above the diagonal
  double* xs = reinterpret_cast<double*>(smem_raw + S.xs);        // [16][kSTd] X = L11^-1
  uint2* xf = reinterpret_cast<uint2*>(smem_raw + S.xf);          // its slices, two tiles
  int* xe = reinterpret_cast<int*>(smem_raw + S.xe);              // [16] its column scales
  double* prow = reinterpret_cast<double*>(smem_raw + S.prow);    // [16] the pivot row right of the pivot
  double* inv = reinterpret_cast<double*>(smem_raw + S.inv);      // [16] reciprocal pivots
  uint2* bf = reinterpret_cast<uint2*>(smem_raw + S.bf);          // [ch / 8][kSplit][32] slices of P
  int* fexp = reinterpret_cast<int*>(smem_raw + S.fexp);          // [ch] column scales of P
  int* piv = reinterpret_cast<int*>(smem_raw + S.piv);            // [n] pivot row of column k
  int* qinv = reinterpret_cast<int*>(smem_raw + S.qinv);          // [n]
  int* act = reinterpret_cast<int*>(smem_raw + S.act);            // [n] rows in work: all, or those without a pivot
  unsigned char* used = smem_raw + S.used;                        // [n] 0, or 1 + block that pivoted the row
  const int cta = C == 1 ? 0 : (int)cg::this_cluster().block_rank();
  auto sync_all = [] {
    if constexpr (C == 1) __syncthreads();
    else cg::this_cluster().sync();
  };
  __shared__ uint4 cand[NW];
  __shared__ int prr[kSW];  // panel rows of the block's pivots
  __shared__ unsigned char queue[NW][128];  // a tile's weak elements, 8 row + column
  __shared__ int s_nact, s_sgn;

  double* A = mats + (size_t)b * n * n;
  // inverse: [16][n] the block's old pivot rows P
  double* pk = nullptr;
  if constexpr (kInverse)
    pk = n <= kSPkMax ? reinterpret_cast<double*>(smem_raw + S.pk)
                      : reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(binv + (size_t)b * n * n) + 7) & ~(uintptr_t)7);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const bool vec = (n & 1) == 0;  // rows of A start on 16 bytes

  for (int i = tid; i < n; i += TH) {
    used[i] = 0;
    act[i] = i;
  }
  if (tid == 0) {
    s_nact = n;
    s_sgn = 1;
  }
  __syncthreads();

  bool singular = false;
  for (int K0 = 0; K0 < n; K0 += kSW) {
    const int w = min(kSW, n - K0), nact = s_nact;
    const unsigned char blk = (unsigned char)(1 + K0 / kSW);
    // (1) panel: the thread's rows act[tid + TH m] (past L1: another CTA may have written them)
    int row[R], own[R];  // own: the pivot the row became
    bool open[R];        // may become a pivot row
    double a[R][kSW];
#pragma unroll
    for (int m = 0; m < R; ++m) {
      row[m] = tid + TH * m < nact ? act[tid + TH * m] : -1;
      open[m] = row[m] >= 0 && !used[row[m]];
      own[m] = -1;
      const double* src = A + (size_t)max(row[m], 0) * n + K0;
      if (vec && w == kSW) {
#pragma unroll
        for (int k = 0; k < kSW; k += 2) {
          const double2 v = row[m] >= 0 ? __ldcg(reinterpret_cast<const double2*>(src + k)) : make_double2(0.0, 0.0);
          a[m][k] = v.x;
          a[m][k + 1] = v.y;
        }
      } else {
#pragma unroll
        for (int k = 0; k < kSW; ++k) a[m][k] = (row[m] >= 0 && k < w) ? __ldcg(src + k) : 0.0;
      }
    }
    if constexpr (C > 1) cg::this_cluster().barrier_arrive();  // the matrix is read as far as this block needs it
    if (tid < kSW * kSW) tri[(tid / kSW) * kSTd + tid % kSW] = tid / kSW == tid % kSW ? 1.0 : 0.0;
    for (int q = TH + tid; q < kSW * kSW; q += TH) tri[(q / kSW) * kSTd + q % kSW] = q / kSW == q % kSW ? 1.0 : 0.0;
    if (tid < kSW) {
      inv[tid] = 1.0;
      prr[tid] = -1;
    }
#pragma unroll
    for (int jj = 0; jj < kSW; ++jj) {
      if (jj >= w || singular) continue;  // uniform
      // the candidate of each warp: largest key (0: none; the key's upper word + 1, lower word),
      // ties to the lowest row
      unsigned hi[R], lo[R], h = 0u, l = 0u;
#pragma unroll
      for (int m = 0; m < R; ++m) {
        const uint64_t key = dbits(a[m][jj]) & 0x7fffffffffffffffull;
        const bool valid = open[m] && own[m] < 0;
        hi[m] = valid ? (unsigned)(key >> 32) + 1u : 0u;
        lo[m] = valid ? (unsigned)key : 0u;
        h = max(h, hi[m]);
      }
      const unsigned m1 = __reduce_max_sync(0xffffffffu, h);
#pragma unroll
      for (int m = 0; m < R; ++m) l = max(l, hi[m] == m1 ? lo[m] : 0u);
      const unsigned m2 = __reduce_max_sync(0xffffffffu, l);
      unsigned r = 0x7fffffffu;
#pragma unroll
      for (int m = R - 1; m >= 0; --m)
        if (hi[m] == m1 && lo[m] == m2) r = (unsigned)(tid + TH * m);
      r = __reduce_min_sync(0xffffffffu, r);
      if (lane == 0) cand[warp] = make_uint4(m1, m2, r, 0u);
      __syncthreads();
      const uint4 c = lane < NW ? cand[lane] : make_uint4(0u, 0u, 0x7fffffffu, 0u);
      const unsigned g1 = __reduce_max_sync(0xffffffffu, c.x);
      const unsigned g2 = __reduce_max_sync(0xffffffffu, c.x == g1 ? c.y : 0u);
      const int rp = (int)__reduce_min_sync(0xffffffffu, c.x == g1 && c.y == g2 ? c.z : 0x7fffffffu);
      // no row left, a zero column, or a NaN in it
      if (g1 == 0u || (g1 == 1u && g2 == 0u) || g1 > 0x7ff00001u || (g1 == 0x7ff00001u && g2 != 0u)) {
        singular = true;
        continue;
      }
      const int rt = rp % TH, rm = rp / TH;
      if (warp == (rt >> 5)) {
        double pv = a[0][jj];
#pragma unroll
        for (int m = 1; m < R; ++m) pv = rm == m ? a[m][jj] : pv;
        pv = __shfl_sync(0xffffffffu, pv, rt & 31);
        const double ip = __drcp_rn(pv);
#pragma unroll
        for (int m = 0; m < R; ++m) {
          if (lane != (rt & 31) || rm != m) continue;
          own[m] = jj;
#pragma unroll
          for (int k = jj + 1; k < kSW; ++k) prow[k] = a[m][k];
          inv[jj] = ip;
          prr[jj] = rp;
          piv[K0 + jj] = row[m];
          used[row[m]] = blk;
          pabs[K0 + jj] = fabs(pv);
          if (dbits(pv) >> 63) s_sgn = -s_sgn;
        }
      }
      __syncthreads();
#pragma unroll
      for (int m = 0; m < R; ++m) {
        if (row[m] < 0 || own[m] >= 0) continue;  // the inverse's earlier pivot rows take part
        const double f = a[m][jj] * inv[jj];
        a[m][jj] = f;
#pragma unroll
        for (int k = jj + 1; k < kSW; ++k) a[m][k] = fma(-f, prow[k], a[m][k]);
      }
    }
    if constexpr (C > 1) cg::this_cluster().barrier_wait();  // ... by every CTA: stores may follow
    if (singular) break;
    const int c_lo = kInverse ? 0 : K0 + w;
    if (c_lo >= n) break;  // determinant: the last block is done
#pragma unroll
    for (int m = 0; m < R; ++m) {
      if (own[m] < 0) continue;
#pragma unroll
      for (int k = 0; k < kSW; ++k) tri[own[m] * kSTd + k] = a[m][k];
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < R; ++m) {
      if (row[m] < 0 || own[m] >= 0) continue;
#pragma unroll
      for (int k = 0; k < kSW; k += 2)
        *reinterpret_cast<double2*>(panel + (tid + TH * m) * kSLd + k) = make_double2(a[m][k], a[m][k + 1]);
    }
    // (2)
    if (warp == 0) {
      // lanes 0..15: column `lane` of L11^-1 by forward substitution; lanes 16..31 (inverse): column
      // lane - 16 of U11^-1 by backward substitution, with every index reversed (i -> 15 - i)
      const bool up = lane >= kSW;
      const int col = up ? 2 * kSW - 1 - lane : lane;
      const double* tp = up ? tri + (kSW - 1) * (kSTd + 1) : tri;
      const int dir = up ? -1 : 1;
      double x[kSW];
#pragma unroll
      for (int i = 0; i < kSW; ++i) x[i] = i == col ? 1.0 : 0.0;
#pragma unroll
      for (int s = 0; s < kSW; ++s) {
        double l[kSW];
#pragma unroll
        for (int i = s + 1; i < kSW; ++i) l[i] = tp[dir * (i * kSTd + s)];
        if (kInverse) x[s] *= up ? inv[kSW - 1 - s] : 1.0;
#pragma unroll
        for (int i = s + 1; i < kSW; ++i) x[i] = fma(-l[i], x[s], x[i]);
      }
      if (!up) {
#pragma unroll
        for (int i = 0; i < kSW; ++i) xs[i * kSTd + col] = x[i];
      } else if (kInverse) {  // the pivot rows of (3): -U11^-1
#pragma unroll
        for (int i = 0; i < kSW; ++i)
          if (prr[kSW - 1 - i] >= 0) panel[prr[kSW - 1 - i] * kSLd + kSW - 1 - col] = -x[i];
      }
      __syncwarp();
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        uint64_t v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = 2 * t + (q & 1) + 8 * (q >> 1), c = 8 * nt + g;
          v[q] = k == c ? 0ull : dbits(xs[k * kSTd + c]);
        }
        split_column_tile(v, xf + nt * kSplit * 32, xe + 8 * nt);
      }
    }
    // this CTA's column blocks from c_lo on: tile nt is half of block jb0 + (nt >> 1) C
    const int nb = (n + kSW - 1) / kSW, lo_b = c_lo / kSW;
    const int jb0 = lo_b + ((cta - lo_b) % C + C) % C;
    const int ntiles = jb0 < nb ? 2 * ((nb - 1 - jb0) / C + 1) : 0;
    for (int t0 = 0; t0 < ntiles; t0 += ch / 8) {
      const int ntile = min(ch / 8, ntiles - t0);
      auto tile_col = [&](int nt) { return (jb0 + ((t0 + nt) >> 1) * C) * kSW + 8 * ((t0 + nt) & 1); };
      // column slices of the block's old pivot rows: a warp per 8-column tile (warp 0 joins late)
      const int w0 = t0 == 0 ? (warp + NW - 1) % NW : warp;
      for (int nt = w0; nt < ntile; nt += NW) {
        const int c0 = tile_col(nt), c = c0 + g;
        if (kInverse && (unsigned)(c0 - K0) < (unsigned)kSW) continue;
        uint64_t x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = 2 * t + (q & 1) + 8 * (q >> 1);
          x[q] = (k < w && c < n) ? dbits(A[(size_t)piv[K0 + k] * n + c]) : 0ull;
          if (kInverse && c < n) pk[(size_t)k * n + c] = __longlong_as_double((long long)x[q]);
        }
        split_column_tile(x, bf + (size_t)nt * kSplit * 32, fexp + 8 * nt);
      }
      __syncthreads();
      // strips of 16 rows in runs of column tiles; as many runs per strip as even out the warps
      // best (a run's row slices cost about five tiles)
      const int nstrip = (nact + 15) >> 4;
      int cs = 1, best = 1 << 30;
      for (int q = 1; q <= min(ntile, 8); ++q) {
        const int cost = ((nstrip * q + NW - 1) / NW) * ((ntile + q - 1) / q + 5);
        if (cost < best) {
          best = cost;
          cs = q;
        }
      }
      const int per = (ntile + cs - 1) / cs;
      for (int task = warp; task < nstrip * cs; task += NW) {
        const int strip = task % nstrip, run = task / nstrip;
        const int r0 = strip * 16 + g, r1 = r0 + 8;
        const int i0 = r0 < nact ? act[r0] : 0, i1 = r1 < nact ? act[r1] : 0;
        // rows to write; a pivot row of this block starts from zero (inverse) or is done with
        const bool on0 = r0 < nact && (kInverse || !used[i0]), on1 = r1 < nact && (kInverse || !used[i1]);
        const bool add0 = on0 && !(kInverse && used[i0] == blk), add1 = on1 && !(kInverse && used[i1] == blk);
        double* A0 = A + (size_t)i0 * n;
        double* A1 = A + (size_t)i1 * n;
        uint32_t as[kSplit][4];
        int ex[2];
        float acc[kSplit][4], wt[4];
        // (3)
        double u[4][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          double2 v = make_double2(0.0, 0.0);
          if ((q & 1) ? on1 : on0)
            v = *reinterpret_cast<const double2*>(panel + ((q & 1) ? r1 : r0) * kSLd + 2 * t + 8 * (q >> 1));
          u[q][0] = v.x;
          u[q][1] = v.y;
        }
        split_row_tile(u, as, ex);
        unsigned weak = 0;  // bit 2 q + e: u[q][e]
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          split_mma(acc, as, xf + nt * kSplit * 32);
          split_weight(wt, as[0], xf[nt * kSplit * 32 + lane]);
          const int2 f = *reinterpret_cast<const int2*>(xe + 8 * nt + 2 * t);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            double& l = u[2 * nt + (i >> 1)][i & 1];
            const int e = ex[i >> 1], fe = (i & 1) ? f.y : f.x;
            // the diagonal's term counts too: at least 1/16 of the scales
            if (fe != 0 && split_weak(wt[i], e, fe) && !(e > 0 && fe > 0 && exp_field(dbits(l)) >= e + fe - 1026))
              weak |= 1u << (4 * nt + i);
            l = -(l + split_value(acc, i, e, fe));
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (!((weak >> j) & 1u)) continue;
          const int c = 2 * t + (j & 1) + 8 * (j >> 2);
          const double* l = panel + (((j >> 1) & 1) ? r1 : r0) * kSLd;
          double v = -l[c];
          for (int k = c + 1; k < kSW; ++k) v = fma(-l[k], xs[k * kSTd + c], v);
          u[j >> 1][j & 1] = v;
        }
        if (kInverse && run == 0 && t0 == 0 && (K0 / kSW) % C == cta) {  // the block's columns after the sweep
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            double* dst = ((q & 1) ? A1 : A0) + K0;
            const int c = 2 * t + 8 * (q >> 1);
            if (!((q & 1) ? on1 : on0)) continue;
            if (c < w) dst[c] = u[q][0];
            if (c + 1 < w) dst[c + 1] = u[q][1];
          }
        }
        split_row_tile(u, as, ex);
        // (4)
        for (int nt = run * per; nt < min(ntile, (run + 1) * per); ++nt) {
          const int c0 = tile_col(nt), c = c0 + 2 * t;
          if (kInverse && (unsigned)(c0 - K0) < (unsigned)kSW) continue;
          const bool in0 = c < n, in1 = c + 1 < n;
          double v[4] = {0.0, 0.0, 0.0, 0.0};
          if (vec) {
            if (in0 && add0) {
              const double2 q = *reinterpret_cast<const double2*>(A0 + c);
              v[0] = q.x;
              v[1] = q.y;
            }
            if (in0 && add1) {
              const double2 q = *reinterpret_cast<const double2*>(A1 + c);
              v[2] = q.x;
              v[3] = q.y;
            }
          } else {
            if (in0 && add0) v[0] = A0[c];
            if (in1 && add0) v[1] = A0[c + 1];
            if (in0 && add1) v[2] = A1[c];
            if (in1 && add1) v[3] = A1[c + 1];
          }
          const uint2* bt = bf + (size_t)nt * kSplit * 32;
          split_mma(acc, as, bt);
          split_weight(wt, as[0], bt[lane]);
          const int2 f = *reinterpret_cast<const int2*>(fexp + 8 * nt + 2 * t);
          v[0] += split_value(acc, 0, ex[0], f.x);
          v[1] += split_value(acc, 1, ex[0], f.y);
          v[2] += split_value(acc, 2, ex[1], f.x);
          v[3] += split_value(acc, 3, ex[1], f.y);
          const bool k0 = split_weak(wt[0], ex[0], f.x) && on0 && in0, k1 = split_weak(wt[1], ex[0], f.y) && on0 && in1;
          const bool k2 = split_weak(wt[2], ex[1], f.x) && on1 && in0, k3 = split_weak(wt[3], ex[1], f.y) && on1 && in1;
          const bool some = __any_sync(0xffffffffu, k0 || k1 || k2 || k3);
          if (vec && !some) {
            if (on0 && in0) *reinterpret_cast<double2*>(A0 + c) = make_double2(v[0], v[1]);
            if (on1 && in0) *reinterpret_cast<double2*>(A1 + c) = make_double2(v[2], v[3]);
            continue;
          }
          if (on0 && in0 && !k0) A0[c] = v[0];
          if (on0 && in1 && !k1) A0[c + 1] = v[1];
          if (on1 && in0 && !k2) A1[c] = v[2];
          if (on1 && in1 && !k3) A1[c + 1] = v[3];
          if (!some) continue;
          int cnt = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const bool k = i == 0 ? k0 : i == 1 ? k1 : i == 2 ? k2 : k3;
            const unsigned bal = __ballot_sync(0xffffffffu, k);
            if (k) queue[warp][cnt + __popc(bal & ((1u << lane) - 1u))] = (unsigned char)(8 * (g + 8 * (i >> 1)) + 2 * t + (i & 1));
            cnt += __popc(bal);
          }
          __syncwarp();
          for (int q0 = 0; q0 < cnt; q0 += 32) {
            const bool mine = q0 + lane < cnt;
            const int code = mine ? queue[warp][q0 + lane] : 0, rr = code >> 3, cc = c0 + (code & 7);
            const int i = act[strip * 16 + (mine ? rr : 0)];
            double* dst = A + (size_t)i * n + cc;
            double s0 = mine && !(kInverse && used[i] == blk) ? *dst : 0.0, s1 = 0.0;
#pragma unroll
            for (int k = 0; k < kSW; ++k) {
              const int src = 4 * (rr & 7) + ((k >> 1) & 3);
              const double ua = __shfl_sync(0xffffffffu, u[2 * (k >> 3)][k & 1], src);
              const double ub = __shfl_sync(0xffffffffu, u[2 * (k >> 3) + 1][k & 1], src);
              double p = 0.0;
              if (mine && k < w) p = kInverse ? pk[(size_t)k * n + cc] : A[(size_t)piv[K0 + k] * n + cc];
              if (k & 1) s1 = fma(rr < 8 ? ua : ub, p, s1);
              else s0 = fma(rr < 8 ? ua : ub, p, s0);
            }
            if (mine) *dst = s0 + s1;
          }
          __syncwarp();
        }
      }
      __syncthreads();
    }
    if (!kInverse && warp == 0) {  // the rows not yet pivoted, compacted in place
      int m = 0;
      for (int r0 = 0; r0 < nact; r0 += 32) {
        const int i = r0 + lane < nact ? act[r0 + lane] : 0;
        const bool on = r0 + lane < nact && !used[i];
        const unsigned bal = __ballot_sync(0xffffffffu, on);
        if (on) act[m + __popc(bal & ((1u << lane) - 1u))] = i;
        m += __popc(bal);
        __syncwarp();
      }
      if (lane == 0) s_nact = m;
    }
    sync_all();
  }
  __syncthreads();

  const double logdet = warp == 0 ? sum_log_pivots(pabs, n, singular) : 0.0;  // on thread 0
  if (tid == 0 && cta == 0) {
    int st = 0;
    double la = logdet;
    int sg = s_sgn;
    if (singular) {
      st = SCALE_SAMPLE_SINGULAR;
      la = -INFINITY;
      sg = 0;
    } else {
      // sign of the permutation k -> piv[k]
      for (int k = 0; k < n; ++k) qinv[k] = 0;
      int parity = 0;
      for (int k = 0; k < n; ++k) {
        if (qinv[k]) continue;
        int j = k, len = 0;
        while (!qinv[j]) {
          qinv[j] = 1;
          j = piv[j];
          ++len;
        }
        parity += len - 1;
      }
      if (parity & 1) sg = -sg;
    }
    if (logabs_out) logabs_out[b] = la;
    if (sign_out) sign_out[b] = sg;
    if (status && st) status[b] |= st;
  }
  if (!kInverse) return;
  __syncthreads();
  if (singular) {
    if (binv)
      for (int q = cta * TH + tid; q < n * n; q += C * TH) binv[(size_t)b * n * n + q] = TOUT(0);
    return;
  }
  for (int k = tid; k < n; k += TH) qinv[piv[k]] = k;
  __syncthreads();
  // Binv[s][cf] = A^-1[cf][s] = A_final[piv[cf]][qinv[s]]
  for (int q = cta * TH + tid; q < n * n; q += C * TH) {
    const int s = q / n, cf = q - s * n;
    binv[(size_t)b * n * n + q] = (TOUT)__ldcg(A + (size_t)piv[cf] * n + qinv[s]);
  }
}

// All B matrices, the listed ones (entries below 0 are skipped), or the first *count entries of a
// compacted list, from a grid of at most the resident CTAs in that case.
template <typename TOUT, bool kInverse, int TH, int MINB, int R, int C>
__global__ void __launch_bounds__(TH, MINB) k_gj_split(double* __restrict__ mats, int n, int ch, int B,
                                                       const int32_t* __restrict__ list, const int32_t* __restrict__ count,
                                                       TOUT* __restrict__ binv, double* __restrict__ logabs_out,
                                                       int32_t* __restrict__ sign_out, int32_t* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int total = count ? min(*count, B) : B;
  for (int e = blockIdx.x / C; e < total; e += gridDim.x / C) {
    const int b = list ? list[e] : e;
    if (b >= 0) gj_split_one<TOUT, kInverse, TH, R, C>(smem_raw, mats, n, ch, b, binv, logabs_out, sign_out, status);
    // the next matrix takes the same shared memory; a cluster goes on to it together
    if constexpr (C == 1) __syncthreads();
    else cg::this_cluster().sync();
  }
}

struct GjArgs {
  cudaStream_t st;
  double* mats;
  int n, B;
  const int32_t* list;
  const int32_t* count;
  int expect;  // matrices the caller expects in this call (<= B)
  double* la;
  int32_t* sg;
  int32_t* status;
};

template <typename TOUT, bool kInverse, int TH, int MINB, int R, int C>
cudaError_t run_gj_split(const GjArgs& a, TOUT* binv) {
  // (a determinant's updates leave out the first block)
  const int ch = std::min(std::max(((a.n + 15) & ~15) - (kInverse ? 0 : kSW), kSW), R == 1 ? kSCols : kSColsTall);
  auto kern = k_gj_split<TOUT, kInverse, TH, MINB, R, C>;
  const size_t smem = split_smem(a.n, ch).total;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.count ? std::min(a.B, kSMs * MINB / C) : a.B) * C);
  cfg.blockDim = dim3(TH);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = a.st;
  cudaLaunchAttribute attr[1];
  if (C > 1) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  e = cudaLaunchKernelEx(&cfg, kern, a.mats, a.n, ch, a.B, a.list, a.count, binv, a.la, a.sg, a.status);
  if constexpr (C > 1) {  // a partition without room for a cluster: one CTA per matrix, the same bits
    if (e != cudaSuccess) {
      cudaGetLastError();
      return run_gj_split<TOUT, kInverse, TH, MINB, R, 1>(a, binv);
    }
  }
  return e;
}

// Launch shapes (inverses of Gaussian n x n matrices, ms per call on a GB300; "old": every product on the
// FP64 pipe):
//   n <= 128: 128 threads, four CTAs per SM. n = 56: 1500 matrices 0.50 (old 2.12).
//   n <= 256: many matrices 256 threads, two CTAs per SM, one matrix's panel beside the other's
//     updates: n = 224, 1500 matrices 8.8 (old 38.3; of 16x16 walkers, some of whose products go by FP64
//     chains, 9.7). Up to one per SM 512 threads, whose warps share the updates: 1.10 alone (1.32 with 256
//     threads, old 3.83). Up to 32 matrices clusters of 4 CTAs: 0.68. (Clusters of 4 fill the GPCs' SMs at
//     about 36: 38 matrices 1.36.) Up to 72 clusters of 2, of which 76 run at once: 0.82.
//   n <= 512: 512 threads; clusters of 4 also pay in two waves: n = 448 alone 2.44 against 6.18,
//     38 to 64 matrices 4.92 against 6.3.
//   n <= 1024: two panel rows per thread; n = 896: 152 matrices 50 (old 189); alone 46.9, in a
//     cluster of 8 CTAs 8.9 (old cluster of 8 about 30); clusters of 8 run one wave up to 14, and 32 to 64
//     matrices take clusters of 4 (30.5 for 38, 48.7 with one CTA each).
template <typename TOUT, bool kInverse>
cudaError_t gj_split(const GjArgs& a, TOUT* binv) {
  if (a.n <= 128) return run_gj_split<TOUT, kInverse, 128, 4, 1, 1>(a, binv);
  if (a.n <= 512) {
    if (a.expect <= (a.n <= 256 ? 32 : 64)) return run_gj_split<TOUT, kInverse, 512, 1, 1, 4>(a, binv);
    if (a.n <= 256 && a.expect <= 72) return run_gj_split<TOUT, kInverse, 512, 1, 1, 2>(a, binv);
    if (a.n <= 256 && a.expect > kSMs) return run_gj_split<TOUT, kInverse, 256, 2, 1, 1>(a, binv);
    return run_gj_split<TOUT, kInverse, 512, 1, 1, 1>(a, binv);
  }
  if (a.expect <= 14) return run_gj_split<TOUT, kInverse, 512, 1, 2, 8>(a, binv);
  if (a.expect <= 64) return run_gj_split<TOUT, kInverse, 512, 1, 2, 4>(a, binv);
  return run_gj_split<TOUT, kInverse, 512, 1, 2, 1>(a, binv);
}

}  // namespace

// Inverses up to this many rows take k_gj: most of a split block's work is padding and fixed steps (us, k_gj_split / k_gj
// with 128 threads: n = 8 40 inverses 29 / 18, 8000 354 / 140; n = 14 35 / 34, 431 / 369; n = 17 53 / 45, 784 / 564;
// n = 24 61 / 58, 898 / 770, but 600 at a time 70 / 84).
constexpr int kSmallInverse = 20;

// FP64 inverse (out_fp64: Binv in double, else float) or determinant only, for B matrices
// [B][n][n] stored in Phi (overwritten). count (optional, device): the list is compacted, its
// first *count entries are taken. expect: how many matrices the caller expects (0: B); it
// chooses the launch shape and no result depends on it.
cudaError_t launch_gj(scale_ctx* c, const double* Phi, int n, int B, const int32_t* list, bool inverse,
                      bool out_fp64, void* Binv, double* logabs, int32_t* sign, int32_t* status, const int32_t* count,
                      int expect) {
  double* A = const_cast<double*>(Phi);
  if (B <= 0) return cudaSuccess;
  if (inverse && n <= kSmallInverse)
    return out_fp64 ? run_gj<double, double, true, 8, 128>(c->stream, A, n, B, list, (double*)Binv, logabs, sign, status)
                    : run_gj<double, float, true, 8, 128>(c->stream, A, n, B, list, (float*)Binv, logabs, sign, status);
  if (n <= kSplitMaxN) {
    const GjArgs a{c->stream, A, n, B, list, count, expect > 0 ? std::min(expect, B) : B, logabs, sign, status};
    if (!inverse) return gj_split<double, false>(a, nullptr);
    return out_fp64 ? gj_split<double, true>(a, (double*)Binv) : gj_split<float, true>(a, (float*)Binv);
  }
  if (inverse && list) {  // a refresh of a few samples is latency-bound
    const cudaError_t e =
        out_fp64 ? run_gj_cluster<double, 8, 8>(c->stream, A, n, B, list, (double*)Binv, logabs, sign, status)
                 : run_gj_cluster<float, 8, 8>(c->stream, A, n, B, list, (float*)Binv, logabs, sign, status);
    if (e != cudaErrorNotSupported) return e;
  }
  if (inverse)
    return out_fp64 ? run_gj<double, double, true, 8>(c->stream, A, n, B, list, (double*)Binv, logabs, sign, status)
                    : run_gj<double, float, true, 8>(c->stream, A, n, B, list, (float*)Binv, logabs, sign, status);
  return run_gj<double, double, false, 8, 512>(c->stream, A, n, B, list, (double*)nullptr, logabs, sign, status);
}

}  // namespace scale
