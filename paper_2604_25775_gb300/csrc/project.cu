// project.cu -- what the rank-r update reads of the inverse: the projector Pt_s = W_s Phi^-1 and
// the feature-independent part of every Slater row's product with the inverse,
// G0t = (M0 + proj_b) Phi^-1 (Sec. II.C, Eq. SMW).
#include <algorithm>

#include "scale_internal.cuh"

namespace scale {

namespace {

// Mixed precision: both are products of the walker's inverse with rows shared by all walkers,
//   out[j][col] = sum_k Binv[j][k] row_col[k],  rows: M0[o] + proj_b (G0t), proj_w[c] of spin s (Pt),
// 2 Ne^2 (2N + 2h) flops a walker, 4 Ne (2N + 2h) bytes written: bound by FP32 FMA. One kernel takes
// all columns (two read the inverse twice, the projector's with one row a thread). Register tiles of
// 8 slots x TN columns, 16-byte shared-memory loads along the slots: 5 loads per 48 FMA. Each
// output is one FMA chain over k ascending, so no result depends on the tile. 1500 walkers of
// 16x16: 4.82 ms as two kernels, 2.43 here. (On the tensor cores as three TF32 products with rounded
// additions every 16 terms: 2.33 ms, and the truncation inside the tensor core biased all ratios one way:
// the error of local energies of well-conditioned walkers grew 1.7-fold.)
constexpr int kGThreads = 224, kGK = 16;

struct ProjArgs {
  int Ne, No, h, ncol;  // ncol: No, or No + 2h with the projector's columns
  const float* Binv;
  const float* M0b;
  const float* proj_w;
  float* G0t;
  float* Pt;
  const int32_t* list;
  int B;
  const int32_t* count;
};

// RG x CG threads of 8 x TN outputs.
template <int RG, int CG, int TN>
__global__ void __launch_bounds__(kGThreads, 2) k_project32(ProjArgs a) {
  static_assert(RG * CG == kGThreads, "one thread per tile");
  constexpr int M = 8 * RG, N = CG * TN, LA = M + 4;  // LA: rows of the staged slots, 16-byte aligned
  __shared__ __align__(16) float As[2][kGK][LA];
  __shared__ __align__(16) float Bs[2][kGK][N];
  const int Ne = a.Ne, No = a.No, h = a.h;
  const int nrows = a.count ? min(*a.count, a.B) : a.B;
  const int j0 = blockIdx.x * M, c0 = blockIdx.y * N;
  const int tid = threadIdx.x, tr = (tid / CG) * 8, tc = (tid % CG) * TN;
  const bool vec = (Ne & 3) == 0 && (reinterpret_cast<uintptr_t>(a.proj_w) & 15) == 0;
  constexpr int kQ = kGK / 4;
  const int nk = (Ne + kGK - 1) / kGK;
  // staging: thread r < M takes slot row j0 + r, thread M + q the row of column c0 + q, 16 values at a time
  static_assert(M + N <= kGThreads, "a thread per staged row");
  const float* col_row = nullptr;
  if (tid >= M && tid < M + N) {
    const int col = c0 + tid - M;
    if (col < No) {
      col_row = a.M0b + (size_t)col * Ne;
    } else if (col < a.ncol) {
      const int s = (col - No) / h, cc = (col - No) - s * h;
      col_row = a.proj_w + (size_t)cc * 2 * Ne + (size_t)s * Ne;
    }
  }
  for (int lrow = blockIdx.z; lrow < nrows; lrow += gridDim.z) {
    const int b = a.list ? a.list[lrow] : lrow;
    if (b < 0) continue;  // uniform
    const float* src =
        tid >= M ? col_row : (j0 + tid < Ne ? a.Binv + (size_t)b * Ne * Ne + (size_t)(j0 + tid) * Ne : nullptr);
    float4 reg[kQ];
    auto fetch = [&](int kt) {
#pragma unroll
      for (int u = 0; u < kQ; ++u) {
        const int k = kt * kGK + 4 * u;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (src) {
          if (vec) {
            if (k < Ne) v = *reinterpret_cast<const float4*>(src + k);
          } else {
            if (k < Ne) v.x = src[k];
            if (k + 1 < Ne) v.y = src[k + 1];
            if (k + 2 < Ne) v.z = src[k + 2];
            if (k + 3 < Ne) v.w = src[k + 3];
          }
        }
        reg[u] = v;
      }
    };
    auto stage = [&](int buf) {
      if (tid >= M + N) return;
      float* dst = tid < M ? &As[buf][0][tid] : &Bs[buf][0][tid - M];
      const int ld = tid < M ? LA : N;
#pragma unroll
      for (int u = 0; u < kQ; ++u) {
        dst[(4 * u) * ld] = reg[u].x;
        dst[(4 * u + 1) * ld] = reg[u].y;
        dst[(4 * u + 2) * ld] = reg[u].z;
        dst[(4 * u + 3) * ld] = reg[u].w;
      }
    };
    float acc[8][TN] = {};
    __syncthreads();  // the previous walker's buffers are consumed
    fetch(0);
    stage(0);
    for (int kt = 0; kt < nk; ++kt) {
      if (kt + 1 < nk) fetch(kt + 1);
      __syncthreads();  // buffer kt & 1 is staged, the other one consumed
#pragma unroll 4
      for (int k = 0; k < kGK; ++k) {
        float x[8], y[TN];
        *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(&As[kt & 1][k][tr]);
        *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(&As[kt & 1][k][tr + 4]);
        if constexpr (TN % 2 == 0) {
#pragma unroll
          for (int v = 0; v < TN; v += 2) {
            const float2 q = *reinterpret_cast<const float2*>(&Bs[kt & 1][k][tc + v]);
            y[v] = q.x;
            y[v + 1] = q.y;
          }
        } else {
#pragma unroll
          for (int v = 0; v < TN; ++v) y[v] = Bs[kt & 1][k][tc + v];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
          for (int v = 0; v < TN; ++v) acc[u][v] = fmaf(x[u], y[v], acc[u][v]);
      }
      if (kt + 1 < nk) stage((kt + 1) & 1);
    }
    float* G = a.G0t + (size_t)b * Ne * No;
    float* P = a.Pt + (size_t)b * 2 * Ne * h;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = j0 + tr + u;
      if (j >= Ne) continue;
#pragma unroll
      for (int v = 0; v < TN; ++v) {
        const int col = c0 + tc + v;
        if (col < No) {
          G[(size_t)j * No + col] = acc[u][v];
        } else if (col < a.ncol) {
          const int s = (col - No) / h;
          P[((size_t)s * Ne + j) * h + (col - No) - s * h] = acc[u][v];
        }
      }
    }
  }
}

template <int RG, int CG, int TN>
cudaError_t project32_launch(scale_ctx* c, const ProjArgs& a) {
  constexpr int M = 8 * RG, N = CG * TN;
  dim3 grid((a.Ne + M - 1) / M, (a.ncol + N - 1) / N);
  grid.z = std::min(a.B, a.count ? listed_ctas(grid.x * grid.y) : 65535);
  k_project32<RG, CG, TN><<<grid, kGThreads, 0, c->stream>>>(a);
  return cudaGetLastError();
}

cudaError_t project32(scale_ctx* c, int B, const int32_t* list, const int32_t* count, bool with_pt) {
  const int No = 2 * c->N;
  const ProjArgs a{c->Ne, No, c->h, No + (with_pt ? 2 * c->h : 0), (const float*)c->Binv, (const float*)c->M0b,
                   make_net<float>(c).proj_w, (float*)c->G0t, (float*)c->Pt, list, B, count};
  // A tile's products for rows and columns past the end are not skipped, so the tile is the one of the least
  // padded area, weighted by the shapes' time per area (112 x 96 and 128 x 84 read the fewest words per FMA).
  // One-step sweeps, us, 112 x 96 / 56 x 160 / 64 x 140 / 128 x 84, 2048 walkers up to 64 electrons, 1024 up to
  // 130, 400 above: 8x8 of 56 electrons 299 / 209 / 211 / 300, of 64 318 / 309 / 232 / 320; 16x16 of 112
  // 557 / 620 / 613 / 616, of 128 1036 / 975 / 711 / 710, of 180 589 / 686 / 538 / 666, of 224
  // 723 / 856 / 844 / 809, of 256 1132 / 1176 / 973 / 940; 24x24 of 450 3528 / 3934 / 3910 / 3387.
  struct Tile {
    int m, n, weight;
    cudaError_t (*launch)(scale_ctx*, const ProjArgs&);
  };
  static constexpr Tile kTiles[] = {{112, 96, 20, project32_launch<14, 16, 6>},
                                    {56, 160, 22, project32_launch<7, 32, 5>},
                                    {64, 140, 22, project32_launch<8, 28, 5>},
                                    {128, 84, 20, project32_launch<16, 14, 6>}};
  const Tile* best = nullptr;
  long long least = 0;
  for (const Tile& t : kTiles) {
    const long long area = (long long)((c->Ne + t.m - 1) / t.m) * t.m * ((a.ncol + t.n - 1) / t.n) * t.n * t.weight;
    if (!best || area < least) {
      best = &t;
      least = area;
    }
  }
  // few walkers: a third of the outputs per thread while the large tiles leave a third of the SMs idle (a
  // one-step sweep of 16x16: 1 walker 92 us against 104, 8 walkers 107 against 111; 12 walkers 128 against 116)
  const long long tiles = (long long)((c->Ne + 111) / 112) * ((a.ncol + 95) / 96) * B;
  if (c->Ne > 56 && tiles <= 100) return project32_launch<7, 32, 2>(c, a);
  return best->launch(c, a);
}

// ---- FP64 mode ------------------------------------------------------------------------------
// Pt[s][c][:] = W_s Binv[c], i.e. the GEMM Pt[s] = Binv (Ne x Ne) * W_s^T (Ne x h),
// W_s^T[k][cc] = proj_w[cc][s*Ne + k]. 32 rows per CTA, K tiles of 32.
template <typename T>
__global__ void __launch_bounds__(256) k_project(int Ne, int h, const T* __restrict__ proj_w,
                                                 const T* __restrict__ Binv, T* __restrict__ Pt,
                                                 const int32_t* __restrict__ list, int B,
                                                 const int32_t* __restrict__ count) {
  __shared__ T Bs[32][33];
  __shared__ T Ws[32][2 * kMaxH + 1];
  const int nrows = count ? min(*count, B) : B;  // a compacted list: its first *count entries
  for (int lrow = blockIdx.y; lrow < nrows; lrow += gridDim.y) {
  __syncthreads();  // the previous sample's tiles are consumed
  const int b = list ? list[lrow] : lrow;
  if (b < 0) continue;
  const int c0 = blockIdx.x * 32;
  const int tid = threadIdx.x;
  const int row = tid >> 3, grp = tid & 7;
  const int ncol = 2 * h;
  T acc[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) acc[u] = T(0);
  const T* Bb = Binv + (size_t)b * Ne * Ne;
  for (int k0 = 0; k0 < Ne; k0 += 32) {
    for (int q = tid; q < 32 * 32; q += 256) {
      const int rr = q >> 5, kk = q & 31;
      const int c = c0 + rr, k = k0 + kk;
      Bs[rr][kk] = (c < Ne && k < Ne) ? Bb[(size_t)c * Ne + k] : T(0);
    }
    for (int q = tid; q < 32 * ncol; q += 256) {
      const int kk = q / ncol, col = q - kk * ncol;
      const int s = col / h, cc = col - s * h, k = k0 + kk;
      Ws[kk][col] = (k < Ne) ? proj_w[(size_t)cc * 2 * Ne + s * Ne + k] : T(0);
    }
    __syncthreads();
    const int kn = c0 + (row & ~3) < Ne ? min(32, Ne - k0) : 0;  // nothing for a warp past the last row
    for (int kk = 0; kk < kn; ++kk) {
      const T bv = Bs[row][kk];
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int col = grp + 8 * u;
        if (col < ncol) acc[u] += bv * Ws[kk][col];
      }
    }
    __syncthreads();
  }
  const int c = c0 + row;
  if (c < Ne) {
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int col = grp + 8 * u;
      if (col < ncol) {
        const int s = col / h, cc = col - s * h;
        Pt[(((size_t)b * 2 + s) * Ne + c) * h + cc] = acc[u];
      }
    }
  }
  }
}

// G0t[b][j][o] = (M0[o] + proj_b[s(o)]) . Binv[b][j]: the part of every Slater row's
// product with the inverse that does not depend on the network features (the moved rows of
// R need it for the target orbital). A GEMM per sample: CTA tiles of 64 slots x 64 orbitals,
// 4 x 4 per thread, K staged 32 at a time through shared memory; the listed samples only
// (their first *count entries when count is given).
template <typename T>
__global__ void __launch_bounds__(256) k_build_g0(int Ne, int No, const T* __restrict__ Binv,
                                                  const T* __restrict__ M0b, T* __restrict__ G0t,
                                                  const int32_t* __restrict__ list, int B,
                                                  const int32_t* __restrict__ count) {
  __shared__ T As[32][65];  // As[k][j] = Binv[j][k]
  __shared__ T Ms[32][65];  // Ms[k][o] = M0b[o][k]
  const int nrows = count ? min(*count, B) : B;
  const int j0 = blockIdx.x * 64, o0 = blockIdx.y * 64;
  const int tid = threadIdx.x, tr = tid >> 4, tc = tid & 15;
  // rows j0 + 16 u + tr of this warp (two tr) that exist: the padding of a tile is not worth the FP64 pipe's time
  const int un = min(4, max(0, (Ne - j0 - (tr & ~1) + 15) >> 4));
  for (int lrow = blockIdx.z; lrow < nrows; lrow += gridDim.z) {
    const int b = list ? list[lrow] : lrow;
    if (b < 0) continue;
    const T* Bb = Binv + (size_t)b * Ne * Ne;
    T acc[4][4] = {};
    for (int k0 = 0; k0 < Ne; k0 += 32) {
      __syncthreads();  // the previous tiles are consumed
      for (int q = tid; q < 64 * 32; q += 256) {
        const int rr = q >> 5, kk = q & 31, k = k0 + kk;
        As[kk][rr] = (j0 + rr < Ne && k < Ne) ? Bb[(size_t)(j0 + rr) * Ne + k] : T(0);
        Ms[kk][rr] = (o0 + rr < No && k < Ne) ? M0b[(size_t)(o0 + rr) * Ne + k] : T(0);
      }
      __syncthreads();
      const int kn = min(32, Ne - k0);
#pragma unroll 4
      for (int kk = 0; kk < kn; ++kk) {
        T x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          x[u] = As[kk][tr + 16 * u];
          y[u] = Ms[kk][tc + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (u >= un) break;
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] += x[u] * y[v];
        }
      }
    }
    T* out = G0t + (size_t)b * Ne * No;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = j0 + tr + 16 * u;
      if (j >= Ne) continue;
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int o = o0 + tc + 16 * v;
        if (o < No) out[(size_t)j * No + o] = acc[u][v];
      }
    }
  }
}

template <typename T>
cudaError_t build_g0_t(scale_ctx* c, int B, const int32_t* list, const int32_t* count) {
  const int No = 2 * c->N;
  const dim3 g0grid((c->Ne + 63) / 64, (No + 63) / 64, count ? std::min(B, 256) : std::min(B, 65535));
  k_build_g0<T><<<g0grid, 256, 0, c->stream>>>(c->Ne, No, (const T*)c->Binv, (const T*)c->M0b, (T*)c->G0t, list, B,
                                               count);
  return cudaGetLastError();
}

template <typename T>
cudaError_t project_t(scale_ctx* c, int B, const int32_t* list, const int32_t* count) {
  dim3 grid((c->Ne + 31) / 32, count ? std::min(B, 1024) : B);
  k_project<T><<<grid, 256, 0, c->stream>>>(c->Ne, c->h, make_net<T>(c).proj_w, (const T*)c->Binv, (T*)c->Pt, list,
                                            B, count);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return build_g0_t<T>(c, B, list, count);
}

}  // namespace

cudaError_t launch_projector(scale_ctx* c, int B, const int32_t* list, const int32_t* count) {
  return c->fp64 ? project_t<double>(c, B, list, count) : project32(c, B, list, count, true);
}

cudaError_t launch_build_g0(scale_ctx* c, int B, const int32_t* list, const int32_t* count) {
  return c->fp64 ? build_g0_t<double>(c, B, list, count) : project32(c, B, list, count, false);
}

}  // namespace scale
