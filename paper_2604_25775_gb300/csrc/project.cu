// project.cu -- what the rank-r update reads of the inverse: the projector Pt_s = W_s Phi^-1 and
// the feature-independent part of every Slater row's product with the inverse,
// G0t = (M0 + proj_b) Phi^-1 (Sec. II.C, Eq. SMW).
#include <algorithm>

#include "mlp_mma.cuh"
#include "scale_internal.cuh"

namespace scale {

namespace {

// Mixed precision: both are products of the walker's inverse with rows shared by all walkers,
//   out[j][col] = sum_k Binv[j][k] row_col[k],  rows: M0[o] + proj_b (G0t), proj_w[c] of spin s (Pt),
// 2 Ne^2 (2N + 2h) flops a walker and 4 Ne (2N + 2h) bytes written. FP32 FMA ran them as two
// kernels at about a third of its rate; here one kernel takes both on mma.sync as three TF32
// products of a hi/lo split. Every 16 values of k start a fresh accumulator that is then added to
// the FP32 sum with rounding to nearest, so the tensor core's truncating accumulation touches 16
// terms and the sum of Ne terms takes Ne / 16 rounded additions instead of Ne.
//
// CTA: 64 slots x 192 columns, six warps of 32 x 64 (64 accumulators a thread); k in steps of 16,
// both operands split while they are staged (once per CTA, not once per warp) in double-buffered
// shared memory, rows padded to 20 words (conflict-free fragment loads).
//
// From kSplitMinNe electrons on: the split leaves about 2^-23 of each product, an FP32 chain of Ne
// rounded additions grows with Ne. Rms error of single ratios against FP64 (which the rounding
// of the stored inverse bounds from below): Ne = 224 3.2e-7 as a chain, 1.7e-7 here; Ne = 56
// 0.99e-7 as a chain, 1.12e-7 here, so short sums keep the chain.
constexpr int kSplitMinNe = 129;
constexpr int kGM = 64, kGN = 192, kGK = 16, kGLd = kGK + 4, kGThreads = 192;
constexpr int kGBuf = (kGM + kGN) * kGLd;  // words of one buffer's hi (or lo) half

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

__global__ void __launch_bounds__(kGThreads, 2) k_project_tc(ProjArgs a) {
  extern __shared__ __align__(16) uint32_t gsm[];  // [2 buffers][hi, lo][kGM + kGN][kGLd]
  const int Ne = a.Ne, No = a.No, h = a.h;
  const int nrows = a.count ? min(*a.count, a.B) : a.B;
  const int j0 = blockIdx.x * kGM, c0 = blockIdx.y * kGN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int wm = (warp & 1) * 32, wn = (warp >> 1) * 64;  // the warp's tile
  const bool vec = (Ne & 3) == 0 && (reinterpret_cast<uintptr_t>(a.proj_w) & 15) == 0;
  constexpr int kQ = kGK / 4;                             // 4-value pieces of a row
  constexpr int kPer = ((kGM + kGN) * kQ + kGThreads - 1) / kGThreads;
  const int nk = (Ne + kGK - 1) / kGK;
  for (int lrow = blockIdx.z; lrow < nrows; lrow += gridDim.z) {
    const int b = a.list ? a.list[lrow] : lrow;
    if (b < 0) continue;  // uniform
    const float* Bb = a.Binv + (size_t)b * Ne * Ne;
    float4 reg[kPer];
    auto fetch = [&](int kt) {
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int q = tid + u * kGThreads, r = q / kQ, k = kt * kGK + (q % kQ) * 4;
        const float* src = nullptr;
        if (r < kGM) {
          if (j0 + r < Ne) src = Bb + (size_t)(j0 + r) * Ne;
        } else if (r < kGM + kGN) {
          const int col = c0 + r - kGM;
          if (col < No) {
            src = a.M0b + (size_t)col * Ne;
          } else if (col < a.ncol) {
            const int s = (col - No) / h, cc = (col - No) - s * h;
            src = a.proj_w + (size_t)cc * 2 * Ne + (size_t)s * Ne;
          }
        }
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
      uint32_t* hi = gsm + (size_t)buf * 2 * kGBuf;
      uint32_t* lo = hi + kGBuf;
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int q = tid + u * kGThreads, r = q / kQ;
        if (r >= kGM + kGN) continue;
        uint4 vh, vl;
        split_tf32(reg[u].x, vh.x, vl.x);
        split_tf32(reg[u].y, vh.y, vl.y);
        split_tf32(reg[u].z, vh.z, vl.z);
        split_tf32(reg[u].w, vh.w, vl.w);
        *reinterpret_cast<uint4*>(hi + r * kGLd + (q % kQ) * 4) = vh;
        *reinterpret_cast<uint4*>(lo + r * kGLd + (q % kQ) * 4) = vl;
      }
    };
    float acc[2][8][4] = {};
    __syncthreads();  // the previous walker's buffers are consumed
    fetch(0);
    stage(0);
    for (int kt = 0; kt < nk; ++kt) {
      if (kt + 1 < nk) fetch(kt + 1);
      __syncthreads();  // buffer kt & 1 is staged, the other one consumed
      const uint32_t* hi = gsm + (size_t)(kt & 1) * 2 * kGBuf;
      const uint32_t* lo = hi + kGBuf;
      uint32_t ah[2][2][4], al[2][2][4];  // [m tile][k step]
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const int o = (wm + 16 * m + g) * kGLd + 8 * s + t;
          ah[m][s][0] = hi[o];
          ah[m][s][1] = hi[o + 8 * kGLd];
          ah[m][s][2] = hi[o + 4];
          ah[m][s][3] = hi[o + 8 * kGLd + 4];
          al[m][s][0] = lo[o];
          al[m][s][1] = lo[o + 8 * kGLd];
          al[m][s][2] = lo[o + 4];
          al[m][s][3] = lo[o + 8 * kGLd + 4];
        }
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        uint32_t bh[2][2], bl[2][2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const int o = (kGM + wn + 8 * n + g) * kGLd + 8 * s + t;
          bh[s][0] = hi[o];
          bh[s][1] = hi[o + 4];
          bl[s][0] = lo[o];
          bl[s][1] = lo[o + 4];
        }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            mma_tf32(c, al[m][s], bh[s][0], bh[s][1]);
            mma_tf32(c, ah[m][s], bl[s][0], bl[s][1]);
          }
#pragma unroll
          for (int s = 0; s < 2; ++s) mma_tf32(c, ah[m][s], bh[s][0], bh[s][1]);
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[m][n][i] += c[i];
        }
      }
      if (kt + 1 < nk) stage((kt + 1) & 1);
    }
    float* G = a.G0t + (size_t)b * Ne * No;
    float* P = a.Pt + (size_t)b * 2 * Ne * h;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int j = j0 + wm + 16 * m + 8 * half + g;
        if (j >= Ne) continue;
#pragma unroll
        for (int n = 0; n < 8; ++n) {
          const int col = c0 + wn + 8 * n + 2 * t;
          const float v0 = acc[m][n][2 * half], v1 = acc[m][n][2 * half + 1];
          if (col + 1 < No) {  // No is even
            *reinterpret_cast<float2*>(G + (size_t)j * No + col) = make_float2(v0, v1);
          } else {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int q = col + e - No;
              if (q >= 0 && col + e < a.ncol) {
                const int s = q / h;
                P[((size_t)s * Ne + j) * h + q - s * h] = e ? v1 : v0;
              }
            }
          }
        }
      }
  }
}

cudaError_t project_tc(scale_ctx* c, int B, const int32_t* list, const int32_t* count, bool with_pt) {
  const int No = 2 * c->N;
  const ProjArgs a{c->Ne, No, c->h, No + (with_pt ? 2 * c->h : 0), (const float*)c->Binv, (const float*)c->M0b,
                   make_net<float>(c).proj_w, (float*)c->G0t, (float*)c->Pt, list, B, count};
  constexpr size_t smem = sizeof(uint32_t) * 4 * kGBuf;
  const cudaError_t e = cudaFuncSetAttribute(k_project_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid((c->Ne + kGM - 1) / kGM, (a.ncol + kGN - 1) / kGN, count ? std::min(B, 64) : std::min(B, 65535));
  k_project_tc<<<grid, kGThreads, smem, c->stream>>>(a);
  return cudaGetLastError();
}

// ---- FP64 mode, and mixed precision up to kSplitMinNe - 1 electrons ---------------------------
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
    for (int kk = 0; kk < 32; ++kk) {
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
#pragma unroll 4
      for (int kk = 0; kk < 32; ++kk) {
        T x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          x[u] = As[kk][tr + 16 * u];
          y[u] = Ms[kk][tc + 16 * u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] += x[u] * y[v];
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
  if (c->fp64) return project_t<double>(c, B, list, count);
  return c->Ne >= kSplitMinNe ? project_tc(c, B, list, count, true) : project_t<float>(c, B, list, count);
}

cudaError_t launch_build_g0(scale_ctx* c, int B, const int32_t* list, const int32_t* count) {
  if (c->fp64) return build_g0_t<double>(c, B, list, count);
  return c->Ne >= kSplitMinNe ? project_tc(c, B, list, count, false) : build_g0_t<float>(c, B, list, count);
}

}  // namespace scale
