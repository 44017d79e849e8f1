// slater.cu -- Slater matrices in ascending orbital order (Sec. II.B "Orbital Projection"):
//   Phi[a][k] = M0[o_a][k] + proj_b[s*Ne+k] + sum_c H(L)_i[c] proj_w[c][s*Ne+k],
// o_a = s*N + i the a-th occupied orbital, stored as FP64. The load and the refresh project in the
// mode's precision; the full-recompute path projects in FP64 (it divides two determinants,
// where an FP32 rounding of the entries would not cancel as the low-rank update's differences do).
#include <algorithm>

#include "fp64_mma.cuh"
#include "scale_internal.cuh"

namespace scale {

namespace {

constexpr int kPThreads = 256, kPWarps = kPThreads / 32;

// Occupied orbitals of one configuration as bit words over o = s*N + i and the number of set
// bits before each word: words[w], before[w] for w < nw = ceil(2N / 32); returns the total. Every
// thread of the CTA takes part.
__device__ int occupied_words(const int8_t* ob, int N, uint32_t* words, int* before) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (2 * N + 31) / 32;
  for (int w = warp; w < nw; w += kPWarps) {
    const int o = 32 * w + lane, s = o >= N ? 1 : 0;
    const unsigned m = __ballot_sync(0xffffffffu, o < 2 * N && ((ob[o - s * N] >> s) & 1));
    if (lane == 0) words[w] = m;
  }
  __syncthreads();
  if (warp == 0) {
    int base = 0;
    for (int w0 = 0; w0 < nw; w0 += 32) {
      const int mine = w0 + lane < nw ? __popc(words[w0 + lane]) : 0;
      int x = mine;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += y;
      }
      if (w0 + lane < nw) before[w0 + lane] = base + x - mine;
      base += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) before[nw] = base;
  }
  __syncthreads();
  return before[nw];
}

// rows[r - r0] = the r-th occupied orbital for r in [r0, r1) of the ascending list.
__device__ __forceinline__ void occupied_rows(int N, const uint32_t* words, const int* before, int r0, int r1,
                                              uint16_t* rows) {
  for (int o = threadIdx.x; o < 2 * N; o += kPThreads) {
    const uint32_t m = words[o >> 5];
    if (!((m >> (o & 31)) & 1)) continue;
    const int r = before[o >> 5] + __popc(m & ((1u << (o & 31)) - 1u));
    if (r >= r0 && r < r1) rows[r - r0] = (uint16_t)o;
  }
}

__device__ __forceinline__ void zero_matrix(double* P, int n2, int part, int parts) {
  for (int q = part * kPThreads + threadIdx.x; q < n2; q += parts * kPThreads) P[q] = 0.0;
}

// ---- FP32 projection ------------------------------------------------------------------------
// CTA: 32 rows x 128 columns at a time of one sample, 4 x 4 entries per thread; the rows' features
// in shared memory, the weights through L1 (h x 2Ne floats for all samples). Bound by the FP64
// stores: 8 Ne^2 bytes against 2 h Ne^2 flops. The sum runs over c ascending from M0 + proj_b, one
// FMA a term. (One entry per thread took 1.11 ms for 1500 samples of 224 x 224, h = 32; this 0.48.)
constexpr int kPRows = 32, kPCols = 128;

__global__ void __launch_bounds__(kPThreads) k_phi32(Lattice lat, int h, const float* __restrict__ proj_w,
                                                     const float* __restrict__ proj_b, const float* __restrict__ M0,
                                                     const int8_t* __restrict__ occ, const int32_t* __restrict__ list,
                                                     const float* __restrict__ HL, double* __restrict__ phi, int B,
                                                     const int32_t* __restrict__ count) {
  extern __shared__ __align__(16) unsigned char psm[];
  const int N = lat.N, Ne = lat.Ne, nw = (2 * N + 31) / 32;
  float* hs = reinterpret_cast<float*>(psm);                       // [kPRows][h rounded up to 4]
  const int h4 = (h + 3) & ~3;
  uint32_t* words = reinterpret_cast<uint32_t*>(hs + kPRows * h4);
  int* before = reinterpret_cast<int*>(words + nw);
  uint16_t* rows = reinterpret_cast<uint16_t*>(before + nw + 1);   // [kPRows]
  const int tid = threadIdx.x, rg = (tid >> 5) * 4, cg = (tid & 31) * 4;
  const int a0 = blockIdx.x * kPRows, a1 = min(Ne, a0 + kPRows);
  const bool vec = (Ne & 3) == 0 && (reinterpret_cast<uintptr_t>(proj_w) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(proj_b) & 15) == 0;
  const int nrows = count ? min(*count, B) : B;
  for (int e = blockIdx.y; e < nrows; e += gridDim.y) {
    const int b = list ? list[e] : e;
    if (b < 0) continue;  // uniform
    __syncthreads();      // the previous sample's use of shared memory is over
    double* P = phi + (size_t)b * Ne * Ne;
    if (occupied_words(occ + (size_t)b * N, N, words, before) != Ne) {
      zero_matrix(P, Ne * Ne, blockIdx.x, gridDim.x);  // invalid sample: a singular matrix
      continue;
    }
    occupied_rows(N, words, before, a0, a1, rows);
    __syncthreads();
    for (int q = tid; q < kPRows * h4; q += kPThreads) {
      const int r = q / h4, c = q - r * h4;
      float v = 0.f;
      if (r < a1 - a0 && c < h) {
        const int o = rows[r];
        v = HL[((size_t)b * N + (o >= N ? o - N : o)) * h + c];
      }
      hs[q] = v;
    }
    __syncthreads();
    // the thread's four rows share a spin but where a group straddles the two (per-row weights then)
    int o[4], s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      o[u] = rg + u < a1 - a0 ? rows[rg + u] : -1;
      s[u] = o[u] >= N ? 1 : 0;
    }
    if (o[0] < 0) continue;
    bool one = true;
#pragma unroll
    for (int u = 1; u < 4; ++u) one = one && (o[u] < 0 || s[u] == s[0]);
    for (int c0 = 0; c0 < Ne; c0 += kPCols) {
      const int k = c0 + cg;
      if (k >= Ne) continue;
      float acc[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v)
          acc[u][v] = (o[u] >= 0 && k + v < Ne) ? M0[(size_t)o[u] * Ne + k + v] + proj_b[s[u] * Ne + k + v] : 0.f;
      if (one && vec) {
        const float* w = proj_w + (size_t)s[0] * Ne + k;
        for (int c = 0; c < h4; c += 4) {
          float4 x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = *reinterpret_cast<const float4*>(hs + (rg + u) * h4 + c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (c + i >= h) break;
            const float4 wv = *reinterpret_cast<const float4*>(w + (size_t)(c + i) * 2 * Ne);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float xv = i == 0 ? x[u].x : i == 1 ? x[u].y : i == 2 ? x[u].z : x[u].w;
              acc[u][0] = fmaf(xv, wv.x, acc[u][0]);
              acc[u][1] = fmaf(xv, wv.y, acc[u][1]);
              acc[u][2] = fmaf(xv, wv.z, acc[u][2]);
              acc[u][3] = fmaf(xv, wv.w, acc[u][3]);
            }
          }
        }
      } else {
        for (int c = 0; c < h; ++c)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float xv = hs[(rg + u) * h4 + c];
            const float* w = proj_w + (size_t)c * 2 * Ne + s[u] * Ne + k;
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (k + v < Ne) acc[u][v] = fmaf(xv, w[v], acc[u][v]);
          }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (o[u] < 0) continue;
        double* dst = P + (size_t)(a0 + rg + u) * Ne + k;
        if ((Ne & 3) == 0) {
          *reinterpret_cast<double2*>(dst) = make_double2(acc[u][0], acc[u][1]);
          *reinterpret_cast<double2*>(dst + 2) = make_double2(acc[u][2], acc[u][3]);
        } else {
#pragma unroll
          for (int v = 0; v < 4; ++v)
            if (k + v < Ne) dst[v] = acc[u][v];
        }
      }
    }
  }
}

// ---- FP64 projection ------------------------------------------------------------------------
// The products of 16 channels at a time as split FP16 products (fp64_mma.cuh): the FP64 pipe keeps
// two additions and one per 16 channels of every entry instead of h multiply-adds. A CTA keeps the
// slices of one spin's weights for up to kFTiles / KS column tiles (KS = ceil(h / 16) <= 4) in
// shared memory and walks over the samples; per sample the slices of up to 16 / KS strips of 16
// feature rows are built once, then the warps share the (strip, tile) pairs. An entry's sum over 16
// channels that the digits would not carry (split_weak: channels of very different size, large features on
// small weights and the other way round; an infinity, a NaN or an extreme scale) is taken by FP64
// multiply-adds. (h DFMA an entry: 15.05 ms for 1850 configurations of 224 x 224, h = 32; this 1.42.)
constexpr int kFTiles = 28, kFStrips = 16;

template <typename TH>
struct Phi64Args {
  Lattice lat;
  int h, ks, tiles, chunks;  // column tiles per CTA, column chunks per spin
  const double* proj_w;      // [h][2Ne]
  const double* proj_b;
  const double* M0;
  const int8_t* occ;
  const int32_t* list;
  const TH* HL;
  double* phi;
  int B;
  const int32_t* count;
};

struct Phi64Smem {
  size_t bf, af, fe, ae, words, before, rows, total;
};
__host__ __device__ inline Phi64Smem phi64_smem(int N) {
  Phi64Smem s{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 15) & ~size_t(15);
    return at;
  };
  const int nw = (2 * N + 31) / 32;
  s.bf = take((size_t)kFTiles * kSplit * 32 * sizeof(uint2));
  s.af = take((size_t)kFStrips * kSplit * 32 * sizeof(uint4));
  s.fe = take((size_t)kFTiles * 8 * sizeof(int));
  s.ae = take((size_t)kFStrips * 16 * sizeof(int));
  s.words = take(sizeof(uint32_t) * nw);
  s.before = take(sizeof(int) * (nw + 1));
  s.rows = take(sizeof(uint16_t) * 16 * kFStrips);
  s.total = off;
  return s;
}

template <typename TH>
__global__ void __launch_bounds__(kPThreads, 2) k_phi64(Phi64Args<TH> a) {
  extern __shared__ __align__(16) unsigned char psm[];
  const int N = a.lat.N, Ne = a.lat.Ne, h = a.h, KS = a.ks;
  const Phi64Smem S = phi64_smem(N);
  uint2* bf = reinterpret_cast<uint2*>(psm + S.bf);   // [tile][KS][kSplit][32]
  uint4* af = reinterpret_cast<uint4*>(psm + S.af);   // [strip][KS][kSplit][32]
  int* fe = reinterpret_cast<int*>(psm + S.fe);       // [tile][KS][8] column scales
  int* ae = reinterpret_cast<int*>(psm + S.ae);       // [strip][KS][16] row scales
  uint32_t* words = reinterpret_cast<uint32_t*>(psm + S.words);
  int* before = reinterpret_cast<int*>(psm + S.before);
  uint16_t* rows = reinterpret_cast<uint16_t*>(psm + S.rows);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
  const int sp = blockIdx.x / a.chunks, col0 = (blockIdx.x % a.chunks) * a.tiles * 8;
  const int ntile = min(a.tiles, (Ne - col0 + 7) / 8);
  const double* W = a.proj_w + (size_t)sp * Ne;
  const bool vec = (Ne & 1) == 0;
  for (int q = warp; q < ntile * KS; q += kPWarps) {
    const int nt = q / KS, ks = q - nt * KS, col = col0 + 8 * nt + g;
    uint64_t x[4];
    int e = 0, nz = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 16 * ks + 2 * t + (i & 1) + 8 * (i >> 1);
      x[i] = (c < h && col < Ne) ? (uint64_t)__double_as_longlong(W[(size_t)c * 2 * Ne + col]) : 0ull;
      e = max(e, exp_field(x[i]));
      nz |= (x[i] << 1) != 0;
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
      nz |= __shfl_xor_sync(0xffffffffu, nz, off);
    }
    if (t == 0) fe[q * 8 + g] = split_scale(e, nz != 0);
    uint32_t s0[kSplit], s1[kSplit];
    split_pair(split_fixed(x[0], e), split_fixed(x[1], e), s0);
    split_pair(split_fixed(x[2], e), split_fixed(x[3], e), s1);
#pragma unroll
    for (int l = 0; l < kSplit; ++l) bf[(q * kSplit + l) * 32 + lane] = make_uint2(s0[l], s1[l]);
  }
  const int total = a.count ? min(*a.count, a.B) : a.B, per = kFStrips / KS;
  for (int ent = blockIdx.y; ent < total; ent += gridDim.y) {
    const int b = a.list ? a.list[ent] : ent;
    if (b < 0) continue;  // uniform
    __syncthreads();      // weights staged; the previous sample's use of shared memory is over
    double* P = a.phi + (size_t)b * Ne * Ne;
    const int8_t* ob = a.occ + (size_t)b * N;
    if (occupied_words(ob, N, words, before) != Ne) {
      zero_matrix(P, Ne * Ne, blockIdx.x, gridDim.x);
      continue;
    }
    // rows of this spin: [lo, hi) of the ascending list
    const int bw = N >> 5, n_first = before[bw] + __popc(words[bw] & ((1u << (N & 31)) - 1u));
    const int lo = sp ? n_first : 0, hi = sp ? Ne : n_first;
    const TH* Hb = a.HL + (size_t)b * N * h;
    for (int r0 = lo; r0 < hi; r0 += 16 * per) {
      const int nr = min(16 * per, hi - r0), nstrip = (nr + 15) / 16;
      __syncthreads();  // the previous strips are consumed
      occupied_rows(N, words, before, r0, r0 + nr, rows);
      __syncthreads();
      for (int q = warp; q < nstrip * KS; q += kPWarps) {
        const int st = q / KS, ks = q - st * KS;
        uint32_t d[kSplit][4];
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int r = st * 16 + g + 8 * hh;
          const TH* x = r < nr ? Hb + (size_t)(rows[r] - sp * N) * h : nullptr;
          uint64_t v[4];
          int e = 0, nz = 0;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = 16 * ks + 2 * t + (i & 1) + 8 * (i >> 1);
            v[i] = (x && c < h) ? (uint64_t)__double_as_longlong((double)x[c]) : 0ull;
            e = max(e, exp_field(v[i]));
            nz |= (v[i] << 1) != 0;
          }
#pragma unroll
          for (int off = 1; off < 4; off <<= 1) {
            e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
            nz |= __shfl_xor_sync(0xffffffffu, nz, off);
          }
          if (t == 0) ae[q * 16 + g + 8 * hh] = split_scale(e, nz != 0);
          uint32_t s0[kSplit], s1[kSplit];
          split_pair(split_fixed(v[0], e), split_fixed(v[1], e), s0);
          split_pair(split_fixed(v[2], e), split_fixed(v[3], e), s1);
#pragma unroll
          for (int l = 0; l < kSplit; ++l) {
            d[l][hh] = s0[l];
            d[l][2 + hh] = s1[l];
          }
        }
#pragma unroll
        for (int l = 0; l < kSplit; ++l) af[(q * kSplit + l) * 32 + lane] = make_uint4(d[l][0], d[l][1], d[l][2], d[l][3]);
      }
      __syncthreads();
      for (int task = warp; task < nstrip * ntile; task += kPWarps) {
        const int st = task % nstrip, nt = task / nstrip;
        const int ra = st * 16 + g, rb = ra + 8, k = col0 + 8 * nt + 2 * t;
        const int oa = ra < nr ? rows[ra] : -1, obr = rb < nr ? rows[rb] : -1;
        double v[4];  // (ra, k), (ra, k + 1), (rb, k), (rb, k + 1)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int o = i < 2 ? oa : obr, kk = k + (i & 1);
          v[i] = (o >= 0 && kk < Ne) ? a.M0[(size_t)o * Ne + kk] + a.proj_b[sp * Ne + kk] : 0.0;
        }
        for (int ks = 0; ks < KS; ++ks) {
          const uint2* bp = bf + (size_t)(nt * KS + ks) * kSplit * 32 + lane;
          const uint4* ap = af + (size_t)(st * KS + ks) * kSplit * 32 + lane;
          uint2 bq[kSplit];
#pragma unroll
          for (int l = 0; l < kSplit; ++l) bq[l] = bp[l * 32];
          float acc[kSplit][4], wt[4];
#pragma unroll
          for (int l = 0; l < kSplit; ++l)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[l][i] = __uint_as_float(kAccBits);
#pragma unroll
          for (int sa = 0; sa < kSplit; ++sa) {
            const uint4 q = ap[sa * 32];
            const uint32_t aq[4] = {q.x, q.y, q.z, q.w};
            if (sa == 0) split_weight(wt, aq, bq[0]);
#pragma unroll
            for (int sb = 0; sa + sb < kSplit; ++sb) mma_f16(acc[sa + sb], aq, bq[sb].x, bq[sb].y);
          }
          const int2 f = *reinterpret_cast<const int2*>(fe + (nt * KS + ks) * 8 + 2 * t);
          const int ea = ae[(st * KS + ks) * 16 + g], eb = ae[(st * KS + ks) * 16 + g + 8];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int o = i < 2 ? oa : obr, kk = k + (i & 1), er = i < 2 ? ea : eb, fc = (i & 1) ? f.y : f.x;
            if (!split_weak(wt[i], er, fc)) {
              v[i] += split_value(acc, i, er, fc);
            } else if (o >= 0 && kk < Ne) {
              const TH* x = Hb + (size_t)(o - sp * N) * h;
              for (int c = 16 * ks; c < min(h, 16 * ks + 16); ++c) v[i] = fma((double)x[c], W[(size_t)c * 2 * Ne + kk], v[i]);
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
          if ((i ? obr : oa) < 0 || k >= Ne) continue;
          double* dst = P + (size_t)(r0 + (i ? rb : ra)) * Ne + k;
          if (vec) {
            *reinterpret_cast<double2*>(dst) = make_double2(v[i], v[i + 1]);
          } else {
            dst[0] = v[i];
            if (k + 1 < Ne) dst[1] = v[i + 1];
          }
        }
      }
    }
  }
}

template <typename TH>
cudaError_t phi64(scale_ctx* c, const double* proj_w, const double* proj_b, const int8_t* occ, const int32_t* list,
                  const TH* HL, double* phi, int B, const int32_t* count) {
  Phi64Args<TH> a{};
  a.lat = c->lat;
  a.h = c->h;
  a.ks = (c->h + 15) / 16;
  a.tiles = kFTiles / a.ks;
  a.chunks = ((c->Ne + 7) / 8 + a.tiles - 1) / a.tiles;
  a.proj_w = proj_w;
  a.proj_b = proj_b;
  a.M0 = c->M0_64;
  a.occ = occ;
  a.list = list;
  a.HL = HL;
  a.phi = phi;
  a.B = B;
  a.count = count;
  const size_t smem = phi64_smem(c->N).total;
  const cudaError_t e = cudaFuncSetAttribute(k_phi64<TH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // about two resident CTAs per SM, each with its share of the samples
  const int gx = 2 * a.chunks, gy = std::max(1, std::min(B, (2 * 152 + gx - 1) / gx));
  k_phi64<TH><<<dim3(gx, gy), kPThreads, smem, c->stream>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_phi(scale_ctx* c, const int8_t* occ, int B, const int32_t* list, const int32_t* count, const void* HL,
                       double* phi, bool proj64) {
  // the projection's parameters end the flat vector: [h][2Ne], [2Ne]
  const int64_t off_w = c->P - (int64_t)(c->h + 1) * 2 * c->Ne, off_b = c->P - 2 * c->Ne;
  if (c->fp64) return phi64(c, c->params64 + off_w, c->params64 + off_b, occ, list, (const double*)HL, phi, B, count);
  if (proj64) return phi64(c, c->params64 + off_w, c->params64 + off_b, occ, list, (const float*)HL, phi, B, count);
  const int nw = (2 * c->N + 31) / 32;
  const size_t smem = sizeof(float) * kPRows * ((c->h + 3) & ~3) + sizeof(int) * (2 * nw + 1) + 2 * kPRows;
  dim3 grid((c->Ne + kPRows - 1) / kPRows);
  grid.y = std::min(B, count ? listed_ctas(grid.x) : 65535);
  k_phi32<<<grid, kPThreads, smem, c->stream>>>(c->lat, c->h, c->params32 + off_w, c->params32 + off_b, c->M0_32, occ, list,
                                                (const float*)HL, phi, B, count);
  return cudaGetLastError();
}

}  // namespace scale
