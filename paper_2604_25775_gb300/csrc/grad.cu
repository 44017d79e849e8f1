// grad.cu -- per-sample d log|psi| / d theta by a hand-written backward pass.
//
//   d log|det Phi| / d Phi[a][k] = (Phi^-1)[k][a] = Binv[a][k]   (row a = slot a)
//   proj_b[s*Ne+k]     += sum_{slots a of spin s} Binv[a][k]
//   proj_w[c][s*Ne+k]  += sum_{slots a of spin s} H(L)_{i_a}[c] Binv[a][k]
//   dH(L)_i[c]          = sum_{s: (s,i) occupied} Pt[s][slot(s,i)][c]     (Pt = W_s Binv)
//   layer l (out = res*in + act(z), z = b + sum_d K[d]^T in_{i+d}, d over the stencil's taps:
//   the k x k box, or its offsets within L2 distance (k-1)/2, weights stored per tap):
//     dz = dout * act'(z); db = sum_i dz_i; dK[d][ci][co] = sum_i in_{i+d}[ci] dz_i[co]
//     din_j = res*dout_j + sum_d K[d] dz_{j-d}
//   embedding row E_i[n_i] += dH(0)_i.
// The forward is recomputed from the current occupations (all layers stored, or, with
// recompute = 1, only every ceil(sqrt(L))-th layer input, the rest recomputed per segment).
#include <algorithm>
#include <cmath>

#include "scale_internal.cuh"
#include "tcgen05.cuh"

namespace scale {

namespace {

// Forward layer writing explicit output / pre-activation slabs ([B][N][h] each).
template <typename T>
__global__ void k_fwd_layer(Lattice lat, Net<T> net, int l, const int8_t* __restrict__ occ, const T* __restrict__ in,
                            T* __restrict__ out, T* __restrict__ zout) {
  const int h = net.h, N = lat.N;
  const int b = blockIdx.y;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= N * h) return;
  const int i = idx / h, c = idx - i * h;
  const int k = net.ksize[l], r = (k - 1) / 2;
  const int8_t* ob = occ + (size_t)b * N;
  T z = net.bias[l][c];
  int d = 0;  // tap index, row-major over the box
  for (int ky = 0; ky < k; ++ky)
    for (int kx = 0; kx < k; ++kx) {
      if (!stencil_in(net.stencil, k, kx - r, ky - r)) continue;
      const int t = d++;
      const int j = site_off(lat, i, kx - r, ky - r);
      if (j < 0) continue;
      const T* w = net.kernel[l] + (size_t)t * h * h + c;
      const T* x = (l == 0) ? net.embed + ((size_t)(net.per_site ? j * 4 : 0) + (ob[j] & 3)) * h
                            : in + ((size_t)b * N + j) * h;
      for (int ci = 0; ci < h; ++ci) z += x[ci] * w[(size_t)ci * h];
    }
  T self = T(0);
  if (net.resid[l])
    self = (l == 0) ? net.embed[((size_t)(net.per_site ? i * 4 : 0) + (ob[i] & 3)) * h + c] : in[((size_t)b * N + i) * h + c];
  out[(size_t)b * N * h + idx] = self + act_fn<T>(net.act, z);
  zout[(size_t)b * N * h + idx] = z;
}

// Four consecutive elements through the read-only path (16-byte aligned: h % 4 == 0 and
// every slab, table and weight block starts on a multiple of four elements).
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
  const float4 q = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
  const double2 a = __ldg(reinterpret_cast<const double2*>(p)), c = __ldg(reinterpret_cast<const double2*>(p) + 1);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = c.x;
  v[3] = c.y;
}

// Input row of site j for layer l: the embedding row E_j[n_j] for layer 0, else the slab row.
template <typename T>
__device__ __forceinline__ const T* layer_in_row(const Net<T>& net, int l, const int8_t* ob, const T* in_b, int j,
                                                 int h) {
  return l == 0 ? net.embed + ((size_t)(net.per_site ? j * 4 : 0) + (ob[j] & 3)) * h : in_b + (size_t)j * h;
}

// Forward layer (h % 4 == 0), 4 sites x 4 output channels per thread, the same summation order
// as k_fwd_layer (bias, taps in row-major order, input channels ascending).
template <typename T, int HC>
__global__ void k_fwd_tile(Lattice lat, Net<T> net, int l, const int8_t* __restrict__ occ, const T* __restrict__ in,
                           T* __restrict__ out, T* __restrict__ zout) {
  const int h = HC ? HC : net.h, N = lat.N, hq = h >> 2;
  const int b = blockIdx.y;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= ((N + 3) >> 2) * hq) return;
  const int sq = q / hq, c0 = (q - sq * hq) * 4;
  const int k = net.ksize[l], r = (k - 1) / 2;
  const int8_t* ob = occ + (size_t)b * N;
  const T* in_b = in + (size_t)b * N * h;  // unused for layer 0
  T acc[4][4];
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[s][m] = net.bias[l][c0 + m];
  int d = 0;
  for (int ky = 0; ky < k; ++ky)
    for (int kx = 0; kx < k; ++kx) {
      if (!stencil_in(net.stencil, k, kx - r, ky - r)) continue;
      const int t = d++;
      const T* row[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int i = sq * 4 + s;
        const int j = i < N ? site_off(lat, i, kx - r, ky - r) : -1;
        row[s] = j < 0 ? nullptr : layer_in_row(net, l, ob, in_b, j, h);
      }
      const T* w = net.kernel[l] + (size_t)t * h * h + c0;
#pragma unroll
      for (int ci = 0; ci < h; ci += 4) {
        T wv[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) ld4(w + (size_t)(ci + a) * h, wv[a]);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (!row[s]) continue;
          T xv[4];
          ld4(row[s] + ci, xv);
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[s][m] = fma(xv[a], wv[a][m], acc[s][m]);
        }
      }
    }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int i = sq * 4 + s;
    if (i >= N) break;
    const size_t o = ((size_t)b * N + i) * h + c0;
    const T* self = net.resid[l] ? layer_in_row(net, l, ob, in_b, i, h) + c0 : nullptr;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      out[o + m] = (self ? self[m] : T(0)) + act_fn<T>(net.act, acc[s][m]);
      zout[o + m] = acc[s][m];
    }
  }
}

// dK[d][ci][co] = sum_i in_{i+d}[ci] dz_i[co] (h % 8 == 0): one thread per (tap, 4 input
// channels, 8 output channels), sites in ascending order as in k_grad_kernel.
template <typename T, int HC>
__global__ void k_dk_tile(Lattice lat, Net<T> net, int l, int taps, const int8_t* __restrict__ occ,
                          const T* __restrict__ in, const T* __restrict__ dz, int64_t off_k, int64_t P,
                          double* __restrict__ grad) {
  const int b = blockIdx.y;
  const int N = lat.N, h = HC ? HC : net.h, hq = h >> 2, ho = h >> 3, k = net.ksize[l];
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= taps * hq * ho) return;
  const int t = q / (hq * ho), rem = q - t * hq * ho, ci0 = (rem / ho) * 4, co0 = (rem % ho) * 8;
  int dx, dy;
  stencil_tap(net.stencil, k, t, dx, dy);
  const int8_t* ob = occ + (size_t)b * N;
  const T* in_b = in + (size_t)b * N * h;
  const T* dz_b = dz + (size_t)b * N * h + co0;
  T acc[4][8] = {};
  for (int y = 0; y < lat.Ly; ++y) {  // every branch below is uniform over a warp (same tap, site)
    int yy = y + dy;
    if (yy < 0 || yy >= lat.Ly) {
      if (!lat.pbc_y) continue;
      yy = ((yy % lat.Ly) + lat.Ly) % lat.Ly;
    }
#pragma unroll 2
    for (int x = 0; x < lat.Lx; ++x) {
      int xx = x + dx;
      if (xx < 0 || xx >= lat.Lx) {
        if (!lat.pbc_x) continue;
        xx = ((xx % lat.Lx) + lat.Lx) % lat.Lx;
      }
      T xv[4], gv[2][4];
      ld4(layer_in_row(net, l, ob, in_b, yy * lat.Lx + xx, h) + ci0, xv);
      const T* gr = dz_b + (size_t)(y * lat.Lx + x) * h;
      ld4(gr, gv[0]);
      ld4(gr + 4, gv[1]);
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int m = 0; m < 8; ++m) acc[a][m] = fma(xv[a], gv[m >> 2][m & 3], acc[a][m]);
    }
  }
  double* g = grad + (size_t)b * P + off_k + (size_t)t * h * h + co0;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int m = 0; m < 8; ++m) g[(size_t)(ci0 + a) * h + m] = (double)acc[a][m];
}

// din_j[ci] = res*dout_j[ci] + sum_d sum_co K[d][ci][co] dz_{j-d}[co] (h % 4 == 0), 4 sites x
// 4 input channels per thread; KT = the layer's kernel transposed per tap ([d][co][ci]).
template <typename T, int HC>
__global__ void k_din_tile(Lattice lat, Net<T> net, int l, const T* __restrict__ KT, const T* __restrict__ dout,
                           const T* __restrict__ dz, T* __restrict__ din) {
  const int h = HC ? HC : net.h, N = lat.N, hq = h >> 2;
  const int b = blockIdx.y;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= ((N + 3) >> 2) * hq) return;
  const int sq = q / hq, c0 = (q - sq * hq) * 4;
  const int k = net.ksize[l], r = (k - 1) / 2;
  const size_t base = (size_t)b * N * h;
  T acc[4][4];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int j = sq * 4 + s;
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[s][m] = (net.resid[l] && j < N) ? dout[base + (size_t)j * h + c0 + m] : T(0);
  }
  int d = 0;
  for (int ky = 0; ky < k; ++ky)
    for (int kx = 0; kx < k; ++kx) {
      if (!stencil_in(net.stencil, k, kx - r, ky - r)) continue;
      const int t = d++;
      const T* g[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int j = sq * 4 + s;
        const int i = j < N ? site_off(lat, j, -(kx - r), -(ky - r)) : -1;  // site i with i + d = j
        g[s] = i < 0 ? nullptr : dz + base + (size_t)i * h;
      }
      const T* w = KT + (size_t)t * h * h + c0;
#pragma unroll
      for (int co = 0; co < h; co += 4) {
        T wv[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) ld4(w + (size_t)(co + a) * h, wv[a]);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (!g[s]) continue;
          T gv[4];
          ld4(g[s] + co, gv);
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[s][m] = fma(wv[a][m], gv[a], acc[s][m]);
        }
      }
    }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int j = sq * 4 + s;
    if (j >= N) break;
#pragma unroll
    for (int m = 0; m < 4; ++m) din[base + (size_t)j * h + c0 + m] = acc[s][m];
  }
}

// ---- one sample's slabs staged in shared memory (up to kStagedSites sites) ------------------
// CTA per sample: the rows a layer reads (its input, the embedding rows for layer 0, or dz) copied
// to shared memory once with 16-byte loads, and the site table nbr[t][i] (the site reached
// from i by tap t; -1 past an open edge). The summation order is that of the kernels above, so the
// results are the same. Row stride h plus one 16-byte vector: rows read by the lanes of one warp
// then lie in different banks (with stride h four site groups hit the same ones). The weights come
// through shared memory in chunks ahead of their use: all walkers' CTAs run in one wave and step through
// the taps together, so each read of a weight row through L1 waited for L2.
// What bounds them: 512 walkers are 3.4 CTAs per SM, so staging, sums and output of a layer follow one
// another with little to overlap (sums about half of it). Per layer of the 16x4 cylinder, 512 walkers:
// forward 45 -> 25 us, input gradient with dz 53 -> 25, dK 50 -> 29 (of which the FP64 output of
// 38 MB takes 7).
constexpr int kStagedSites = 128;
constexpr int kConvThreads = 256;
// Sites per thread of the convolutions and input rows per thread of dK, by 8 channels. In FP32 a
// 16-byte load from shared memory occupies the SM for four cycles and a warp's FMA for a quarter:
// 2 x 4 sums per thread ran at the loads' rate (33 us a layer of the 16x4 cylinder, 512 walkers; the
// FMAs alone take 8), 2 x 8 take 25 and 4 x 8 29 (two warps per walker hide too little). In FP64 the
// FP64 pipe is the limit and one site per thread keeps more warps (an update of 8x8, 200 walkers:
// 1.42 ms, with two sites 1.55, with four 1.73). dK by 8 x 8: 31 us a layer against 29 by 4 x 8.
template <typename T>
constexpr int kConvSites = sizeof(T) == 4 ? 2 : 1;
constexpr int kDkRows = 4;
template <typename T>
constexpr int kDkThreads = sizeof(T) == 4 ? 640 : 288;  // registers for a full block
__host__ __device__ constexpr int bias_threads(int h) { return (h + 31) / 32 * 32; }
// The conversion to FP64 in integers (the FP64 pipe is 64 times narrower): exponent and mantissa of
// a normal number; the rest by the instruction.
__device__ __forceinline__ double to_double(float x) {
  const uint32_t u = __float_as_uint(x), e = u & 0x7f800000u;
  if (e == 0 || e == 0x7f800000u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ void lds4(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
  v[3] = q.w;
}
__device__ __forceinline__ void lds4(const double* p, double (&v)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p), c = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x;
  v[1] = a.y;
  v[2] = c.x;
  v[3] = c.y;
}

// The table of a layer lies in device memory (k_grad_prep; with the divisions per CTA the staging
// took longer than the sums), padded to whole 16-byte pieces.
__host__ __device__ constexpr int nbr_size(int N, int taps) { return (N * taps + 7) & ~7; }
__device__ __forceinline__ void stage_nbr(const int16_t* __restrict__ table, int n, int16_t* nbr) {
  for (int q = threadIdx.x * 8; q < n; q += blockDim.x * 8) tc::cp_async16(nbr + q, table + q);
}
__device__ __forceinline__ void sts4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void sts4(double* p, const double (&v)[4]) {
  *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}

template <typename T>
__host__ __device__ constexpr int staged_ld(int h) {
  return h + (int)(16 / sizeof(T));
}
// Bytes of shared memory of the staged kernels: [slabs][N][staged_ld] rows and the [taps][N] table.
template <typename T>
inline size_t staged_bytes(int N, int h, int taps, int slabs) {
  return (size_t)slabs * N * staged_ld<T>(h) * sizeof(T) + (size_t)nbr_size(N, taps) * sizeof(int16_t);
}

// Weight rows of one tap that are in shared memory at a time: at most 8 KB, a divisor of h.
constexpr int kWStages = 3;
template <typename T>
__host__ __device__ constexpr int conv_rows(int h) {
  int r = h;
  while (r > 4 && ((size_t)r * h * sizeof(T) > 8192 || h % r || r % 4)) r -= 4;
  return r;
}
template <typename T>
inline size_t conv_bytes(int N, int h, int taps) {
  return staged_bytes<T>(N, h, taps, 1) + (size_t)kWStages * conv_rows<T>(h) * h * sizeof(T);
}

// SM sites x CM channels per thread of
//   BACK = 0: out = res in + act(z), zout = z = b + sum_d W[d]^T in_{i+d}     (W = kernel)
//   BACK = 1: out = res dout + sum_d W[d]^T dz_{i-d}, dz = dout act'(z)       (W = kernel transposed),
//             kept for dK, and the bias gradient sum_i dz_i by the block's last threads
// a: in, or dout; z: zout (written), or z (read).
template <typename T, int HC, int BACK>
__global__ void __launch_bounds__(kConvThreads + 64, 2)
    k_conv_staged(Lattice lat, Net<T> net, int l, int taps, const int16_t* __restrict__ table,
                  const T* __restrict__ W, const int8_t* __restrict__ occ, const T* __restrict__ a, T* __restrict__ z, T* __restrict__ out, T* __restrict__ dz, int64_t off_b, int64_t P,
                  double* __restrict__ grad) {
  constexpr int SM = kConvSites<T>, CM = 8;
  extern __shared__ __align__(16) unsigned char gsm[];
  const int h = HC ? HC : net.h, N = lat.N, hq = h / CM, ld = staged_ld<T>(h);
  const int R = conv_rows<T>(h), per = h / R, chunks = taps * per;
  const int b = blockIdx.x;
  T* ws = reinterpret_cast<T*>(gsm);  // [kWStages][R][h] weight rows
  T* xs = ws + (size_t)kWStages * R * h;
  int16_t* nbr = reinterpret_cast<int16_t*>(xs + (size_t)N * ld);
  const int8_t* ob = occ + (size_t)b * N;
  const size_t base = (size_t)b * N * h;
  constexpr int V = 16 / sizeof(T);
  auto load = [&](int k) {  // one commit group per call, empty past the last chunk
    if (k < chunks)
      for (int q = threadIdx.x * V; q < R * h; q += blockDim.x * V)
        tc::cp_async16(ws + (size_t)(k % kWStages) * R * h + q, W + (size_t)k * R * h + q);
    tc::cp_async_commit();
  };
  const int tiles = ((N + SM - 1) / SM) * hq, workers = BACK ? blockDim.x - bias_threads(h) : blockDim.x;
  const int cb = BACK ? (int)threadIdx.x - workers : -1, bsites = (N + chunks - 1) / chunks;
  double db = 0.0;
  for (int q0 = 0; q0 < tiles; q0 += workers) {
    if (q0 == 0) stage_nbr(table, nbr_size(N, taps), nbr);  // in the group of the first chunk
    for (int k = 0; k < kWStages - 1; ++k) load(k);
    if (q0 == 0) {
#pragma unroll 4
      for (int q = threadIdx.x * 4; q < N * h; q += blockDim.x * 4) {
        const int i = q / h, c = q - i * h;
        T v[4];
        if constexpr (BACK) {
          T zv[4];
          ld4(a + base + q, v);
          ld4(z + base + q, zv);
#pragma unroll
          for (int m = 0; m < 4; ++m) v[m] *= act_grad<T>(net.act, zv[m]);
          sts4(dz + base + q, v);
        } else {
          ld4(layer_in_row(net, l, ob, a + base, i, h) + c, v);
        }
        sts4(xs + i * ld + c, v);
      }
    }
    const int q = q0 + threadIdx.x;
    // i0 = N: no sites (a thread past the tiles, or of the bias sums)
    const int i0 = q < tiles && (int)threadIdx.x < workers ? (q / hq) * SM : N, c0 = (q % hq) * CM;
    T acc[SM][CM];
#pragma unroll
    for (int s = 0; s < SM; ++s)
#pragma unroll
      for (int m = 0; m < CM; ++m) {
        if constexpr (BACK)
          acc[s][m] = (net.resid[l] && i0 + s < N) ? a[base + (size_t)(i0 + s) * h + c0 + m] : T(0);
        else
          acc[s][m] = net.bias[l][c0 + m];
      }
    for (int k = 0; k < chunks; ++k) {
      tc::cp_async_wait<kWStages - 2>();
      __syncthreads();  // chunk k has landed for every thread; chunk k - 1 is no longer read
      load(k + kWStages - 1);
      if (BACK && q0 == 0 && cb >= 0 && cb < h)  // a few sites per chunk, in order
        for (int i = k * bsites; i < min(N, (k + 1) * bsites); ++i) db += to_double(xs[i * ld + cb]);
      const int t = k / per, ci0 = (k - t * per) * R;
      int row[SM], n_in = 0;
#pragma unroll
      for (int s = 0; s < SM; ++s) {
        row[s] = i0 + s < N ? nbr[t * N + i0 + s] : -1;
        n_in += row[s] >= 0;
      }
      const T* w = ws + (size_t)(k % kWStages) * R * h + c0;
      const T* x = xs + ci0;
      auto step = [&](int ci, bool all) {
        T xv[SM][4];
#pragma unroll
        for (int s = 0; s < SM; ++s)
          if (all || row[s] >= 0) lds4(x + row[s] * ld + ci, xv[s]);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          T wv[CM];
#pragma unroll
          for (int m = 0; m < CM; m += 4) lds4(w + (ci + r) * h + m, reinterpret_cast<T(&)[4]>(wv[m]));
#pragma unroll
          for (int s = 0; s < SM; ++s) {
            if (!all && row[s] < 0) continue;
#pragma unroll
            for (int m = 0; m < CM; ++m) acc[s][m] = fma(xv[s][r], wv[m], acc[s][m]);
          }
        }
      };
      if (n_in == SM) {
#pragma unroll 2
        for (int ci = 0; ci < R; ci += 4) step(ci, true);
      } else if (n_in) {
#pragma unroll 1
        for (int ci = 0; ci < R; ci += 4) step(ci, false);
      }
    }
#pragma unroll
    for (int s = 0; s < SM; ++s) {
      const int i = i0 + s;
      if (i >= N) break;
      const size_t o = base + (size_t)i * h + c0;
#pragma unroll
      for (int m = 0; m < CM; m += 4) {
        T(&v)[4] = reinterpret_cast<T(&)[4]>(acc[s][m]);
        if constexpr (!BACK) {
          T r[4] = {};
          if (net.resid[l]) lds4(xs + i * ld + c0 + m, r);
#pragma unroll
          for (int e = 0; e < 4; ++e) r[e] += act_fn<T>(net.act, v[e]);
          sts4(z + o + m, v);
          sts4(out + o + m, r);
        } else {
          sts4(out + o + m, v);
        }
      }
    }
    __syncthreads();  // the weight rows of this pass are no longer read
  }
  if (BACK && cb >= 0 && cb < h) grad[(size_t)b * P + off_b + cb] = db;
}

// dK: RI input x 8 output channels of a tap per thread.
// U sites of a tap at a time, their loads in flight before the first use. A thread's eight columns
// are co = m h/8 + its group, so that the lanes of a store write neighbouring words; the columns of dz
// lie in that order in shared memory.
template <typename T, int HC>
__global__ void __launch_bounds__(kDkThreads<T>)
    k_dk_staged(Lattice lat, Net<T> net, int l, int taps, const int16_t* __restrict__ table,
                const int8_t* __restrict__ occ, const T* __restrict__ in, const T* __restrict__ dz, int64_t off_k, int64_t P,
                double* __restrict__ grad) {
  constexpr int RI = kDkRows, U = 4;
  extern __shared__ __align__(16) unsigned char gsm[];
  const int N = lat.N, h = HC ? HC : net.h, hq = h / RI, ho = h >> 3, ld = staged_ld<T>(h);
  const int b = blockIdx.x;
  T* xs = reinterpret_cast<T*>(gsm);
  T* gs = xs + (size_t)N * ld;
  int16_t* nbr = reinterpret_cast<int16_t*>(gs + (size_t)N * ld);
  const int8_t* ob = occ + (size_t)b * N;
  const size_t base = (size_t)b * N * h;
  stage_nbr(table, nbr_size(N, taps), nbr);
  tc::cp_async_commit();
#pragma unroll 4
  for (int q = threadIdx.x * 4; q < N * h; q += blockDim.x * 4) {
    const int i = q / h, c = q - i * h;
    T v[4], gv[4];
    ld4(layer_in_row(net, l, ob, in + base, i, h) + c, v);
    ld4(dz + base + q, gv);
    sts4(xs + i * ld + c, v);
#pragma unroll
    for (int m = 0; m < 4; ++m) gs[i * ld + ((c + m) % ho) * 8 + (c + m) / ho] = gv[m];
  }
  tc::cp_async_wait<0>();
  __syncthreads();
  for (int q = threadIdx.x; q < taps * hq * ho; q += blockDim.x) {
    const int t = q / (hq * ho), rem = q - t * hq * ho, ci0 = (rem / ho) * RI, cg = rem % ho;
    T acc[RI][8] = {};
    const int16_t* nt = nbr + t * N;
    const T* x = xs + ci0;
    const T* gp = gs + cg * 8;
    int i = 0;
    for (; i + U <= N; i += U) {
      T xv[U][RI], gv[U][8];
      int j[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        j[u] = nt[i + u];
#pragma unroll
        for (int a = 0; a < RI; a += 4)
          lds4(x + (j[u] < 0 ? 0 : j[u]) * ld + a, reinterpret_cast<T(&)[4]>(xv[u][a]));
        lds4(gp + (i + u) * ld, reinterpret_cast<T(&)[4]>(gv[u][0]));
        lds4(gp + (i + u) * ld + 4, reinterpret_cast<T(&)[4]>(gv[u][4]));
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (j[u] < 0) continue;
#pragma unroll
        for (int a = 0; a < RI; ++a)
#pragma unroll
          for (int m = 0; m < 8; ++m) acc[a][m] = fma(xv[u][a], gv[u][m], acc[a][m]);
      }
    }
    for (; i < N; ++i) {
      const int j = nt[i];
      if (j < 0) continue;
#pragma unroll
      for (int a = 0; a < RI; ++a)
#pragma unroll
        for (int m = 0; m < 8; ++m) acc[a][m] = fma(x[j * ld + a], gp[i * ld + m], acc[a][m]);
    }
    double* g = grad + (size_t)b * P + off_k + (size_t)t * h * h + cg;
#pragma unroll
    for (int a = 0; a < RI; ++a)
#pragma unroll
      for (int m = 0; m < 8; ++m) g[(size_t)(ci0 + a) * h + m * ho] = to_double(acc[a][m]);
  }
}

// Projection gradients and dH(L).
template <typename T>
__global__ void k_grad_proj(Lattice lat, Net<T> net, const int32_t* __restrict__ orb_of_slot,
                            const int32_t* __restrict__ slot_of_orb, const T* __restrict__ Binv,
                            const T* __restrict__ Pt, const T* __restrict__ HLr, int64_t off_pw, int64_t off_pb,
                            int64_t P, double* __restrict__ grad, T* __restrict__ dH) {
  const int b = blockIdx.x;
  const int N = lat.N, Ne = lat.Ne, h = net.h;
  const T* Bb = Binv + (size_t)b * Ne * Ne;
  const T* Hb = HLr + (size_t)b * N * h;
  double* g = grad + (size_t)b * P;
  const int32_t* os = orb_of_slot + (size_t)b * Ne;
  const int groups = (h + 7) / 8 + 1;  // eight channels each; the last is the bias
  for (int q = threadIdx.x; q < 2 * Ne * groups; q += blockDim.x) {
    const int s = q / (Ne * groups);
    const int rem = q - s * Ne * groups;
    const int cg = rem / Ne, k = rem - cg * Ne;
    if (cg == groups - 1) {
      T acc = T(0);  // the mode's precision, as the layer gradients
      for (int a = 0; a < Ne; ++a) {
        const int i = os[a] - s * N;
        if (i >= 0 && i < N) acc += Bb[(size_t)a * Ne + k];  // else a slot of the other spin
      }
      g[off_pb + s * Ne + k] = to_double(acc);
      continue;
    }
    const int c0 = cg * 8, nc = min(8, h - c0);
    T acc[8] = {};
    for (int a = 0; a < Ne; ++a) {
      const int i = os[a] - s * N;
      if (i < 0 || i >= N) continue;
      const T bv = Bb[(size_t)a * Ne + k];
      const T* hr = Hb + (size_t)i * h + c0;
      if (h % 4 == 0) {
        T v[4];
        ld4(hr, v);
#pragma unroll
        for (int m = 0; m < 4; ++m) acc[m] += v[m] * bv;
        if (nc > 4) {
          ld4(hr + 4, v);
#pragma unroll
          for (int m = 0; m < 4; ++m) acc[4 + m] += v[m] * bv;
        }
      } else {
#pragma unroll
        for (int m = 0; m < 8; ++m)
          if (m < nc) acc[m] += hr[m] * bv;
      }
    }
#pragma unroll
    for (int m = 0; m < 8; ++m)
      if (m < nc) g[off_pw + (size_t)(c0 + m) * 2 * Ne + s * Ne + k] = to_double(acc[m]);
  }
  const int32_t* so = slot_of_orb + (size_t)b * 2 * N;
  const T* Pb = Pt + (size_t)b * 2 * Ne * h;
  for (int q = threadIdx.x; q < N * h; q += blockDim.x) {
    const int i = q / h, c = q - i * h;
    T acc = T(0);
    for (int s = 0; s < 2; ++s) {
      const int a = so[s * N + i];
      if (a >= 0) acc += Pb[((size_t)s * Ne + a) * h + c];
    }
    dH[(size_t)b * N * h + q] = acc;
  }
}

// dz = dout * act'(z), and the bias gradient.
template <typename T>
__global__ void k_grad_dz(Lattice lat, Net<T> net, int l, const T* __restrict__ dout, const T* __restrict__ z,
                          T* __restrict__ dz, int64_t off_b, int64_t P, double* __restrict__ grad) {
  const int b = blockIdx.x;
  const int N = lat.N, h = net.h;
  for (int q = threadIdx.x; q < N * h; q += blockDim.x)
    dz[(size_t)b * N * h + q] = dout[(size_t)b * N * h + q] * act_grad<T>(net.act, z[(size_t)b * N * h + q]);
  __syncthreads();
  for (int c = threadIdx.x; c < h; c += blockDim.x) {
    double acc = 0.0;
    for (int i = 0; i < N; ++i) acc += (double)dz[((size_t)b * N + i) * h + c];
    grad[(size_t)b * P + off_b + c] = acc;
  }
}

// dK[d][ci][co] = sum_i in_{i+d}[ci] dz_i[co], accumulated in the mode's precision (FP32 in
// mixed precision: an FP64 sum would run on GB300's few FP64 units for no accuracy the FP32
// activations carry)
template <typename T>
__global__ void k_grad_kernel(Lattice lat, Net<T> net, int l, int taps, const int8_t* __restrict__ occ,
                              const T* __restrict__ in, const T* __restrict__ dz, int64_t off_k, int64_t P,
                              double* __restrict__ grad) {
  const int b = blockIdx.y;
  const int N = lat.N, h = net.h, k = net.ksize[l];
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= taps * h * h) return;
  const int d = q / (h * h), rem = q - d * h * h, ci = rem / h, co = rem - ci * h;
  int dx, dy;
  stencil_tap(net.stencil, k, d, dx, dy);
  const int8_t* ob = occ + (size_t)b * N;
  T acc = T(0);
  for (int i = 0; i < N; ++i) {
    const int j = site_off(lat, i, dx, dy);
    if (j < 0) continue;
    const T xin = (l == 0) ? net.embed[((size_t)(net.per_site ? j * 4 : 0) + (ob[j] & 3)) * h + ci]
                           : in[((size_t)b * N + j) * h + ci];
    acc += xin * dz[((size_t)b * N + i) * h + co];
  }
  grad[(size_t)b * P + off_k + q] = (double)acc;
}

// KT[d][co][ci] = K[d][ci][co] of every layer (blockIdx.y), one after another (the loads of
// k_grad_din are then consecutive across the lanes of a warp), and, with `table`, each layer's site
// tables: [2][taps][N], by i + d and by i - d.
template <typename T>
__global__ void k_grad_prep(Lattice lat, Net<T> net, T* __restrict__ KT, int16_t* __restrict__ table) {
  const int h = net.h, l = blockIdx.y, total = stencil_taps(net.stencil, net.ksize[l]) * h * h;
  const T* K = net.kernel[l];
  for (int m = 0; m < l; ++m) KT += (size_t)stencil_taps(net.stencil, net.ksize[m]) * h * h;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < total; q += gridDim.x * blockDim.x) {
    const int d = q / (h * h), rem = q - d * h * h, ci = rem / h, co = rem - ci * h;
    KT[(size_t)d * h * h + (size_t)co * h + ci] = K[q];
  }
  if (!table) return;
  const int N = lat.N, taps = total / (h * h), k = net.ksize[l];
  for (int m = 0; m < l; ++m) table += 2 * nbr_size(N, stencil_taps(net.stencil, net.ksize[m]));
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < 2 * N * taps; q += gridDim.x * blockDim.x) {
    const int neg = q >= N * taps, e = q - neg * N * taps, t = e / N, i = e - t * N;
    int dx, dy;
    stencil_tap(net.stencil, k, t, dx, dy);
    table[neg * nbr_size(N, taps) + e] = (int16_t)site_off(lat, i, neg ? -dx : dx, neg ? -dy : dy);
  }
}

// din_j[ci] = res*dout_j[ci] + sum_d sum_co K[d][ci][co] dz_{j-d}[co]; KT = the layer's
// kernel transposed per tap ([d][co][ci]).
template <typename T>
__global__ void k_grad_din(Lattice lat, Net<T> net, int l, const T* __restrict__ KT, const T* __restrict__ dout,
                           const T* __restrict__ dz, T* __restrict__ din) {
  const int b = blockIdx.y;
  const int N = lat.N, h = net.h, k = net.ksize[l], r = (k - 1) / 2;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= N * h) return;
  const int j = q / h, ci = q - j * h;
  T acc = net.resid[l] ? dout[(size_t)b * N * h + q] : T(0);
  int d = 0;  // tap index, row-major over the box
  for (int ky = 0; ky < k; ++ky)
    for (int kx = 0; kx < k; ++kx) {
      if (!stencil_in(net.stencil, k, kx - r, ky - r)) continue;
      const int t = d++;
      const int i = site_off(lat, j, -(kx - r), -(ky - r));  // site i with i + d = j
      if (i < 0) continue;
      const T* w = KT + (size_t)t * h * h + ci;
      const T* g = dz + ((size_t)b * N + i) * h;
      for (int co = 0; co < h; ++co) acc += w[(size_t)co * h] * g[co];
    }
  din[(size_t)b * N * h + q] = acc;
}

// Embedding rows: E_i[n_i] (per-site tables) or E[n] summed over sites (shared table).
template <typename T>
__global__ void k_grad_embed(Lattice lat, Net<T> net, const int8_t* __restrict__ occ, const T* __restrict__ dH0,
                             int64_t P, double* __restrict__ grad) {
  const int b = blockIdx.x;
  const int N = lat.N, h = net.h;
  const int8_t* ob = occ + (size_t)b * N;
  double* g = grad + (size_t)b * P;
  if (net.per_site) {  // every row written: the three rows of a site's other states get 0
    for (int q = threadIdx.x; q < N * 4 * h; q += blockDim.x) {
      const int i = q / (4 * h), rem = q - i * 4 * h, n = rem / h, c = rem - n * h;
      g[q] = n == (ob[i] & 3) ? (double)dH0[((size_t)b * N + i) * h + c] : 0.0;
    }
  } else {
    for (int q = threadIdx.x; q < 4 * h; q += blockDim.x) {
      const int n = q / h, c = q - n * h;
      double acc = 0.0;
      for (int i = 0; i < N; ++i)
        if (ob[i] == n) acc += (double)dH0[((size_t)b * N + i) * h + c];
      g[q] = acc;
    }
  }
}

__global__ void k_nan_bad(int B, int64_t P, const int32_t* __restrict__ status, double* __restrict__ grad) {
  const int b = blockIdx.x;
  if (!(status[b] & (SCALE_SAMPLE_BAD_COUNT | SCALE_SAMPLE_DOUBLE_OCC | SCALE_SAMPLE_SINGULAR))) return;
  for (int64_t q = threadIdx.x; q < P; q += blockDim.x) grad[(size_t)b * P + q] = CUDART_NAN;
}

// One CTA per sample of `block` threads with `smem` bytes of staged slabs.
template <typename... KA, typename... A>
cudaError_t staged_launch(void (*kern)(KA...), int B, int block, size_t smem, cudaStream_t st, A... args) {
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<B, block, smem, st>>>(args...);
  return cudaGetLastError();
}
// Threads for `work` items: one each up to `most`, beyond that each thread loops over its share.
inline int staged_block(int work, int most) { return std::min(most, std::max(32, (work + 31) / 32 * 32)); }

constexpr size_t kGradSmemMax = 96 * 1024;  // staged slabs up to this size (a few CTAs per SM)

template <typename T>
cudaError_t grad_t(scale_ctx* c, double* grad, int recompute) {
  const Net<T> net = make_net<T>(c);
  const int B = c->B, N = c->N, h = c->h, L = c->L;
  const size_t slab = (size_t)B * N * h;  // elements of one layer slab
  const bool tiled = h % 8 == 0;          // the register-tiled kernels (vector loads of 4)
  int max_taps = 1;
  for (int l = 0; l < L; ++l) max_taps = std::max(max_taps, stencil_taps(net.stencil, net.ksize[l]));
  // one sample's slabs staged in shared memory on small lattices; at 256 sites the 73 KB of slabs
  // per sample cost more than the L1-served kernels (measured). One CTA a sample: in FP64, where the
  // FP64 pipe of the SMs in use is the limit, a sample of more tiles than a CTA's threads is spread over
  // several CTAs by the L1-served kernels while fewer than half of the SMs had one (us, staged / L1-served: 66
  // sites, h = 32, 64 walkers 1519 / 1236, 100 walkers 1517 / 1798; 128 sites, h = 40, 64 walkers 3515 / 2593,
  // 152 walkers 3541 / 3962; 64 sites, h = 24, 32 walkers 754 / 962).
  const bool spread = sizeof(T) == 8 && B <= 76 && (N + kConvSites<T> - 1) / kConvSites<T> * (h / 8) > kConvThreads;
  const bool staged = tiled && !spread && N <= kStagedSites && staged_bytes<T>(N, h, max_taps, 2) <= kGradSmemMax &&
                      conv_bytes<T>(N, h, max_taps) <= kGradSmemMax + 32 * 1024;
  // stored: every layer's input and pre-activation kept from the one forward pass; recompute:
  // only every stride-th layer input, each segment's forward recomputed during the backward
  const int stride = recompute ? std::max(1, (int)std::ceil(std::sqrt((double)L))) : 1;
  const int n_ck = (L + stride - 1) / stride;
  // slabs: checkpoints (layer inputs at multiples of stride), segment H and z (stored: all L
  // pre-activations, no segment H), H(L), dH ping-pong (2), dz (1)
  const size_t n_seg = recompute ? (size_t)(stride + 1) + stride : (size_t)L;
  size_t ktaps = 0;  // transposed kernels of every layer
  for (int l = 0; l < L; ++l) ktaps += (size_t)stencil_taps(net.stencil, net.ksize[l]) * h * h;
  size_t ntab = 0;  // site tables of the staged kernels
  for (int l = 0; staged && l < L; ++l) ntab += 2 * (size_t)nbr_size(N, stencil_taps(net.stencil, net.ksize[l]));
  const size_t need = sizeof(T) * (slab * (n_ck + n_seg + 4) + ktaps) + sizeof(int16_t) * ntab;
  if (need > c->grad_scratch_bytes) {
    if (c->grad_scratch) cudaFree(c->grad_scratch);
    c->grad_scratch = nullptr;
    c->grad_scratch_bytes = 0;
    cudaError_t e = cudaMalloc(&c->grad_scratch, need);
    if (e != cudaSuccess) return e;
    c->grad_scratch_bytes = need;
  }
  T* base = (T*)c->grad_scratch;
  T* ck = base;                          // [n_ck] slabs: input of layer m*stride (slab 0 unused)
  T* seg = ck + (size_t)n_ck * slab;     // recompute: segH [stride+1], segZ [stride]; stored: Z [L]
  T* segH = seg;
  T* segZ = recompute ? seg + (size_t)(stride + 1) * slab : seg;
  T* HL = seg + n_seg * slab;
  T* dA = HL + slab;
  T* dB = dA + slab;
  T* dZ = dB + slab;
  T* KT = dZ + slab;  // [sum over layers of taps * h * h]
  T* KTl[kMaxLayers];
  int16_t* table = reinterpret_cast<int16_t*>(KT + ktaps);
  const int16_t* tabl[kMaxLayers];
  {
    size_t o = 0, ot = 0;
    for (int l = 0; l < L; ++l) {
      const int tl = stencil_taps(net.stencil, net.ksize[l]);
      KTl[l] = KT + o;
      tabl[l] = table + ot;
      ot += 2 * nbr_size(N, tl);
      o += (size_t)tl * h * h;
    }
    k_grad_prep<T><<<dim3((max_taps * h * h + 255) / 256, L), 256, 0, c->stream>>>(c->lat, net, KT,
                                                                                  staged ? table : nullptr);
  }
  // offsets (every parameter is written below: no clearing pass over the B x P gradients)
  int64_t off = (int64_t)(c->arch.per_site_embed ? N : 1) * 4 * h;
  int64_t offK[kMaxLayers], offB[kMaxLayers];
  int taps[kMaxLayers];
  for (int l = 0; l < L; ++l) {
    taps[l] = stencil_taps(net.stencil, net.ksize[l]);
    offK[l] = off;
    off += (int64_t)taps[l] * h * h;
    offB[l] = off;
    off += h;
  }
  const int64_t off_pw = off, off_pb = off + (int64_t)h * 2 * c->Ne;
  const dim3 gridL((N * h + 127) / 128, B), gridT((((N + 3) / 4) * (h / 4) + 127) / 128, B);
  // the tiled kernels with the width as a compile-time constant where it is a common one
#define SCALE_GRAD_TILED(KERNEL, GRID, ...)                                                \
  switch (h) {                                                                             \
    case 8: KERNEL<T, 8><<<GRID, 128, 0, c->stream>>>(__VA_ARGS__); break;                 \
    case 16: KERNEL<T, 16><<<GRID, 128, 0, c->stream>>>(__VA_ARGS__); break;               \
    case 32: KERNEL<T, 32><<<GRID, 128, 0, c->stream>>>(__VA_ARGS__); break;               \
    case 64: KERNEL<T, 64><<<GRID, 128, 0, c->stream>>>(__VA_ARGS__); break;               \
    default: KERNEL<T, 0><<<GRID, 128, 0, c->stream>>>(__VA_ARGS__);                       \
  }
#define SCALE_GRAD_STAGED(CALL)     \
  switch (h) {                      \
    case 8: CALL(8); break;         \
    case 16: CALL(16); break;       \
    case 32: CALL(32); break;       \
    case 64: CALL(64); break;       \
    default: CALL(0);               \
  }
  const int conv_block = staged_block(((N + kConvSites<T> - 1) / kConvSites<T>) * (h / 8), kConvThreads);
  cudaError_t e = cudaSuccess;
  auto fwd = [&](int l, const T* in, T* out, T* z) {
    if (staged) {
      const int tl = stencil_taps(net.stencil, net.ksize[l]);
#define SCALE_CALL(HC)                                                                                                \
  e = staged_launch(k_conv_staged<T, HC, 0>, B, conv_block, conv_bytes<T>(N, h, tl), c->stream, c->lat, net, l, tl,   \
                    tabl[l], net.kernel[l], c->occ, in, z, out, (T*)nullptr, (int64_t)0, c->P, grad)
      SCALE_GRAD_STAGED(SCALE_CALL)
#undef SCALE_CALL
    } else if (tiled) {
      SCALE_GRAD_TILED(k_fwd_tile, gridT, c->lat, net, l, c->occ, in, out, z);
    } else {
      k_fwd_layer<T><<<gridL, 128, 0, c->stream>>>(c->lat, net, l, c->occ, in, out, z);
    }
  };
  // forward pass: layer inputs at the checkpoints (every layer when stored), H(L) last
  {
    const T* in = nullptr;
    for (int l = 0; l < L; ++l) {
      T* out = HL;
      if (l < L - 1) {
        const bool keep = (l + 1) % stride == 0;
        out = keep ? ck + (size_t)((l + 1) / stride) * slab : segH + (size_t)((l + 1) % 2) * slab;
      }
      fwd(l, in, out, recompute ? segZ : segZ + (size_t)l * slab);
      if (e != cudaSuccess) return e;
      in = out;
    }
  }
  k_grad_proj<T><<<B, 256, 0, c->stream>>>(c->lat, net, c->orb_of_slot, c->slot_of_orb, (const T*)c->Binv,
                                           (const T*)c->Pt, HL, off_pw, off_pb, c->P, grad, dA);
  T* dcur = dA;   // d/dH(l+1)
  T* dnext = dB;  // d/dH(l)
  for (int sg = n_ck - 1; sg >= 0; --sg) {
    const int l0 = sg * stride, l1 = std::min(L, l0 + stride);
    if (recompute) {  // segment forward from its checkpoint: segH[m] = H(l0+m), segZ[m] = z(l0+m)
      const T* in = (l0 == 0) ? nullptr : ck + (size_t)sg * slab;
      for (int l = l0; l < l1; ++l) {
        T* out = segH + (size_t)(l - l0 + 1) * slab;
        fwd(l, in, out, segZ + (size_t)(l - l0) * slab);
        if (e != cudaSuccess) return e;
        in = out;
      }
    }
    for (int l = l1 - 1; l >= l0; --l) {
      const T* lin = (l == 0) ? nullptr : (l == l0 ? ck + (size_t)sg * slab : segH + (size_t)(l - l0) * slab);
      T* zl = recompute ? segZ + (size_t)(l - l0) * slab : segZ + (size_t)l * slab;
      const int kq = tiled ? taps[l] * (h / 4) * (h / 8) : taps[l] * h * h;
      if (!staged) k_grad_dz<T><<<B, 256, 0, c->stream>>>(c->lat, net, l, dcur, zl, dZ, offB[l], c->P, grad);
      if (staged) {
#define SCALE_CALL(HC)                                                                                               \
  e = staged_launch(k_conv_staged<T, HC, 1>, B, conv_block + bias_threads(h), conv_bytes<T>(N, h, taps[l]), c->stream, \
                    c->lat, net, l, taps[l], tabl[l] + nbr_size(N, taps[l]), KTl[l], c->occ, dcur, zl, dnext, dZ,     \
                    offB[l], c->P, grad)
        SCALE_GRAD_STAGED(SCALE_CALL)
#undef SCALE_CALL
        if (e != cudaSuccess) return e;
#define SCALE_CALL(HC)                                                                                               \
  e = staged_launch(k_dk_staged<T, HC>, B, staged_block(taps[l] * (h / kDkRows) * (h / 8), kDkThreads<T>),          \
                    staged_bytes<T>(N, h, taps[l], 2), c->stream, c->lat, net, l, taps[l], tabl[l], c->occ, lin, dZ,  \
                    offK[l], c->P, grad)
        SCALE_GRAD_STAGED(SCALE_CALL)
#undef SCALE_CALL
        if (e != cudaSuccess) return e;
      } else if (tiled) {
        const dim3 gridK((kq + 127) / 128, B);
        SCALE_GRAD_TILED(k_dk_tile, gridK, c->lat, net, l, taps[l], c->occ, lin, dZ, offK[l], c->P, grad);
        SCALE_GRAD_TILED(k_din_tile, gridT, c->lat, net, l, KTl[l], dcur, dZ, dnext);
      } else {
        k_grad_kernel<T><<<dim3((kq + 127) / 128, B), 128, 0, c->stream>>>(c->lat, net, l, taps[l], c->occ, lin,
                                                                            dZ, offK[l], c->P, grad);
        k_grad_din<T><<<gridL, 128, 0, c->stream>>>(c->lat, net, l, KTl[l], dcur, dZ, dnext);
      }
      std::swap(dcur, dnext);
    }
  }
#undef SCALE_GRAD_TILED
#undef SCALE_GRAD_STAGED
  k_grad_embed<T><<<B, 256, 0, c->stream>>>(c->lat, net, c->occ, dcur, c->P, grad);
  k_nan_bad<<<B, 256, 0, c->stream>>>(B, c->P, c->status, grad);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_grad(scale_ctx* c, double* grad, int recompute) {
  return c->fp64 ? grad_t<double>(c, grad, recompute) : grad_t<float>(c, grad, recompute);
}

}  // namespace scale
