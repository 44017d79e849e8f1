// eloc.cuh -- low-rank local energies, one CTA per sample (Sec. II.C): the kernel and its launch,
// instantiated per working type by eloc_f32.cu and eloc_f64.cu.
//
// Connected configurations are enumerated on the device in the fixed order of eloc_common.cuh,
// compacted chunk by chunk, and handed to the warps (one move per warp at a time, move.cuh).
// Per-move contributions are summed in enumeration order, so E_loc does not depend on scheduling.
//
// Matrix elements in slot order (a moved electron keeps its determinant row):
//   hop     -t (NN) / -t' (NNN) times det R   (its Jordan-Wigner sign and the row
//           permutation sign of the ascending convention cancel),
//   exchange (J/2)(S+_i S-_j + h.c.) = -(J/2) (c+_{i up} c_{j up})(c+_{j dn} c_{i dn}):
//           -J/2 times det R.
// Diagonal: Hubbard U * (doubly occupied sites); t-J J sum_<ij> Sz_i Sz_j; the
// particle-hole transformed Hubbard model U sum_i n_up (1 - n_dn).
#pragma once

#include <algorithm>

#include "eloc_common.cuh"

namespace scale {

namespace {

// WARPS warps per sample; the sample's cached rows (Pt, z0, H(L), G0t) are read through L1/L2,
// shared memory holds the per-warp move scratch and the move list. Bound by the instructions and
// the dependent chain of a move (an FP32-FMA peak of 80.5 TFLOP/s, 14-15 reached; DRAM under 2%).
// ms per 4096 walkers of the 16x16 Hubbard workload, in the order of the steps: 24.48 with 20 warps
// and 10 KB of scratch a warp; the scratch cut to 6 KB (Delta H in place of H', 14 sites, 28
// electrons), 28 warps 23.09; the row length a constant, no run-time division by the tap count
// and the tanh of small arguments alone after a vote 19.58 (20 warps 20.68, 24 warps 20.34); layer-0
// rows straight from the cache and the tables, tap offsets kept per lane, list positions of the
// moved electrons 17.93. t-J at 32x32 (16 channels, 133 walkers) 1.584 -> 0.990, 64 walkers of 8x8
// 0.168 -> 0.106.
template <typename T, int H, int WARPS, typename MS>
__global__ void __launch_bounds__(WARPS * 32, 1) k_eloc(LowrankArgs a, Net<T> net) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int N = a.lat.N, Ne = a.lat.Ne, h = MS::kExact ? H : net.h;
  MS* ms_all = reinterpret_cast<MS*>(smem);
  uint32_t* mlist = reinterpret_cast<uint32_t*>(ms_all + WARPS);     // [kMoveChunk]
  double* contrib = reinterpret_cast<double*>(mlist + kMoveChunk);   // [kMoveChunk]
  int32_t* slot_s = reinterpret_cast<int32_t*>(contrib + kMoveChunk);
  int8_t* occ_s = reinterpret_cast<int8_t*>(slot_s + 2 * N);
  __shared__ int warp_cnt[WARPS];
  __shared__ double s_diag;
  __shared__ int s_next;

  const int b = a.list ? a.list[blockIdx.x] : blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int st = a.status[b];
  if (st & (SCALE_SAMPLE_BAD_COUNT | SCALE_SAMPLE_DOUBLE_OCC | SCALE_SAMPLE_SINGULAR)) {
    if (tid == 0) {
      a.out[b] = CUDART_NAN;
      if (a.move_count) a.move_count[b] = 0;
    }
    return;
  }
  for (int i = tid; i < N; i += blockDim.x) occ_s[i] = a.occ[(size_t)b * N + i];
  for (int o = tid; o < 2 * N; o += blockDim.x) slot_s[o] = a.slot_of_orb[(size_t)b * 2 * N + o];
  __syncthreads();
  if (tid == 0) s_diag = diag_energy(a, occ_s);
  SampleView<T> sv;
  sv.occ = occ_s;
  sv.slot_of_orb = slot_s;
  sv.z0 = (const T*)a.z0 + (size_t)b * N * h;
  sv.HL = (const T*)a.HL + (size_t)b * N * h;
  sv.Binv = (const T*)a.Binv + (size_t)b * Ne * Ne;
  sv.Pt = (const T*)a.Pt + (size_t)b * 2 * Ne * h;
  sv.G0t = (const T*)a.G0t + (size_t)b * Ne * 2 * N;
  MS& ms = ms_all[warp];

  const LaneTap lt = lane_tap(a.lat, net, a.k0);
  const int ncand = candidate_count(a);
  double total = 0.0;  // thread 0
  int nmoves = 0;
  for (int cs = 0; cs < ncand; cs += kMoveChunk) {
    const int ce = min(ncand, cs + kMoveChunk);
    // enumerate and compact the allowed moves of this chunk (enumeration order)
    const int nm = enumerate_chunk<WARPS>(a, occ_s, cs, ce, mlist, warp_cnt);
    if (tid == 0) s_next = 0;
    __syncthreads();
    // warps take the next move as they finish the previous one
    for (;;) {
      int mi = 0;
      if (lane == 0) mi = atomicAdd(&s_next, 1);
      mi = __shfl_sync(0xffffffffu, mi, 0);
      if (mi >= nm) break;
      const uint32_t pm = mlist[mi];
      if (lane == 0) {
        const MoveDesc m = unpack_move(pm);
        ms.src = m.src;
        ms.dst = m.dst;
        ms.spin = m.spin;
        ms.kind = m.kind;
      }
      __syncwarp();
      move_features<T, H>(a.lat, net, lt, sv, a.mf, ms);
      const int r = move_matrix<T, H>(a.lat, net, sv, ms);
      const T det = (r < 0) ? T(CUDART_NAN) : warp_det<T>(ms, r);
      if (lane == 0) contrib[mi] = move_coeff(a.lat, pm) * (double)det;
      __syncwarp();
    }
    __syncthreads();
    // fixed-order sum of the chunk: lane l adds contributions l, l+32, ..., then an xor tree
    // (both orders independent of which warp evaluated which move)
    if (warp == 0) {
      double s = 0.0;
      for (int q = lane; q < nm; q += 32) s += contrib[q];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) {
        total += s;
        nmoves += nm;
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    a.out[b] = s_diag + total;
    if (a.move_count) a.move_count[b] = nmoves;
  }
}

// The scratch of a neighbour hop: 3x3 boxes around two sites a nearest or diagonal step apart
// cover at most 14 sites (the 13-site plus 18), so at most 28 electrons.
template <typename T, int H, bool EXACT>
using ElocBox = MoveScratch<T, H, 14, 28, true, EXACT>;
template <typename T, int H, bool EXACT>
using ElocDisk = MoveScratch<T, H, kSMax, kRMax, true, EXACT>;

template <int WARPS, typename MS>
size_t eloc_smem(int N) {
  return sizeof(MS) * WARPS + (sizeof(uint32_t) + sizeof(double)) * kMoveChunk + sizeof(int32_t) * 2 * N + N + 16;
}

template <int H>
constexpr int kElocWarps = H == 64 ? 16 : 28;  // 64 channels keep 32 activations a lane: registers
template <typename T, int H, int WARPS, typename MS>
cudaError_t eloc_launch(scale_ctx* c, const LowrankArgs& a, int n) {
  const size_t smem = eloc_smem<WARPS, MS>(c->N);
  cudaError_t e = cudaFuncSetAttribute(k_eloc<T, H, WARPS, MS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_eloc<T, H, WARPS, MS><<<n, WARPS * 32, smem, c->stream>>>(a, make_net<T>(c));
  return cudaGetLastError();
}

// Launch shape: the most warps per CTA (one CTA per SM) whose move scratch fits shared memory.
constexpr size_t kElocSmemMax = 227 * 1024;
template <typename T, int H, typename MS, int W, int... REST>
cudaError_t eloc_shape(scale_ctx* c, const LowrankArgs& a, int n) {
  if constexpr (sizeof...(REST) == 0) {
    return eloc_launch<T, H, W, MS>(c, a, n);
  } else {
    if constexpr (sizeof(MS) * W < kElocSmemMax)
      if (eloc_smem<W, MS>(c->N) <= kElocSmemMax) return eloc_launch<T, H, W, MS>(c, a, n);
    return eloc_shape<T, H, MS, REST...>(c, a, n);
  }
}

template <typename T, int H>
cudaError_t eloc_t(scale_ctx* c, double* eloc, const int32_t* list, int n) {
  LowrankArgs a = make_args(c);
  a.out = eloc;
  a.move_count = c->move_count;
  a.list = list;
  const bool box = c->k0 <= 3;
  if constexpr (sizeof(T) == 4) {
    if (c->h == H)
      return box ? eloc_shape<T, H, ElocBox<T, H, true>, kElocWarps<H>, 12>(c, a, n)
                 : eloc_shape<T, H, ElocDisk<T, H, true>, H == 64 ? 16 : 20, 12>(c, a, n);
  }
  return box ? eloc_shape<T, H, ElocBox<T, H, false>, H == 64 ? 16 : 20, 12, 8>(c, a, n)
             : eloc_shape<T, H, ElocDisk<T, H, false>, H == 64 ? 16 : 20, 12, 8>(c, a, n);
}

template <typename T>
cudaError_t eloc_width(scale_ctx* c, double* eloc, const int32_t* list, int n) {
  return c->hpad == 16   ? eloc_t<T, 16>(c, eloc, list, n)
         : c->hpad == 32 ? eloc_t<T, 32>(c, eloc, list, n)
                         : eloc_t<T, 64>(c, eloc, list, n);
}

}  // namespace

}  // namespace scale
