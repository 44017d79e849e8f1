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

#include <cooperative_groups.h>

#include <algorithm>

#include "eloc_common.cuh"

namespace cg = cooperative_groups;

namespace scale {

namespace {

constexpr int kElocList = 2048;  // moves of one list

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
  uint32_t* mlist = reinterpret_cast<uint32_t*>(ms_all + WARPS);    // [kElocList]
  double* contrib = reinterpret_cast<double*>(mlist + kElocList);   // [kElocList]
  int32_t* slot_s = reinterpret_cast<int32_t*>(contrib + kElocList);
  int8_t* occ_s = reinterpret_cast<int8_t*>(slot_s + 2 * N);
  __shared__ int warp_cnt[WARPS];
  __shared__ int s_diag, s_next;

  // the CTAs of a cluster share one sample's moves: CTA `rank` takes moves rank, rank + cs, ... of
  // the list they all enumerate, and the first one collects and sums the contributions
  const cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int w = blockIdx.x / cs;
  const int b = a.list ? a.list[w] : w;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int st = a.status[b];
  if (st & (SCALE_SAMPLE_BAD_COUNT | SCALE_SAMPLE_DOUBLE_OCC | SCALE_SAMPLE_SINGULAR)) {
    if (tid == 0 && rank == 0) {
      a.out[b] = CUDART_NAN;
      if (a.move_count) a.move_count[b] = 0;
    }
    return;
  }
  if (tid == 0) s_diag = 0;
  for (int i = tid; i < N; i += blockDim.x) occ_s[i] = a.occ[(size_t)b * N + i];
  for (int o = tid; o < 2 * N; o += blockDim.x) slot_s[o] = a.slot_of_orb[(size_t)b * 2 * N + o];
  __syncthreads();
  if (rank == 0) {
    const int d = __reduce_add_sync(0xffffffffu, diag_count(a, occ_s, tid, WARPS * 32));
    if (lane == 0) atomicAdd(&s_diag, d);
  }
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
  double* sums = cs == 1 ? contrib : cluster.map_shared_rank(contrib, 0);
  double total = 0.0;  // thread 0
  int nmoves = 0;
  for (int id = 0; id < ncand;) {
    // the allowed moves of as many candidates as surely fit the list (enumeration order)
    int nm = 0;
    for (; id < ncand && nm + WARPS * 32 <= kElocList; id += WARPS * 32)
      nm = enumerate_window<WARPS>(a, occ_s, id, ncand, nm, mlist, warp_cnt);
    if (tid == 0) s_next = 0;
    if (cs == 1) __syncthreads();
    else cluster.sync();  // the first CTA has summed the previous list
    // warps take the next move as they finish the previous one
    for (;;) {
      int mi = 0;
      if (lane == 0) mi = atomicAdd(&s_next, 1);
      mi = __shfl_sync(0xffffffffu, mi, 0) * cs + rank;
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
      if (lane == 0) sums[mi] = move_coeff(a.lat, pm) * (double)det;
      __syncwarp();
    }
    if (cs == 1) __syncthreads();
    else cluster.sync();
    // fixed-order sum of the list: lane l adds contributions l, l+32, ..., then an xor tree
    // (both orders independent of which warp evaluated which move)
    if (warp == 0 && rank == 0) {
      double s = 0.0;
      for (int q = lane; q < nm; q += 32) s += contrib[q];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
      if (lane == 0) {
        total += s;
        nmoves += nm;
      }
    }
    if (cs == 1) __syncthreads();
  }
  if (tid == 0 && rank == 0) {
    a.out[b] = (a.lat.model == SCALE_MODEL_TJ ? (0.25 * a.lat.J) * s_diag : a.lat.U * s_diag) + total;
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
  return sizeof(MS) * WARPS + (sizeof(uint32_t) + sizeof(double)) * kElocList + sizeof(int32_t) * 2 * N + N + 16;
}

template <int H>
constexpr int kElocWarps = H == 64 ? 16 : 28;  // 64 channels keep 32 activations a lane: registers
// Connected configurations of a sample at the sector's mean densities.
inline double expected_moves(const scale_ctx* c) {
  const double fu = (double)c->lat.n_up / c->N, fd = (double)c->lat.n_dn / c->N, bonds = c->nb_nn + c->nb_nnn;
  if (c->lat.model == SCALE_MODEL_TJ)
    return 2.0 * bonds * (fu + fd) * (1.0 - fu - fd) + (c->lat.J != 0.0 ? 2.0 * c->nb_nn * fu * fd : 0.0);
  return 2.0 * bonds * (fu * (1.0 - fu) + fd * (1.0 - fd));
}
// CTAs per sample for n samples of `moves` moves: the number of the least time, waves x rounds, in units of
// one round of moves (a move per warp). Rounds of a sample: 1 up to 0.6 moves per warp (their number varies),
// 1.1 up to one, then 0.6 + 1.05 per move and warp, the set-up of each CTA included. Waves: samples in flight
// are one CTA per SM, and clusters of 4 and 8 leave SMs of a GPC over (38 clusters of 4 and 16 of 8 run as
// two waves); a further wave starts as the last one thins out. FP64: the FP64 pipe is busy with any number
// of moves, so a CTA's time goes with its share, 3% per further CTA for the repeated set-up. Local energies
// do not depend on it. (us, C = 1 / 2 / 4 / 8: 16x16 Hubbard 1 walker 677 / 347 / 186 / 107, 40 walkers
// 720 / 375 / 367 / 310, 100 walkers 725 / 707 / 565 / 719; 8x8 60 walkers 211 / 115 / 129 / 147; 4x4, some 31
// moves, 14 walkers 38 / 25 / 22 / 22, 40 walkers 39 / 25 / 37 / 52, 100 walkers 40 / 43 / 55 / 112.)
inline int eloc_split(int n, double moves, int warps, bool fp64) {
  int best = 1;
  double least = 0.0;
  for (int k = 0; k < 4; ++k) {
    const int C = 1 << k;
    const int slots = k == 0 ? 152 : k == 1 ? 76 : k == 2 ? 36 : (fp64 || n <= 14) ? 14 : 16;
    const int waves = C == 8 && n > 14 ? std::max(2, (n + slots - 1) / slots) : (n + slots - 1) / slots;
    const double m = moves / (C * warps), rounds = m <= 0.6 ? 1.0 : m <= 1.0 ? 1.1 : 0.6 + 1.05 * m;
    const double time = fp64 ? waves * (1.0 + 0.03 * (C - 1)) / C : waves == 1 ? rounds : 0.95 * waves * rounds;
    if (k == 0 || time < least || (!fp64 && time == least)) {
      best = C;
      least = time;
    }
  }
  return best;
}

template <typename T, int H, int WARPS, typename MS>
cudaError_t eloc_launch(scale_ctx* c, const LowrankArgs& a, int n) {
  const size_t smem = eloc_smem<WARPS, MS>(c->N);
  auto kern = k_eloc<T, H, WARPS, MS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int C = eloc_split(n, expected_moves(c), WARPS, sizeof(T) == 8);
  if (C > 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n * C);
    cfg.blockDim = dim3(WARPS * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, a, make_net<T>(c));
    if (e == cudaSuccess) return e;
    cudaGetLastError();  // a partition without room for a cluster: one CTA per sample
  }
  kern<<<n, WARPS * 32, smem, c->stream>>>(a, make_net<T>(c));
  return cudaGetLastError();
}

// Launch shape: the most warps per CTA (one CTA per SM) whose move scratch fits shared memory beside the
// kernel's static arrays (WARPS + 2 words).
constexpr size_t kElocSmemMax = 227 * 1024 - 256;
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
