// lowrank.cu -- amplitude ratios of explicit moves by the cached-network + rank-r determinant
// update of Sec. II.C, and the choice of the local-energy kernel (eloc.cuh).
#include <algorithm>

#include "eloc_common.cuh"

namespace scale {

namespace {

constexpr int kWarps = 8;

// psi(n')/psi(n) in the ascending convention for M explicit moves per sample.
template <typename T, int H>
__global__ void __launch_bounds__(kWarps * 32) k_ratios(LowrankArgs a, Net<T> net) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int N = a.lat.N, Ne = a.lat.Ne, h = net.h;
  MoveScratch<T, H>* ms_all = reinterpret_cast<MoveScratch<T, H>*>(smem);
  int32_t* slot_s = reinterpret_cast<int32_t*>(ms_all + kWarps);
  int8_t* occ_s = reinterpret_cast<int8_t*>(slot_s + 2 * N);
  const int b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int st = a.status[b];
  const bool bad = st & (SCALE_SAMPLE_BAD_COUNT | SCALE_SAMPLE_DOUBLE_OCC | SCALE_SAMPLE_SINGULAR);
  if (bad) {
    for (int m = tid; m < a.M; m += blockDim.x) a.out[(size_t)b * a.M + m] = CUDART_NAN;
    return;
  }
  for (int i = tid; i < N; i += blockDim.x) occ_s[i] = a.occ[(size_t)b * N + i];
  for (int o = tid; o < 2 * N; o += blockDim.x) slot_s[o] = a.slot_of_orb[(size_t)b * 2 * N + o];
  __syncthreads();
  SampleView<T> sv;
  sv.occ = occ_s;
  sv.slot_of_orb = slot_s;
  sv.z0 = (const T*)a.z0 + (size_t)b * N * h;
  sv.HL = (const T*)a.HL + (size_t)b * N * h;
  sv.Binv = (const T*)a.Binv + (size_t)b * Ne * Ne;
  sv.Pt = (const T*)a.Pt + (size_t)b * 2 * Ne * h;
  sv.G0t = (const T*)a.G0t + (size_t)b * Ne * 2 * N;
  MoveScratch<T, H>& ms = ms_all[warp];
  const LaneTap lt = lane_tap(a.lat, net, a.k0);
  for (int mi = warp; mi < a.M; mi += kWarps) {
    const int32_t* mv = a.moves + ((size_t)b * a.M + mi) * 4;
    const int kind = mv[0], src = mv[1], dst = mv[2], spin = mv[3];
    double out;
    if (kind < 0) {
      out = 1.0;
    } else if (!move_allowed(a.lat, kind, src, dst, spin, occ_s)) {
      out = 0.0;
    } else {
      if (lane == 0) {
        ms.kind = kind;
        ms.src = src;
        ms.dst = dst;
        ms.spin = spin;
      }
      __syncwarp();
      move_features<T, H>(a.lat, net, lt, sv, a.mf, ms);
      const int r = move_matrix<T, H>(a.lat, net, sv, ms);
      const T det = (r < 0) ? T(CUDART_NAN) : warp_det<T>(ms, r);
      int par;
      if (kind == 0) {
        par = between_parity(occ_s, N, spin * N + src, spin * N + dst);
      } else {
        // exchange: the up electron and the down electron each hop between src and dst
        par = between_parity(occ_s, N, src, dst) ^ between_parity(occ_s, N, N + src, N + dst);
      }
      out = (par ? -1.0 : 1.0) * (double)det;
    }
    if (lane == 0) a.out[(size_t)b * a.M + mi] = out;
    __syncwarp();
  }
}

template <typename T, int H>
size_t ratio_smem(int N) {
  return sizeof(MoveScratch<T, H>) * kWarps + sizeof(int32_t) * 2 * N + N + 16;
}


template <typename T, int H>
cudaError_t ratios_t(scale_ctx* c, const int32_t* moves, int M, double* ratio) {
  LowrankArgs a = make_args(c);
  a.out = ratio;
  a.moves = moves;
  a.M = M;
  const size_t smem = ratio_smem<T, H>(c->N);
  cudaError_t e = cudaFuncSetAttribute(k_ratios<T, H>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_ratios<T, H><<<c->B, kWarps * 32, smem, c->stream>>>(a, make_net<T>(c));
  return cudaGetLastError();
}

}  // namespace

#define SCALE_DISPATCH_H(c, FN, ...)                                                          \
  ((c)->hpad == 16   ? ((c)->fp64 ? FN<double, 16>(__VA_ARGS__) : FN<float, 16>(__VA_ARGS__)) \
   : (c)->hpad == 32 ? ((c)->fp64 ? FN<double, 32>(__VA_ARGS__) : FN<float, 32>(__VA_ARGS__)) \
                     : ((c)->fp64 ? FN<double, 64>(__VA_ARGS__) : FN<float, 64>(__VA_ARGS__)))

// E_loc of the n listed samples (outputs indexed by sample), or of samples 0..n-1.
static cudaError_t launch_eloc(scale_ctx* c, double* eloc, const int32_t* list, int n) {
  if (c->et_wimg) return launch_eloc_tc(c, eloc, list, n);  // the batched kernel was asked for
  return c->fp64 ? launch_eloc_f64(c, eloc, list, n) : launch_eloc_f32(c, eloc, list, n);
}

cudaError_t launch_eloc_lowrank(scale_ctx* c, double* eloc) { return launch_eloc(c, eloc, nullptr, c->B); }

cudaError_t launch_eloc_lowrank_list(scale_ctx* c, const int32_t* list, int n, double* eloc) {
  return launch_eloc(c, eloc, list, n);
}

cudaError_t launch_ratios(scale_ctx* c, const int32_t* moves, int M, double* ratio) {
  return SCALE_DISPATCH_H(c, ratios_t, c, moves, M, ratio);
}

}  // namespace scale
