// fp64_mma.cuh -- FP64 products on the 16-bit tensor cores by an error-free splitting
// (Ozaki, Ogita, Oishi, Rump 2012; on FP16 tensor cores: Mukunoki et al. 2020).
//
// sm_103a issues one warp-wide FP64 instruction per SM about every 19 cycles (measured: DFMA
// and DADD alike), a 16x8x16 FP16 mma.sync every 2.04. A sum of 16 FP64 products per element
// costs 16 DFMA = 304 cycles per warp-element; the same sum as 28 FP16 products of 7 slices
// costs 7 mma.sync shares (14 cycles) plus about 40 integer instructions and one DADD (19).
//
// Split. Row i of the left factor is scaled by a power of two 2^E > max_k |x_ik| (column c of
// the right factor by 2^F likewise), rounded to a multiple of 2^-56, and written in digits
//     x = 2^E (s_0 2^-8 + s_1 2^-16 + ... + s_6 2^-56),  |s_0| <= 256, s_l in [-128, 127],
// small integers that FP16 holds exactly. The products of two digits are integers of at most
// 2^16, and the sum over k = 16 and over the pairs (a, b) of one level l = a + b,
//     t_l = sum_{a+b=l} sum_k s_a(x_ik) s_b(y_kc),   |t_l| <= 2^20 + 5 2^18 < 2^22,
// is exact in the FP32 accumulator. The accumulators start at 1.5 2^23, so the bit pattern of
// a finished one is 0x4B400000 + t_l, with no conversion instruction. Levels 0..6 are kept:
//     sum_k x_ik y_kc = 2^(E+F) sum_l t_l 2^(-16-8l) + e,  |e| below 2^-50 2^(E+F) at worst and about
// 2^-56 2^(E+F) in the mean (what rounding to 2^-56 and the dropped levels leave), against about
// 2^-53 of the running sum for a chain of 16 rounded FP64 multiply-adds.
//
// The error is relative to the two scales, not to the terms: where a row's large values meet the
// column's small ones and the other way round, the digits that make up the sum lie low in both factors
// and rounding to 2^-56 cuts them. split_weight's one extra product of the leading digits,
//     S = sum_k |s_0(x_ik)| |s_0(y_kc)|  (2^16 for one term as large as the scales),
// tells such sums: below kSplitFloor = 2^16 / 16 (split_weak) the caller takes FP64 arithmetic for that
// element, so that a split sum's error stays at that of the FP64 chain. The test depends on the row
// and the column alone, so no result depends on how a product is cut into tiles or launches. (log|det| of
// 56 x 56 matrices against binary128, median / 90% of 100, FP64 chains; the split unguarded; guarded at 1/16:
// Gaussian 7e-15 / 2e-14 in all; entries exp(-d / 0.3) in the distance 1.7e-13 / 4e-11; 8e-11 / 9e-9;
// 2.3e-13 / 5e-11; one column times 2^0..2^90 1.4e-14 / 3e-14; 21 / 26; 1.1e-14 / 3e-14. At 1/64 rows of
// size exp(4 N) lose a factor of 2.) It also takes the rows and columns that hold an infinity, a NaN or a
// scale near the exponent range's ends (kScaleBad).
#pragma once

#include <cuda_fp16.h>

#include "mlp_mma.cuh"

namespace scale {

constexpr int kSplit = 7;                      // digits of a value
constexpr uint32_t kAccBits = 0x4B400000u;     // bits of 1.5 2^23, the accumulators' start
constexpr int kSplitExpMin = 1023 - 400, kSplitExpMax = 1023 + 400;  // biased exponents of a scale
constexpr int kScaleBad = -1;                  // in the place of one: no split of this row or column
constexpr float kSplitFloor = 4096.f;

// Biased exponent of |x| (0 for zero and subnormals, 2047 for infinities and NaN).
__host__ __device__ __forceinline__ int exp_field(uint64_t bits) { return (int)(bits >> 52) & 0x7ff; }

// The scale of a row or column from its largest exponent field: 0 when all its values are zero.
// (A subnormal counts as zero beside normal values; alone it makes a bad scale.)
__host__ __device__ __forceinline__ int split_scale(int emax, bool any_nonzero) {
  return !any_nonzero ? 0 : (emax >= kSplitExpMin && emax <= kSplitExpMax ? emax : kScaleBad);
}

// x / 2^E as digits with offsets: Y = round(x 2^(56-E)) + 128 (1 + 2^8 + ... + 2^40) + 256 2^48,
// E = emax - 1022 with emax the largest exponent field. Bytes 0..5 of Y are s_6 + 128, ..., s_1 + 128; Y >> 48 is s_0 + 256.
__host__ __device__ __forceinline__ uint64_t split_fixed(uint64_t bits, int emax) {
  const int e = exp_field(bits);
  const uint64_t m = e ? (bits & 0xfffffffffffffull) | 0x10000000000000ull : 0ull;
  const int d = emax - e;                                   // >= 0
  uint64_t X = (((m << 4) >> (d < 63 ? d : 63)) + 1) >> 1;  // round half up in magnitude
  if (bits >> 63) X = 0 - X;
  return X + 0x0100808080808080ull;
}

// Digits of a pair of values as FP16 pairs: half2 (s_l(a), s_l(b)), l = 0..6.
__device__ __forceinline__ void split_pair(uint64_t Ya, uint64_t Yb, uint32_t (&s)[kSplit]) {
  const uint32_t al = (uint32_t)Ya, ah = (uint32_t)(Ya >> 32), bl = (uint32_t)Yb, bh = (uint32_t)(Yb >> 32);
  // 1024 + d has the FP16 bits 0x6400 | d; subtracting 1024 + offset leaves the digit exactly
  const __half2 off0 = __float2half2_rn(1280.f), off = __float2half2_rn(1152.f);
  auto digit = [](uint32_t r, __half2 o) {
    r = (r & 0x03ff03ffu) | 0x64006400u;
    const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&r), o);
    return *reinterpret_cast<const uint32_t*>(&v);
  };
  s[0] = digit(__byte_perm(ah, bh, 0x7632), off0);
  s[1] = digit(__byte_perm(ah, bh, 0x7531) & 0x00ff00ffu, off);
  s[2] = digit(__byte_perm(ah, bh, 0x7430) & 0x00ff00ffu, off);
  s[3] = digit(__byte_perm(al, bl, 0x0703) & 0x00ff00ffu, off);
  s[4] = digit(__byte_perm(al, bl, 0x0602) & 0x00ff00ffu, off);
  s[5] = digit(__byte_perm(al, bl, 0x0501) & 0x00ff00ffu, off);
  s[6] = digit(__byte_perm(al, bl, 0x0400) & 0x00ff00ffu, off);
}

// J = round(2^58 sum_l t_l 2^(-16-8l)) from the accumulators' bit patterns u_l = 0x4B400000 + t_l:
// |sum| <= 16 keeps J in 64 bits; sums modulo 2^64 (only J itself has to fit).
__host__ __device__ __forceinline__ int64_t split_sum(const uint32_t (&u)[kSplit]) {
  constexpr uint64_t M = kAccBits;
  const uint64_t lo = (uint64_t)u[4] * 65536u + (uint64_t)u[5] * 256u + u[6] - M * (65536u + 256u + 1u) + 32u;
  const uint64_t lo6 = (uint64_t)((int64_t)lo >> 6);
  const uint64_t hi = ((uint64_t)((u[0] << 10) + (u[1] << 2)) << 32) + (uint64_t)u[2] * (1u << 26) + (uint64_t)u[3] * (1u << 18);
  return (int64_t)(hi - ((((M << 10) + (M << 2)) << 32) + M * (1u << 26) + M * (1u << 18)) + lo6);
}

// Bits of the double nearest to J 2^(E+F-58), E = ex - 1022 and F = fx - 1022 (biased exponents
// ex, fx of the two scales): integer arithmetic only, the FP64 pipe is the scarce one.
__host__ __device__ __forceinline__ uint64_t split_to_double(int64_t J, int ex, int fx) {
  const uint64_t a = J < 0 ? 0 - (uint64_t)J : (uint64_t)J;
  if (a == 0) return 0;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = __builtin_clzll(a);
#endif
  const uint64_t m = a << lz;
  const uint64_t mant = (m >> 11) + ((m >> 10) & 1);  // leading one at bit 52 (53 after a carry)
  // leading bit of J: 63 - lz; value = 1.x 2^(63 - lz + ex + fx - 2044 - 58)
  const uint64_t expo = (uint64_t)(1023 + 63 - 58 - 2044 - 1 - lz + ex + fx);
  return ((expo << 52) + mant) | ((uint64_t)J & 0x8000000000000000ull);
}

// One m16n8k16 tile of FP64 products: the A fragment's slices in registers, the B fragment's
// slices in shared memory (bf: [kSplit][32] uint2 of this column tile). acc_l are the level sums.
__device__ __forceinline__ void split_mma(float (&acc)[kSplit][4], const uint32_t (&a)[kSplit][4],
                                          const uint2* __restrict__ bf) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int l = 0; l < kSplit; ++l)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[l][i] = __uint_as_float(kAccBits);
#pragma unroll
  for (int sb = 0; sb < kSplit; ++sb) {
    const uint2 b = bf[sb * 32 + lane];
#pragma unroll
    for (int sa = 0; sa + sb < kSplit; ++sa) mma_f16(acc[sa + sb], a[sa], b.x, b.y);
  }
}

// The weights S of one tile's sums: the product of the leading digits' absolute values.
__device__ __forceinline__ void split_weight(float (&s)[4], const uint32_t (&a0)[4], uint2 b0) {
  constexpr uint32_t kAbs = 0x7fff7fffu;
  const uint32_t a[4] = {a0[0] & kAbs, a0[1] & kAbs, a0[2] & kAbs, a0[3] & kAbs};
#pragma unroll
  for (int i = 0; i < 4; ++i) s[i] = 0.f;
  mma_f16(s, a, b0.x & kAbs, b0.y & kAbs);
}
// Whether an element of weight s between the scales ex and fx is to be taken in FP64 arithmetic.
__device__ __forceinline__ bool split_weak(float s, int ex, int fx) {
  return ex < 0 || fx < 0 || (ex > 0 && fx > 0 && s < kSplitFloor);
}

// Element i (C fragment order) of a finished tile as a double.
__device__ __forceinline__ double split_value(const float (&acc)[kSplit][4], int i, int ex, int fx) {
  uint32_t u[kSplit];
#pragma unroll
  for (int l = 0; l < kSplit; ++l) u[l] = __float_as_uint(acc[l][i]);
  return __longlong_as_double((long long)split_to_double(split_sum(u), ex, fx));
}

}  // namespace scale
