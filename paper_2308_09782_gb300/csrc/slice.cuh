// Complex FP64 products on the BF16 tensor cores without rounding in the
// products: every row of an operand is scaled by a power of two and cut into
// kSlices signed 8-bit digits, the digit matrices are multiplied exactly
// (BF16 operands, FP32 accumulation of integers below 2^24), and the integer
// group sums are put together into one correctly rounded FP64 number per real
// part.  The scheme is the error-free transformation of matrix products of
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012) with a fixed number
// of slices.
//
// Operand row:  x[k] = 2^e sum_{s=1..7} d_s[k] 2^{-8s},  |d_1| <= 128,
//   d_s in [-128, 127] for s > 1, e from the row's largest part so that
//   max |x| 2^-e is in [1/4, 1/2): the row is held to 2^-57 of 2^e, 2^-55 of its
//   largest entry at worst.
// Product:      C = A R^dagger, C[m][n] = 2^{eA[m] + eR[n]} sum_{g=2..9} 2^{-8g} P_g[m][n],
//   P_g = sum_{s+t=g} A_s R_t^dagger.  Pairs with s + t > 9 are left out: a term of
//   theirs is below 2^-66 of 2^{eA + eR}.  (Without group 9, 28 instead of 34 pairs,
//   products of matrices that decay away from the diagonal came out 1.3e-15 off in the
//   2-norm at N = 128, against 3.6e-16 for FP64 multiply-adds.)
// Exactness: a digit product is at most 2^14, so a run of 512 complex (1024
//   real) k keeps every partial sum at or below 2^24, which FP32 holds exactly;
//   the kernel takes the accumulator out after each run and adds the runs as
//   32-bit integers.
// Integer sums do not depend on their order: results are the same for every
// tiling, batch composition and schedule.
//
// What bounds it: 34 digit products of 8 N^3 BF16 flops stand in for one FP64
// product, 34 / 1750 TFLOP/s against 1 / 1.2 TFLOP/s on the FP64 pipe.
#pragma once
#include "vgtb_internal.h"

namespace vgtb {

constexpr int kSlices = 7;
constexpr int kSliceGroups = 8;            // s + t = 2 .. 9
constexpr int kSliceNaN = 1 << 24;         // row exponent of a row with a non-finite entry
constexpr int kSliceMaxN = 8192;           // 32-bit group sums: 7 pairs x 2 N x 2^14 < 2^31

// digits of `rows` rows of K complex numbers: dig[s][row][2 Kp], planar [Re | Im], Kp = K rounded up to 64
struct SliceMat {
  __nv_bfloat16* dig;
  int* ex;                // [rows]
  int rows, K, Kp;
};

// SlicePlanes (vgtb_internal.h): group g owns np(g) consecutive planes, which add up to P_g.
// pairs (s, g - s) of group g, 1 <= s, t <= kSlices
__host__ __device__ constexpr int slice_pairs(int g) { return g - 1 <= kSlices ? g - 1 : 2 * kSlices + 1 - g; }
// planes of group g when a plane takes at most MP pairs
template <int MP>
__host__ __device__ constexpr int slice_np(int g) {
  return (slice_pairs(g) + MP - 1) / MP;
}
template <int MP>
__host__ __device__ constexpr int slice_planes() {
  int n = 0;
  for (int g = 2; g < 2 + kSliceGroups; ++g) n += slice_np<MP>(g);
  return n;
}

// m 2^q where the exponent leaves the normal range, or NaN for a row marked so (rare: kept out of line)
static __device__ __noinline__ double slice_scaled(double m, int k, int q) {
  return k >= kSliceNaN / 2 ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(m, q);
}

// 2^k (sum over groups of G[g - 2] 2^{72 - 8g}) correctly rounded to FP64 (NaN for k = kSliceNaN)
// with integer operations (the FP64 pipe runs at a small fraction of the integer rate).
__device__ __forceinline__ double slice_value(const int (&G)[kSliceGroups], int k) {
  // weights relative to the last group: 2^56, 2^48, ..., 2^0
  long long hi = ((long long)G[0] << 24) + ((long long)G[1] << 16) + ((long long)G[2] << 8) + G[3];  // x 2^32
  long long lo = ((long long)G[4] << 24) + ((long long)G[5] << 16) + ((long long)G[6] << 8) + G[7];
  hi += lo >> 32;
  uint32_t l = (uint32_t)lo;
  const bool neg = hi < 0;
  if (neg) {  // magnitude of the 96-bit number
    l = 0u - l;
    hi = ~hi + (l == 0u ? 1 : 0);
  }
  unsigned long long top;
  uint32_t rest = 0;
  int len;  // bits of the magnitude
  if (hi == 0) {
    if (l == 0u) return k >= kSliceNaN / 2 ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
    const int z = __clz((int)l);
    top = (unsigned long long)l << (32 + z);
    len = 32 - z;
  } else {
    const int z = __clzll(hi);
    len = 96 - z;
    if (z < 32) {
      top = ((unsigned long long)hi << z) | ((unsigned long long)l >> (32 - z));
      rest = l << z;
    } else {
      top = ((unsigned long long)hi << z) | ((unsigned long long)l << (z - 32));
    }
  }
  // top has its first bit set: value = top 2^(len - 64) (plus the sticky rest)
  unsigned long long m = top >> 11;
  const uint32_t r = ((uint32_t)top & 0x7ffu);
  const bool up = r > 0x400u || (r == 0x400u && (rest != 0u || (m & 1ull)));
  m += up ? 1ull : 0ull;  // a carry out of the 53 bits raises the exponent below
  const int ef = 1023 + len - 1 + k;
  if (ef > 0 && ef < 2046) {
    const unsigned long long bits =
        ((unsigned long long)(ef - 1) << 52) + m + (neg ? 0x8000000000000000ull : 0ull);
    return __longlong_as_double((long long)bits);
  }
  return slice_scaled(neg ? -(double)m : (double)m, k, len - 53 + k);
}

template <int MP>
__device__ __forceinline__ double2 slice_load(const SlicePlanes& S, long long row, int col) {
  const int* p = S.p + row * 2 * S.Nw + col;
  int gr[kSliceGroups], gi[kSliceGroups];
  int q = 0;
#pragma unroll
  for (int g = 2; g < 2 + kSliceGroups; ++g) {
    int a = 0, b = 0;
#pragma unroll
    for (int j = 0; j < slice_np<MP>(g); ++j, ++q) {
      a += p[q * S.stride];
      b += p[q * S.stride + S.Nw];
    }
    gr[g - 2] = a;
    gi[g - 2] = b;
  }
  const int ea = S.exA[row], er = S.exR[col];
  const int k = (ea == kSliceNaN || er == kSliceNaN) ? kSliceNaN : ea + er - 72;
  return make_double2(slice_value(gr, k), slice_value(gi, k));
}

}  // namespace vgtb
