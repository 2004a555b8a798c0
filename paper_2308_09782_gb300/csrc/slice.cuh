// Complex FP64 products on the BF16 tensor cores without rounding in the
// products: every row of an operand is scaled by a power of two and cut into
// kSlices signed 8-bit digits, the digit matrices are multiplied exactly
// (BF16 operands, FP32 accumulation of integers below 2^24), and the integer
// group sums are put together into one correctly rounded FP64 number per real
// part.  The scheme is the error-free transformation of matrix products of
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012) with a fixed number
// of slices.
//
// Operand row:  x[k] = 2^e sum_{s=1..8} d_s[k] 2^{-8s},  d_s in [-128, 127],
//   e from the row's largest part so that max |x| 2^-e is in [1/4, 1/2): the row
//   is held to 2^-65 of 2^e.  Every entry down to 2^-10 of the row's largest
//   keeps all of its 53 bits.
// Product:      C = A R^dagger, C[m][n] = 2^{eA[m] + eR[n]} sum_{g=2..10} 2^{-8g} P_g[m][n],
//   P_g = sum_{s+t=g} A_s R_t^dagger.  Pairs with s + t > 10 are left out: a term of
//   theirs is at most 2^-74 of 2^{eA + eR}.
// Error against 64-bit results, relative in the Frobenius norm | largest over the
//   elements relative to (|A| |R|)_mn, of the products of 512 silicon atoms:
//                          D H                    S^-1 W
//   FP64 multiply-adds     2.3e-16 | 1.0e-15      5.7e-16 | 1.7e-15
//   7 digits, s + t <= 9   3.7e-16 | 4.1e-14      1.3e-15 | 5.2e-13    (34 pairs)
//   8 digits, s + t <= 9   5.5e-17 | 1.7e-15      2.6e-16 | 1.3e-13    (36)
//   8 digits, s + t <= 10  5.2e-17 | 1.5e-16      4.2e-17 | 2.1e-15    (43, this form)
//   Rows that decay much faster (e^{-0.2 |m - k|} and more over a hundred orbitals) keep
//   the norm, but not the elements far below their row's scale.
// Exactness: a digit product is at most 2^14, so a run of 512 complex (1024
//   real) k keeps every partial sum at or below 2^24, which FP32 holds exactly;
//   the kernel takes the accumulator out after each run and adds the runs as
//   32-bit integers.
// Integer sums do not depend on their order: results are the same for every
// tiling, batch composition and schedule.
//
// What bounds it: 43 digit products of 8 N^3 BF16 flops stand in for one FP64
// product, 43 / 1750 TFLOP/s against 1 / 1.2 TFLOP/s on the FP64 pipe.
#pragma once
#include "vgtb_internal.h"

namespace vgtb {

constexpr int kSlices = 8;
constexpr int kSliceGroups = 9;            // s + t = 2 .. 10
constexpr int kSliceShift = 8 * (kSliceGroups + 1);  // the last group's weight is 2^-kSliceShift
constexpr int kSlicePairs = 8;             // most pairs of a group
constexpr int kSliceNaN = 1 << 24;         // row exponent of a row with a non-finite entry
// 32-bit group sums: 8 pairs x 2 N x 2^14 = 2^31, which would take 128 for the magnitude of every
// digit, i.e. -128, and so |x| 2^-e above 1/2
constexpr int kSliceMaxN = 8192;

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

// exponent field of a row's scale from the largest high word of its parts: e = field - 1021.  A
// largest part within 1/64 of the next power of two takes that power's scale, so that the first digit
// never rounds up to 128.
__device__ __forceinline__ int slice_field(uint32_t high) { return max((int)((high + 0x4000u) >> 20), 1); }

// 2^k (sum over groups of G[g - 2] 2^{80 - 8g}) correctly rounded to FP64 (NaN for k = kSliceNaN)
// with integer operations (the FP64 pipe runs at a small fraction of the integer rate).
__device__ __forceinline__ double slice_value(const int (&G)[kSliceGroups], int k) {
  // weights relative to the last group: 2^64, 2^56, ..., 2^0.  The sum as a 128-bit number hi : lo
  // (|G[4]| has 5 pairs: the second part stays below 2^63)
  const long long a = ((long long)G[0] << 24) + ((long long)G[1] << 16) + ((long long)G[2] << 8) + G[3];  // x 2^40
  const long long b = ((long long)G[4] << 32) + ((long long)G[5] << 24) + ((long long)G[6] << 16) +
                      ((long long)G[7] << 8) + G[8];
  unsigned long long lo = ((unsigned long long)a << 40) + (unsigned long long)b;
  long long hi = (a >> 24) + (b >> 63) + (lo < (unsigned long long)b ? 1 : 0);
  const bool neg = hi < 0;
  if (neg) {  // magnitude
    lo = 0ull - lo;
    hi = ~hi + (lo == 0ull ? 1 : 0);
  }
  unsigned long long top = lo, rest = 0;
  int len;  // bits of the magnitude
  if (hi == 0) {
    if (lo == 0ull) return k >= kSliceNaN / 2 ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
    const int z = __clzll((long long)lo);
    top = lo << z;
    len = 64 - z;
  } else {
    const int z = __clzll(hi);  // hi is below 2^30
    top = ((unsigned long long)hi << z) | (lo >> (64 - z));
    rest = lo << z;
    len = 128 - z;
  }
  // top has its first bit set: value = top 2^(len - 64) (plus the sticky rest)
  unsigned long long m = top >> 11;
  const uint32_t r = ((uint32_t)top & 0x7ffu);
  const bool up = r > 0x400u || (r == 0x400u && (rest != 0ull || (m & 1ull)));
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
  const int k = (ea == kSliceNaN || er == kSliceNaN) ? kSliceNaN : ea + er - kSliceShift;
  return make_double2(slice_value(gr, k), slice_value(gi, k));
}

}  // namespace vgtb
