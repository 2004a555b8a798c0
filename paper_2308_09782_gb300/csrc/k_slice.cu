// Sliced FP64 complex products (scheme and bounds in slice.cuh):
//   k_slice_rows    - rows of a matrix, or of a finished product, to digits
//   k_slice_hamilton - H_k(t) at its nonzero atom blocks to digits
//   k_slice_gemm    - the digit products, tcgen05 2-SM pairs
#include <algorithm>
#include <cstring>

#include "tc_kernel.cuh"
#include "vgtb_slice.h"

namespace vgtb {

namespace {

// digits of one real number as bytes: byte 8 - s of the result is d_s + 128 for s = 2..8, and the
// first byte d_1 itself.  efm: exponent field of the row's scale (slice_field).
__device__ __forceinline__ unsigned long long slice_bytes(double x, int efm) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int f = (int)((b >> 52) & 0x7ffu);
  unsigned long long m = (b & 0xfffffffffffffull) | (f ? 0x10000000000000ull : 0ull);
  const int sh = efm - (f ? f : 1) - 10;  // x 2^(64 - e) = m 2^-sh, below 2^63 - 2^56
  if (sh <= 0)
    m <<= -sh;
  else
    m = sh < 64 ? ((m >> (sh - 1)) + 1) >> 1 : 0ull;  // to nearest, halves away from zero
  const long long v = (b >> 63) ? -(long long)m : (long long)m;
  return (unsigned long long)(v + 0x0080808080808080ll);
}

// float with the value of digit s (1-based) of slice_bytes' result: an exact integer
__device__ __forceinline__ float slice_digit(unsigned long long w, int s) {
  const uint32_t b = s == 1 ? (uint32_t)(w >> 56) ^ 0x80u : (uint32_t)(w >> (8 * (kSlices - s))) & 0xffu;
  return __uint_as_float(0x4b000000u | b) - 8388736.0f;  // 2^23 + 128
}

__device__ __forceinline__ uint32_t pack_digits(float a, float b) {
  return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);  // both exact in BF16
}

// four adjacent columns (col a multiple of 4, below Nw) of the real or imaginary part, 16 bytes per plane
template <int MP>
__device__ __forceinline__ void slice_part4(const int* p, long long stride, const int (&k)[4], double (&x)[4]) {
  int g4[4][kSliceGroups];
  int q = 0;
#pragma unroll
  for (int g = 0; g < kSliceGroups; ++g) {
    int4 a = make_int4(0, 0, 0, 0);
#pragma unroll
    for (int j = 0; j < slice_np<MP>(g + 2); ++j, ++q) {
      const int4 u = *reinterpret_cast<const int4*>(p + q * stride);
      a.x += u.x; a.y += u.y; a.z += u.z; a.w += u.w;
    }
    g4[0][g] = a.x; g4[1][g] = a.y; g4[2][g] = a.z; g4[3][g] = a.w;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) x[j] = slice_value(g4[j], k[j]);
}

template <int MP>
__device__ __forceinline__ void slice_load4(const SlicePlanes& S, long long row, int col, int cols, double (&xr)[4],
                                            double (&xi)[4], bool add) {
  const int* p = S.p + row * 2 * S.Nw + col;
  const int ea = S.exA[row];
  int k[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int er = col + j < cols ? S.exR[col + j] : 0;
    k[j] = (ea == kSliceNaN || er == kSliceNaN) ? kSliceNaN : ea + er - kSliceShift;
  }
  double r[4], i[4];
  slice_part4<MP>(p, S.stride, k, r);
  slice_part4<MP>(p + S.Nw, S.stride, k, i);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const bool in = col + j < cols;
    xr[j] = (add ? xr[j] : 0.0) + (in ? r[j] : 0.0);
    xi[j] = (add ? xi[j] : 0.0) + (in ? i[j] : 0.0);
  }
}

}  // namespace

// One row per TPR threads, four adjacent columns per thread and iteration (IT iterations), the row
// kept in registers between the search for its largest part and the cut.  Memory bound: at
// N = 2048 it reads 67 MB (a matrix) or 302 MB (planes) and writes 134 MB of digits.  One
// iteration per thread wherever a CTA can hold the row: with four, 128 threads a row, the 130 to
// 150 registers left 16 warps an SM and the loads waited (planes of seven digits, N = 2048: 123 us
// against 98).  Eight digits: a matrix 54 us, planes 116.
template <int TPR, int IT, int MP>
__global__ void __launch_bounds__(TPR > 128 ? TPR : 128)
    k_slice_rows(const SliceRowJob* __restrict__ jobs, const int* __restrict__ step) {
  constexpr int NT = TPR > 128 ? TPR : 128;
  constexpr int RPB = NT / TPR, NW = NT / 32, WPR = TPR / 32;
  __shared__ uint32_t s_max[NW];
  pdl_wait();
  pdl_trigger();
  const SliceRowJob& J = jobs[blockIdx.y];
  const int row = blockIdx.x * RPB + threadIdx.x / TPR;
  const int t = threadIdx.x % TPR;
  const bool live = row < J.rows;
  if (RPB == 1 && !live) return;
  const int width = J.out.dig ? J.out.Kp : J.cols;
  double xr[IT][4], xi[IT][4];
  uint32_t mx = 0;
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int c = 4 * (t + TPR * it);
#pragma unroll
    for (int j = 0; j < 4; ++j) xr[it][j] = xi[it][j] = 0.0;
    if (!live || c >= J.cols) continue;
    if (J.src) {
      const double2* s = J.src + (step ? (*step & 1) : 0) * J.src_par + (long long)row * J.lds + c;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c + j < J.cols) {
          const double2 v = s[j];
          xr[it][j] = v.x;
          xi[it][j] = v.y;
        }
    } else {
      slice_load4<MP>(J.pl[0], row, c, J.cols, xr[it], xi[it], false);
      if (J.n_planes > 1) slice_load4<MP>(J.pl[1], row, c, J.cols, xr[it], xi[it], true);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (J.epi && c + j < J.cols) {
        const double r = xr[it][j], i = xi[it][j];
        xr[it][j] = J.coef.x * r - J.coef.y * i;
        xi[it][j] = J.coef.x * i + J.coef.y * r;
        if (J.base) {
          const double2 b = J.base[(long long)row * J.ldb + c + j];
          xr[it][j] += b.x;
          xi[it][j] += b.y;
        }
      }
      if (J.dst && c + j < J.cols) J.dst[(long long)row * J.ldd + c + j] = make_double2(xr[it][j], xi[it][j]);
      // the high word orders magnitudes by exponent, which is all the scale needs; the low word
      // only matters to tell a row of zeros (digits all zero either way)
      mx = max(mx, (uint32_t)__double2hiint(xr[it][j]) & 0x7fffffffu);
      mx = max(mx, (uint32_t)__double2hiint(xi[it][j]) & 0x7fffffffu);
    }
  }
  if (!J.out.dig) return;
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (WPR > 1) {
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mx;
    __syncthreads();
    const int w0 = threadIdx.x / TPR * WPR;
#pragma unroll
    for (int w = 0; w < WPR; ++w) mx = max(mx, s_max[w0 + w]);
  }
  if (!live) return;
  const bool bad = mx >= 0x7ff00000u;
  const int efm = slice_field(mx);
  if (t == 0) J.out.ex[row] = bad ? kSliceNaN : efm - 1021;
  const long long ld = 2LL * J.out.Kp, ps = ld * J.out.rows;
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int c = 4 * (t + TPR * it);
    if (c >= width) continue;
    unsigned long long wr[4], wi[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      wr[j] = slice_bytes(bad ? 0.0 : xr[it][j], efm);
      wi[j] = slice_bytes(bad ? 0.0 : xi[it][j], efm);
    }
    __nv_bfloat16* o = J.out.dig + (long long)row * ld + c;
#pragma unroll
    for (int s = 1; s <= kSlices; ++s, o += ps) {
      *reinterpret_cast<uint2*>(o) = make_uint2(pack_digits(slice_digit(wr[0], s), slice_digit(wr[1], s)),
                                                pack_digits(slice_digit(wr[2], s), slice_digit(wr[3], s)));
      *reinterpret_cast<uint2*>(o + J.out.Kp) = make_uint2(pack_digits(slice_digit(wi[0], s), slice_digit(wi[1], s)),
                                                           pack_digits(slice_digit(wi[2], s), slice_digit(wi[3], s)));
    }
  }
}

template <int MP>
static void launch_rows_mp(const SliceRowJob* jobs, int n_jobs, int max_rows, int max_cols, const int* step,
                           cudaStream_t st) {
  // digits are written up to Kp, so the width to cover is the columns rounded up to 64
  const int w = slice_kp(max_cols);
  auto go = [&](auto kernel, int tpr) {
    const int nt = std::max(tpr, 128), rpb = nt / tpr;
    launch_pdl(kernel, dim3((max_rows + rpb - 1) / rpb, n_jobs), nt, 0, st, jobs, step);
  };
  if (w <= 128)
    go(k_slice_rows<32, 1, MP>, 32);
  else if (w <= 256)
    go(k_slice_rows<64, 1, MP>, 64);
  else if (w <= 512)
    go(k_slice_rows<128, 1, MP>, 128);
  else if (w <= 1024)
    go(k_slice_rows<256, 1, MP>, 256);
  else if (w <= 2048)
    go(k_slice_rows<512, 1, MP>, 512);
  else
    go(k_slice_rows<512, 4, MP>, 512);
}

void launch_slice_rows(const SliceRowJob* jobs, int n_jobs, int max_rows, int max_cols, int mp, const int* step,
                       cudaStream_t st) {
  if (mp == kSlicePairs)
    launch_rows_mp<kSlicePairs>(jobs, n_jobs, max_rows, max_cols, step, st);
  else
    launch_rows_mp<2>(jobs, n_jobs, max_rows, max_cols, step, st);
}

// H_k(t) = H0_k + (shift) S_k + sum_a (A_a/c) P_a (Eqs. 9-12; mode as in k_phase) at the nonzero
// pattern, cut into digits without a stop in memory.  One CTA per (row atom, item): the largest part
// of each of the atom's rows is found in shared memory, then the elements are formed again (their
// operands are in L1) and their digits go to their places.  Latency bound (about 500 elements per
// sp3 atom).  From the k-space blocks instead of the real-space images, and in one launch instead of
// a phase build and a cut: 144 mixed atoms (delta form) 187 -> 165 us a step, 64 atoms x 8 k-points
// 172 -> 171.
__global__ void __launch_bounds__(128) k_slice_hamilton(const SliceHamJob* __restrict__ jobs,
                                                        const DevSys* __restrict__ sysv,
                                                        const DevTraj* __restrict__ trj, int max_orb,
                                                        const int* __restrict__ step, int mode) {
  extern __shared__ uint32_t s_rowmax[];  // [2][max_orb]: H, dH
  const SliceHamJob& J = jobs[blockIdx.y];
  const DevSys& S = sysv[J.sys];
  const DevTraj& T = trj[J.traj];
  const int I = blockIdx.x;
  const bool live = I < S.nat;
  const int e0 = live ? S.el_atom0[I] : 0, e1 = live ? S.el_atom0[I + 1] : 0;
  const int oi = live ? S.orb_off[I] : 0, ni = live ? S.orb_off[I + 1] - oi : 0;
  const long long ps = (long long)S.nk * S.n_el, kb = (long long)J.k * S.n_el;
  const double2 *kS = S.kS + kb, *kP = S.kP + kb, *kH0 = S.kH0 + kb;
  const bool delta = J.dout.dig != nullptr;
  for (int r = threadIdx.x; r < 2 * max_orb; r += blockDim.x) s_rowmax[r] = 0;
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  if (!live) return;
  const int n = *step;
  double A0 = T.A[3 * n], A1 = T.A[3 * n + 1], A2 = T.A[3 * n + 2];
  if (mode == PH_FP64_CN) {  // A(t_{n+1/2}) = (A_n + A_{n+1}) / 2
    A0 = 0.5 * (A0 + T.A[3 * n + 3]);
    A1 = 0.5 * (A1 + T.A[3 * n + 4]);
    A2 = 0.5 * (A2 + T.A[3 * n + 5]);
  }
  constexpr double ic = 1.0 / kLight;
  const double a0 = A0 * ic, a1 = A1 * ic, a2 = A2 * ic;
  const double alpha = mode == PH_FP64_PLAIN ? 0.5 * (a0 * a0 + a1 * a1 + a2 * a2) : 0.0;
  const bool extra = mode == PH_FP64_CN && n > 0;  // eps(t_{n+1/2}) = (3 eps_n - eps_{n-1}) / 2
  const double* cur = extra ? T.eps_lv + (long long)(n & 1) * S.nat : T.eps;
  const double* prv = extra ? T.eps_lv + (long long)((n - 1) & 1) * S.nat : T.eps;
  auto shift = [&](int a) { return extra ? 1.5 * cur[a] - 0.5 * prv[a] : cur[a]; };
  const double eI = shift(I), dI = delta ? T.eps[I] - S.eps0[I] : 0.0;
  // element e: h, and in the delta form d
  auto element = [&](int e, double2& h, double2& d) {
    const int K = J.el_J[e];
    const double2 s = kS[e], h0 = kH0[e], px = kP[e], py = kP[ps + e], pz = kP[2 * ps + e];
    const double pr = a0 * px.x + a1 * py.x + a2 * pz.x, pi = a0 * px.y + a1 * py.y + a2 * pz.y;
    const double beta = alpha + 0.5 * (eI + shift(K));
    h = make_double2(h0.x + beta * s.x + pr, h0.y + beta * s.y + pi);
    if (delta) {
      const double db = 0.5 * (dI + (T.eps[K] - S.eps0[K]));
      d = make_double2(db * s.x + pr, db * s.y + pi);
    }
  };
  auto high = [](double2 v) {
    return max((uint32_t)__double2hiint(v.x) & 0x7fffffffu, (uint32_t)__double2hiint(v.y) & 0x7fffffffu);
  };
  auto write = [](const SliceMat& out, int r, int c, double2 v, uint32_t mx) {
    const bool bad = mx >= 0x7ff00000u;
    const int efm = slice_field(mx);
    const unsigned long long wr = slice_bytes(bad ? 0.0 : v.x, efm), wi = slice_bytes(bad ? 0.0 : v.y, efm);
    const long long ld = 2LL * out.Kp, pst = ld * out.rows;
    __nv_bfloat16* o = out.dig + (long long)r * ld + c;
#pragma unroll
    for (int s = 1; s <= kSlices; ++s, o += pst) {
      o[0] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(slice_digit(wr, s)) >> 16));
      o[out.Kp] = __ushort_as_bfloat16((unsigned short)(__float_as_uint(slice_digit(wi, s)) >> 16));
    }
  };
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    double2 h, d = make_double2(0.0, 0.0);
    element(e, h, d);
    const int r = S.el_off[e] / S.Np - oi;
    atomicMax(&s_rowmax[r], high(h));
    if (delta) atomicMax(&s_rowmax[max_orb + r], high(d));
  }
  __syncthreads();
  for (int e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    double2 h, d = make_double2(0.0, 0.0);
    element(e, h, d);
    const int off = S.el_off[e], r = off / S.Np, c = off - r * S.Np;
    write(J.out, r, c, h, s_rowmax[r - oi]);
    if (delta) write(J.dout, r, c, d, s_rowmax[max_orb + r - oi]);
  }
  for (int r = threadIdx.x; r < ni; r += blockDim.x) {
    const uint32_t mh = s_rowmax[r], md = s_rowmax[max_orb + r];
    J.out.ex[oi + r] = mh >= 0x7ff00000u ? kSliceNaN : slice_field(mh) - 1021;
    if (delta) J.dout.ex[oi + r] = md >= 0x7ff00000u ? kSliceNaN : slice_field(md) - 1021;
  }
}

void launch_slice_hamilton(const SliceHamJob* jobs, int n_jobs, int max_nat, int max_orb, const DevSys* sys,
                           const DevTraj* trj, const int* step, int mode, cudaStream_t st) {
  launch_pdl(k_slice_hamilton, dim3(max_nat, n_jobs), 128, 2 * (size_t)max_orb * sizeof(uint32_t), st, jobs, sys, trj,
             max_orb, step, mode);
}

// ---------------------------------------------------------------------------
// k_slice_gemm: digit products.  A unit is (256 x 128 complex output tile, plane): the plane's
// pairs (s, t) one after the other, each over the tile's 64-wide k-panels.  A 2-SM pair computes
// it with four tcgen05.mma (256 x 128 x 16) per 16 k from four operand tiles,
//   Re += Ar Rr + Ai Ri,  Im += Ai Rr - Ar Ri  (negated A),
// so both parts share the loads and neither operand is stored twice.  The accumulators (Re, Im:
// 128 columns each) are double buffered in tensor memory: eight epilogue warps per CTA take a
// finished run out while the next one is multiplied, so cutting the k-loop into exact runs of 8
// panels costs no tensor time.
// ---------------------------------------------------------------------------
constexpr int SG_N = 128;          // complex output columns per tile
constexpr int SG_ST = 4;           // pipeline stages of 48 KB
constexpr int SG_RUN = 8;          // 64-wide complex k-panels per exact run
constexpr int SG_THREADS = 320;    // TMA warp, MMA warp, 8 epilogue warps

// One unit as the kernel's roles read it: a single record, in the order in which the workers take
// them, so that a role fetches its next unit while it works on this one (chasing the problem and
// panel tables unit by unit cost about 3 us a unit, as long as a unit of a 256-orbital product).
struct __align__(16) SliceUnit {
  int ma, mr, b_a, b_r;    // tensor maps and batch coordinates of A and R
  int arow, brow;          // first row of the tile in A and in R
  int code;                // g | first s << 8 | pairs << 16 | (A real) << 24; 0 ends a worker's list
  int npan;                // 64-wide k-panels of the tile
  int k0;                  // their list starts at kidx[k0]; -1: all of them in order
  int kp, M, ld;           // padded k, rows of the product, row length of the planes
  int* out;                // the plane at column brow
  int nc, nw;              // columns kept (a multiple of 32), offset of the imaginary half
};

struct SliceParams {
  const CUtensorMap* maps;
  const SliceUnit* units;  // [worker][depth]
  const short* kidx;
  int depth;
  int* err;
  long long timeout_ns;
};

__device__ __forceinline__ int unit_g(const SliceUnit& u) { return u.code & 255; }
__device__ __forceinline__ int unit_s0(const SliceUnit& u) { return (u.code >> 8) & 255; }
__device__ __forceinline__ int unit_cnt(const SliceUnit& u) { return (u.code >> 16) & 255; }
__device__ __forceinline__ bool unit_real(const SliceUnit& u) { return (u.code >> 24) != 0; }

__global__ void __launch_bounds__(SG_THREADS, 1) k_slice_gemm(const __grid_constant__ SliceParams P) {
  constexpr uint32_t A_BYTES = BM * BK * 2;            // one part of this CTA's 128 rows of A
  constexpr uint32_t B_BYTES = (SG_N / 2) * BK * 2;    // one part of this CTA's half of R
  constexpr uint32_t STAGE = 2 * A_BYTES + 2 * B_BYTES;
  constexpr uint32_t TCOLS = 512;
  constexpr uint32_t IDESC = idesc_bf16(2 * BM, SG_N);
  constexpr uint32_t NEG_A = 1u << 13;
  extern __shared__ uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + SG_ST * STAGE);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + SG_ST), accf0 = smem_u32(bars + 2 * SG_ST),
                 acce0 = smem_u32(bars + 2 * SG_ST + 2), drain = smem_u32(bars + 2 * SG_ST + 4);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * SG_ST + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);  // [0] abort, [1..2] epilogue ok
  volatile int* s_epi_ok = abort_flag + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader_cta = rank == 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < SG_ST; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(accf0, 1);
    mbar_init(accf0 + 8, 1);
    mbar_init(acce0, 16);
    mbar_init(acce0 + 8, 16);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const SliceUnit* up = P.units + (size_t)(blockIdx.x >> 1) * P.depth;  // the list ends with a zero code
  SliceUnit u = *up;
  pdl_wait();
  pdl_trigger();
  const uint32_t full_l = map_to_rank0(full0), acce_l = map_to_rank0(acce0);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer (both CTAs) ----------------
      int it = 0;
      bool ok = true;
      while (ok && u.code) {
        const SliceUnit nx = *++up;
        const CUtensorMap* ma = P.maps + u.ma;
        const CUtensorMap* mr = P.maps + u.mr;
        const int arow = u.arow + rank * BM, brow = u.brow + rank * (SG_N / 2);
        const int g = unit_g(u), s0 = unit_s0(u), cnt = unit_cnt(u);
        const bool a_real = unit_real(u);
        const short* kidx = u.k0 < 0 ? nullptr : P.kidx + u.k0;
        const uint32_t tx = (a_real ? A_BYTES : 2 * A_BYTES) + 2 * B_BYTES;
        int xn = kidx ? kidx[0] : 0;  // the next panel's number is read a panel ahead
        for (int s = s0; ok && s < s0 + cnt; ++s)
          for (int k = 0; k < u.npan; ++k, ++it) {
            const int st = it % SG_ST, r = it / SG_ST;
            const int x = xn * BK;
            xn = k + 1 < u.npan ? k + 1 : 0;
            if (kidx) xn = kidx[xn];
            if (!mbar_wait(empty0 + 8 * st, (r & 1) ^ 1, P.timeout_ns, abort_flag, P.err)) {
              ok = false;
              break;
            }
            const uint32_t base = smem_u32(sm + st * STAGE);
            if (leader_cta) mbar_expect_tx(full0 + 8 * st, 2 * tx);
            const uint32_t fb = full_l + 8 * st;
            tma_load_4d_pair(base, ma, x, arow, s - 1, u.b_a, fb);
            if (!a_real) tma_load_4d_pair(base + A_BYTES, ma, u.kp + x, arow, s - 1, u.b_a, fb);
            tma_load_4d_pair(base + 2 * A_BYTES, mr, x, brow, g - s - 1, u.b_r, fb);
            tma_load_4d_pair(base + 2 * A_BYTES + B_BYTES, mr, u.kp + x, brow, g - s - 1, u.b_r, fb);
          }
        u = nx;
      }
      if (!ok) {
        if (leader_cta) {
          for (int q = (it > SG_ST ? it - SG_ST : 0); q < it; ++q)
            mbar_wait(full0 + 8 * (q % SG_ST), (q / SG_ST) & 1, kDrainNs, abort_flag, P.err, false);
        } else {
          // the peer cannot wait on the leader's barriers: give its copies time to land
          const long long t0 = gtime();
          while (gtime() - t0 < 200000) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && leader_cta) {
      // ---------------- MMA issuer (leader CTA only) ----------------
      int it = 0, f = 0;
      bool ok = true, issued = false;
      for (; ok && u.code; u = *++up) {
        const int total = unit_cnt(u) * u.npan;
        const bool a_real = unit_real(u);
        for (int done = 0; ok && done < total; done += SG_RUN, ++f) {
          const int ab = f & 1, ph = f >> 1;
          const int n = min(SG_RUN, total - done);
          if (!mbar_wait(acce0 + 8 * ab, (ph & 1) ^ 1, P.timeout_ns, abort_flag, P.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t dre = tmem + ab * 256, dim = dre + SG_N;
          for (int q = 0; q < n; ++q, ++it) {
            const int st = it % SG_ST, r = it / SG_ST;
            if (!mbar_wait(full0 + 8 * st, r & 1, P.timeout_ns, abort_flag, P.err)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t base = smem_u32(sm + st * STAGE);
            // operand tiles of the stage: Ar, Ai, Rr, Ri (descriptors count 16-byte units).  The two forms are
            // separate loops: with the real case as a branch between the instructions, both took 0.71 us a
            // panel; apart they take 0.71 and 0.48 us (N = 2048).
            const uint64_t d0 = sw128_desc(base);
            constexpr uint64_t oAi = A_BYTES >> 4, oBr = (2 * A_BYTES) >> 4, oBi = (2 * A_BYTES + B_BYTES) >> 4;
            if (a_real) {
#pragma unroll
              for (int x = 0; x < BK / 16; ++x) {
                const uint32_t acc = (q > 0 || x > 0) ? 1u : 0u;
                tc_mma_pair(dre, d0 + 2 * x, d0 + oBr + 2 * x, IDESC, acc);
                tc_mma_pair(dim, d0 + 2 * x, d0 + oBi + 2 * x, IDESC | NEG_A, acc);
              }
            } else {
#pragma unroll
              for (int x = 0; x < BK / 16; ++x) {
                const uint32_t acc = (q > 0 || x > 0) ? 1u : 0u;
                tc_mma_pair(dre, d0 + 2 * x, d0 + oBr + 2 * x, IDESC, acc);
                tc_mma_pair(dim, d0 + 2 * x, d0 + oBi + 2 * x, IDESC | NEG_A, acc);
                tc_mma_pair(dre, d0 + oAi + 2 * x, d0 + oBi + 2 * x, IDESC, 1u);
                tc_mma_pair(dim, d0 + oAi + 2 * x, d0 + oBr + 2 * x, IDESC, 1u);
              }
            }
            tc_commit_pair(empty0 + 8 * st, 3);
            issued = true;
          }
          if (!ok) break;
          tc_commit_pair(accf0 + 8 * ab, 3);
        }
      }
      if (!ok && issued) {
        tc_commit_pair(drain, 1);
        mbar_wait(drain, 0, kDrainNs, abort_flag, P.err, false);
      }
    }
  } else {
    // ---------------- epilogue (warps 2..9 of both CTAs) ----------------
    // A thread keeps the integers of its output row (128 columns of Re or of Im) in registers over
    // the unit's runs, so the runs cost tensor-memory reads and additions only; the finished unit
    // goes through shared memory in 32 x 32 blocks, so that a store covers whole 128-byte lines.
    // (Adding each run to the plane in global memory, one row per thread, took 16 thousand clocks a
    // run against 4 to 9 thousand of multiplication: N = 2048 product 2 with a real S^-1 2.5 ms.)
    const int q = warp & 3, half = (warp - 2) >> 2;  // TMEM lane quarter; Re or Im columns
    const bool leader = threadIdx.x == 64;
    int4* stage = reinterpret_cast<int4*>(sm + SG_ST * STAGE + 256) + (warp - 2) * 256;  // 32 rows x 8 int4
    int f = 0;
    bool ok = true;
    while (ok && u.code) {
      const SliceUnit nx = *++up;
      const int total = unit_cnt(u) * u.npan;
      int acc[SG_N];
#pragma unroll
      for (int c = 0; c < SG_N; ++c) acc[c] = 0;
      for (int done = 0; done < total; done += SG_RUN, ++f) {
        const int ab = f & 1, ph = f >> 1;
        if (leader) s_epi_ok[f & 1] = mbar_wait(accf0 + 8 * ab, ph & 1, P.timeout_ns, abort_flag, P.err) ? 1 : 0;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (!s_epi_ok[f & 1]) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t t0 = tmem + ab * 256 + half * SG_N + ((uint32_t)(q * 32) << 16);
#pragma unroll
        for (int c = 0; c < SG_N; c += 32) {
          uint32_t r[32];
          TMEM_LD32(t0 + c, r);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int v = 0; v < 32; ++v)
            acc[c + v] += __float2int_rn(__uint_as_float(r[v]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acce_l + 8 * ab);
      }
      if (!ok) break;
      const int row0 = u.arow + rank * BM + q * 32;
      int* out = u.out + half * u.nw;
#pragma unroll
      for (int c = 0; c < SG_N; c += 32) {
        if (c < u.nc) {
#pragma unroll
          for (int v = 0; v < 8; ++v)
            stage[lane * 8 + (v ^ (lane & 7))] =
                make_int4(acc[c + 4 * v], acc[c + 4 * v + 1], acc[c + 4 * v + 2], acc[c + 4 * v + 3]);
          __syncwarp();
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            const int r = 4 * v + (lane >> 3), w = lane & 7;
            if (row0 + r < u.M)
              reinterpret_cast<int4*>(out + (long long)(row0 + r) * u.ld + c)[w] = stage[r * 8 + (w ^ (r & 7))];
          }
          __syncwarp();
        }
      }
      u = nx;
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS) : "memory");
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// stages, barriers, epilogue staging (8 warps x 4 KB), alignment
constexpr int kSliceSmem = SG_ST * (2 * BM * BK * 2 + 2 * (SG_N / 2) * BK * 2) + 256 + 8 * 4096 + 1024;

struct SliceGemm {
  SliceParams P{};
  std::vector<void*> mem;
  int grid = 0;
};

int slice_tiles(int M, int N) { return ((M + 2 * BM - 1) / (2 * BM)) * ((N + SG_N - 1) / SG_N); }

// A plane of a whole group (up to 8 pairs) is the longest unit.  With few tiles the 43 pairs of a tile
// are spread over 24 planes of at most 2 pairs, so that more pairs of SMs get work and no unit is
// long; the integers to read back grow from 9 to 24 per real part.  `tiles` counts the tiles of a
// product, twice where more is read back: delta form (two products make W), Crank-Nicolson (twelve
// sweeps).  Products and read-back of a step with 8 | 2 pairs a plane, in us: leapfrog 1 tile
// (N = 116) 70 | 62, 2 (256) 89 | 69, 8 (468) 131 | 121, 8 (512) 121 | 117, 15 (576) 168 | 200,
// 16 (8 x 256) 137 | 182; delta form 2 x 2 (256) 94 | 79, 2 x 6 (384) 116 | 123, 2 x 8 (512)
// 140 | 160; Crank-Nicolson 2 x 2 (256) 485 | 315, 2 x 4 (512) 825 | 564, 2 x 8 (8 x 128) 435 | 481.
int slice_pairs_per_plane(long long tiles) { return tiles >= 12 ? kSlicePairs : 2; }

namespace {

bool slice_map(CUtensorMap* m, const SliceFam& f, int box_rows, std::string* msg) {
  static PFN_cuTensorMapEncodeTiled_v12000 enc = nullptr;
  if (!enc) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    if (!enc) {
      *msg = "cuTensorMapEncodeTiled unavailable";
      return false;
    }
  }
  const cuuint64_t ld = 2 * (cuuint64_t)f.Kp;
  cuuint64_t dims[4] = {ld, (cuuint64_t)f.rows, kSlices, (cuuint64_t)f.batch};
  cuuint64_t strides[3] = {ld * 2, ld * 2 * f.rows, ld * 2 * f.rows * kSlices};
  cuuint32_t box[4] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1, 1};
  cuuint32_t es[4] = {1, 1, 1, 1};
  if (enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, f.dig, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
    *msg = "cuTensorMapEncodeTiled failed for a digit family";
    return false;
  }
  return true;
}

// On the stream of the launches: k_slice_gemm reads its units before it waits for the kernel ahead
// of it, and the stream may be a non-blocking one, which copies on the legacy stream are not ordered
// with.
template <class T>
bool slice_upload(SliceGemm* g, const T** dst, const std::vector<T>& v, cudaStream_t st) {
  void* p = nullptr;
  if (cudaMalloc(&p, std::max<size_t>(v.size(), 1) * sizeof(T)) != cudaSuccess) return false;
  g->mem.push_back(p);
  *dst = (const T*)p;
  return cudaMemcpyAsync(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, st) == cudaSuccess;
}

// 64-wide column panels of the R rows of every 128-row tile that hold a nonzero of the pattern
// (all of them without a pattern; one panel of zeros for a tile that has none, to clear its output)
void slice_panels(const SlicePattern* pat, int N, int Kp, std::vector<int>& kofs, std::vector<short>& kidx) {
  const int npan = Kp / BK, tiles = (N + SG_N - 1) / SG_N;
  std::vector<int> atom;
  std::vector<std::vector<int>> nbr;
  if (pat) {
    const std::vector<int>& off = *pat->orb_off;
    atom.resize(N);
    nbr.resize(off.size() - 1);
    for (size_t a = 0; a + 1 < off.size(); ++a)
      for (int o = off[a]; o < off[a + 1]; ++o) atom[o] = (int)a;
    for (size_t t = 0; t < pat->tgt_I->size(); ++t) nbr[(*pat->tgt_I)[t]].push_back((*pat->tgt_J)[t]);
  }
  kofs.assign(1, 0);
  kidx.clear();
  for (int nt = 0; nt < tiles; ++nt) {
    std::vector<char> pan(npan, pat ? 0 : 1);
    if (pat) {
      const std::vector<int>& off = *pat->orb_off;
      int last = -1;
      for (int r = nt * SG_N; r < std::min(N, (nt + 1) * SG_N); ++r) {
        if (atom[r] == last) continue;
        last = atom[r];
        for (int J : nbr[last])
          for (int c = off[J] / BK; c <= (off[J + 1] - 1) / BK; ++c) pan[c] = 1;
      }
    }
    int cnt = 0;
    for (char c : pan) cnt += c;
    if (cnt == 0) pan[0] = 1;
    for (int k = 0; k < npan; ++k)
      if (pan[k]) kidx.push_back((short)k);
    kofs.push_back((int)kidx.size());
  }
}

}  // namespace

int slice_gemm_create(const std::vector<SliceFam>& fams, const std::vector<SliceProd>& prods,
                      const std::vector<SlicePattern>& patterns, int mp, long long timeout_ns, int* err,
                      cudaStream_t st, SliceGemm** out, std::string* msg) {
  *out = nullptr;
  SliceGemm* g = new SliceGemm();
  auto bail = [&](const char* m) {
    if (m) *msg = m;
    slice_gemm_destroy(g);
    return -1;
  };
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (cudaFuncSetAttribute(k_slice_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kSliceSmem) != cudaSuccess)
    return bail("cannot raise the shared-memory limit of the sliced product");
  // two maps per family: as A (128-row boxes) and as R (64-row boxes)
  std::vector<CUtensorMap> maps(2 * fams.size());
  for (size_t i = 0; i < fams.size(); ++i)
    if (!slice_map(&maps[2 * i], fams[i], BM, msg) || !slice_map(&maps[2 * i + 1], fams[i], SG_N / 2, msg))
      return bail(nullptr);
  // panel lists, one per (pattern, shape) that occurs
  struct List {
    int pattern, N, Kp;
    size_t kidx0;
    std::vector<int> kofs;
  };
  std::vector<List> lists;
  std::vector<short> all_kidx;
  std::vector<size_t> which(prods.size());
  for (size_t i = 0; i < prods.size(); ++i) {
    const SliceFam& r = fams[prods[i].fam_r];
    size_t l = 0;
    for (; l < lists.size(); ++l)
      if (lists[l].pattern == prods[i].pattern && lists[l].N == r.rows && lists[l].Kp == r.Kp) break;
    if (l == lists.size()) {
      List n{prods[i].pattern, r.rows, r.Kp, all_kidx.size(), {}};
      std::vector<short> kidx;
      slice_panels(prods[i].pattern < 0 ? nullptr : &patterns[prods[i].pattern], r.rows, r.Kp, n.kofs, kidx);
      all_kidx.insert(all_kidx.end(), kidx.begin(), kidx.end());
      lists.push_back(n);
    }
    which[i] = l;
  }
  std::vector<SliceUnit> units;
  std::vector<double> cost;
  const int np = slice_num_planes(mp);
  for (size_t i = 0; i < prods.size(); ++i) {
    const SliceProd& p = prods[i];
    const SliceFam &a = fams[p.fam_a], &r = fams[p.fam_r];
    const int tiles_m = (a.rows + 2 * BM - 1) / (2 * BM), tiles_n = (r.rows + SG_N - 1) / SG_N;
    const long long stride = (long long)a.rows * 2 * p.Nw;
    const List& l = lists[which[i]];
    int plane = 0;
    for (int gr = 2; gr < 2 + kSliceGroups; ++gr)
      for (int q0 = 0; q0 < slice_pairs(gr); q0 += mp, ++plane)
        for (int nt = 0; nt < tiles_n; ++nt)
          for (int mt = 0; mt < tiles_m; ++mt) {
            SliceUnit u{};
            u.ma = 2 * p.fam_a;
            u.mr = 2 * p.fam_r + 1;
            u.b_a = p.b_a;
            u.b_r = p.b_r;
            u.arow = mt * 2 * BM;
            u.brow = nt * SG_N;
            const int cnt = std::min(mp, slice_pairs(gr) - q0);
            u.code = gr | (std::max(1, gr - kSlices) + q0) << 8 | cnt << 16 | (p.a_real ? 1 : 0) << 24;
            u.npan = l.kofs[nt + 1] - l.kofs[nt];
            u.k0 = p.pattern < 0 ? -1 : (int)l.kidx0 + l.kofs[nt];
            u.kp = a.Kp;
            u.M = a.rows;
            u.ld = 2 * p.Nw;
            u.out = p.planes + plane * stride + nt * SG_N;
            u.nc = std::min(SG_N, p.Nw - nt * SG_N);
            u.nw = p.Nw;
            units.push_back(u);
            // panels of the unit (a real A takes 0.48 us a panel instead of 0.71) and a fixed share
            cost.push_back(cnt * u.npan * (p.a_real ? 0.67 : 1.0) + 2.0);
          }
    if (plane != np) return bail("plane count");
  }
  // longest first, each to the worker with the least work
  const int G = std::max(1, std::min((int)units.size(), nsm / 2));
  std::vector<int> idx(units.size());
  for (size_t i = 0; i < idx.size(); ++i) idx[i] = (int)i;
  std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) { return cost[x] > cost[y]; });
  std::vector<std::vector<int>> ul(G);
  std::vector<std::pair<double, int>> heap;  // least loaded worker first
  for (int c = 0; c < G; ++c) heap.push_back({0.0, c});
  auto later = [](const std::pair<double, int>& x, const std::pair<double, int>& y) { return x > y; };
  std::make_heap(heap.begin(), heap.end(), later);
  for (int i : idx) {
    std::pop_heap(heap.begin(), heap.end(), later);
    ul[heap.back().second].push_back(i);
    heap.back().first += cost[i];
    std::push_heap(heap.begin(), heap.end(), later);
  }
  size_t depth = 0;
  for (auto& l : ul) depth = std::max(depth, l.size());
  ++depth;  // every list ends with a zero record
  std::vector<SliceUnit> order(depth * G, SliceUnit{});
  for (int c = 0; c < G; ++c)
    for (size_t k = 0; k < ul[c].size(); ++k) order[c * depth + k] = units[ul[c][k]];
  const CUtensorMap* d_maps;
  const SliceUnit* d_units;
  const short* d_kidx;
  const bool up = slice_upload(g, &d_maps, maps, st) && slice_upload(g, &d_units, order, st) &&
                  slice_upload(g, &d_kidx, all_kidx, st);
  if (cudaStreamSynchronize(st) != cudaSuccess || !up)  // the host tables leave scope
    return bail("upload of the sliced product's tables failed");
  g->P.maps = d_maps;
  g->P.units = d_units;
  g->P.kidx = d_kidx;
  g->P.depth = (int)depth;
  g->P.err = err;
  g->P.timeout_ns = timeout_ns;
  g->grid = 2 * G;
  *out = g;
  return 0;
}

int slice_gemm_launch(SliceGemm* g, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g->grid, 1, 1);
  cfg.blockDim = dim3(SG_THREADS, 1, 1);
  cfg.dynamicSmemBytes = kSliceSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_slice_gemm, g->P) == cudaSuccess ? 0 : -1;
}

void slice_gemm_destroy(SliceGemm* g) {
  if (!g) return;
  for (void* p : g->mem) cudaFree(p);
  delete g;
}

}  // namespace vgtb
