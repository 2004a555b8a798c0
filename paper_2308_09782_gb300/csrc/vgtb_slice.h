// Host interface of the sliced FP64 products (k_slice.cu; scheme in slice.cuh).
#pragma once
#include <string>
#include <vector>

#include "slice.cuh"

namespace vgtb {

// Rows to be cut into digits: taken from a matrix, from the planes of a product,
// or from both sets of planes added up; optionally base + coef x value; stored to
// dst and / or cut into digits.
struct SliceRowJob {
  int rows, cols;
  const double2* src;      // matrix source, or null
  long long src_par;       // src + ((*step) & 1) * src_par
  int lds;
  int n_planes;            // plane sources (0, 1, 2)
  SlicePlanes pl[2];
  const double2* base;     // value = base + coef * value when epi != 0 (base may be null)
  int ldb, epi;
  double2 coef;
  double2* dst;            // optional
  int ldd;
  SliceMat out;            // digits wanted when out.dig != null
};
// mp: pairs per plane of the sources (8 or 2)
void launch_slice_rows(const SliceRowJob* jobs, int n_jobs, int max_rows, int max_cols, int mp, const int* step,
                       cudaStream_t st);

// H_k(t) (delta form: and dH_k(t)) of one item from the k-space blocks S_k, H0_k, P_k, straight to
// digits: positions off the nonzero pattern are left as they are (zeros).
struct SliceHamJob {
  int sys, traj, k;
  const int* el_J;         // [n_el] column atom of every nonzero
  SliceMat out, dout;      // H; dH in the delta form, else dout.dig == null
};
void launch_slice_hamilton(const SliceHamJob* jobs, int n_jobs, int max_nat, int max_orb, const DevSys* sys,
                           const DevTraj* trj, const int* step, int mode, cudaStream_t st);

// One operand family: the digits of `batch` matrices of one shape, contiguous.
struct SliceFam {
  __nv_bfloat16* dig = nullptr;
  int* ex = nullptr;
  int rows = 0, K = 0, Kp = 0, batch = 0;
  SliceMat mat(int b) const {
    SliceMat m{};
    if (!dig) return m;
    m.dig = dig + (size_t)b * kSlices * rows * 2 * Kp;
    m.ex = ex + (size_t)b * rows;
    m.rows = rows;
    m.K = K;
    m.Kp = Kp;
    return m;
  }
};

// Nonzero pattern of an R operand (H): orbital offsets and the atom pairs (I, J) of the targets.
struct SlicePattern {
  const std::vector<int>* orb_off = nullptr;
  const std::vector<int>* tgt_I = nullptr;
  const std::vector<int>* tgt_J = nullptr;
};

// product i: planes[i] = A[fam_a[i]][b_a] R[fam_r[i]][b_r]^dagger
struct SliceProd {
  int fam_a, b_a, fam_r, b_r;
  int* planes;
  int Nw;
  bool a_real;             // every imaginary part of A is zero
  int pattern;             // index into the patterns, or -1
};

struct SliceGemm;
int slice_pairs_per_plane(long long tiles);  // 8, or 2 when few units of whole groups leave the chip idle
int slice_tiles(int M, int N);
int slice_gemm_create(const std::vector<SliceFam>& fams, const std::vector<SliceProd>& prods,
                      const std::vector<SlicePattern>& patterns, int mp, long long timeout_ns, int* err,
                      cudaStream_t st, SliceGemm** out,
                      std::string* msg);  // err: device word that an expired wait sets; st: the stream of the launches
int slice_gemm_launch(SliceGemm* g, cudaStream_t st);
void slice_gemm_destroy(SliceGemm* g);
inline int slice_kp(int K) { return (K + 63) / 64 * 64; }
inline int slice_nw(int N) { return (N + 31) / 32 * 32; }
inline int slice_num_planes(int mp) { return mp == kSlicePairs ? slice_planes<kSlicePairs>() : slice_planes<2>(); }

}  // namespace vgtb
