// Column solver: one thread-block cluster runs a whole inner pass of one
// Sternheimer unit (a pair of columns that are real in real space, or one
// complex column) in (distributed) shared memory.  See col_kernel.cuh.
#pragma once

#include "gw_common.cuh"

namespace gw {

// Transform lengths N = N1 N2 the kernel has radices for (N1 in {3,4,5,6,8},
// N2 in {4,5,6,8,9,10}); false for any other N.
bool col_radices(int N, int* N1, int* N2);

constexpr int kColMaxQ = 16;                       // largest cluster (non-portable size)
constexpr int kColNQ = 5;                          // cluster sizes 1, 2, 4, 8, 16

// Sphere entries in half-sphere order, fixed per cell.  The disc pencils
// (i0, i1) come in mirror pairs j = 0 .. npair - 1 (pair 0: the pencil (0, 0),
// its own mirror); half entry h stands for G (in the pair's first pencil) and
// -G (in the second); h = 0 is G = 0.  The CTA of rank r in a cluster of Q owns
// the pairs split[lq][r] .. split[lq][r + 1] (lq = log2 Q) and their entries.
struct ColPlan {
  bool ok = false;                                 // the column solver has radices for N
  int N1 = 0, N2 = 0, P = 0, nm = 0;               // planes |n0| <= nm: P = 2 nm + 1
  int npair = 0, nh = 0;
  int maxpair[kColNQ] = {0}, maxh[kColNQ] = {0};   // per CTA, by log2 Q
  int* split = nullptr;                            // [kColNQ][kColMaxQ + 1]
  int* hstart = nullptr;                           // [npair + 1]
  int* gp = nullptr;                               // [nh] sphere index of G
  int* gm = nullptr;                               // [nh] sphere index of -G
  unsigned* hpos = nullptr;                        // [nh] pair << 8 | i2
  unsigned short* disc = nullptr;                  // [N][P] pair << 1 | mirror of (i1, plane), 0xffff outside
  unsigned char* zmax = nullptr;                   // [npair] largest |n2| of the pair's pencils
};

template <typename T> struct ColPrec {
  T* Vp = nullptr;        // [N i2][N i0][N slot] V / N_g, i1 in the slot order of the first transform
  cpx<T>* Ch = nullptr;   // [rows][nh] projector rows at G
  T* kin = nullptr;       // [nh] |G|^2 / 2
};

// kind of inner solve
enum ColKind { COL_CG_PAIR = 0, COL_QMR = 1, COL_QMR_PAIR = 2 };

// Shape of a launch.
struct ColShape {
  int lq = 0, nsb = 1;           // log2 of the cluster size; slabs transformed together
  bool vec_smem = false;         // solver vectors in shared memory (else in vecs)
  bool c_smem = false;           // projector rows in shared memory
  bool v_smem = false;           // the slabs' potential in shared memory
  size_t smem = 0;
  size_t vec_elems = 0;          // T entries of the global vectors of one unit (0 with vec_smem)
};

template <typename T>
struct ColArgs {
  ColShape sh;
  int N, P, nm, npair, nh, npw, nproj, ncol, nunit, maxit;
  int ldz, nhl;                  // rows of Z (2 maxpair), entries per CTA (maxh)
  FastDiv dP, dnz;               // by P and by the slabs per CTA
  const cpx<T>* tw;
  const T* Vp;
  const cpx<T>* Ch;
  const T* kin;
  const int *split, *hstart, *gp, *gm;
  const unsigned* hpos;
  const unsigned short* disc;
  const unsigned char* zmax;
  const double2* b64;            // [ncol][npw] right-hand sides
  double2* x64;                  // [ncol][npw] the solution of the pass is added here
  const int* outer_active;       // [ncol] or null
  const double2* E;              // [ncol]
  const double* rr_abs;          // [ncol] or null
  const double* tk;              // [ncol] or null
  double tol2;
  double v0;                     // level of V in the outer parts of the cell (two thirds lie below it)
  T* vecs;                       // [nunit][vec_elems]
  int* iters;                    // [ncol]
  int* flags;                    // [ncol]
  double* xmax;                  // [ncol] largest component of x64 (to a factor 2), for the pairs of the residual
};

// FP64 projector and residual on half entries (kernels_half.cu); rows are
// ColPrec<double>::Ch, real: columns real in real space.  launch_gram_half
// leaves the coefficients <C|Y> in partial sums (half_part_elems) and returns
// the number of parts for the kernels that use them:
//   launch_proj_half      Y -= C coef
//   launch_residual_half  r -= C coef; out[3][ncol] = |r|^2, |b|^2, |x|^2
size_t half_part_elems(int nrow, int nh, int ncol);
size_t half_sum_elems(int nh, int ncol);
int launch_gram_half(cudaStream_t s, bool real, const ColPlan& p, const double2* Ch, int nrow, const double2* Y,
                     int npw, int ncol, const int* active, double* part);
void launch_proj_half(cudaStream_t s, bool real, const ColPlan& p, const double2* Ch, int nrow, double2* Y, int npw,
                      int ncol, const int* active, int nchunk, const double* part);
void launch_residual_half(cudaStream_t s, bool real, const ColPlan& p, const double2* Ch, int nrow, double2* r,
                          const double2* b, const double2* x, int npw, int ncol, const int* active, int nchunk,
                          const double* part, double* sums, unsigned* cnt, double* out);

// The fastest shape for nunit units on 1 / cta_div of the GPU (false: no
// cluster size fits).
template <typename T>
bool col_shape(const ColPlan& p, int kind, int N, int nproj, int nunit, int cta_div, ColShape* out);
template <typename T>
cudaError_t launch_col_solve(cudaStream_t s, int kind, const ColArgs<T>& a);
template <typename T>
cudaError_t launch_col_permute(cudaStream_t s, const ColPlan& p, int N, int npw, const T* vloc_s, const cpx<T>* C,
                               int nproj, const T* kin, ColPrec<T>& out);

}  // namespace gw
