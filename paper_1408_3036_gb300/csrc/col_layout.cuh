// Column solver: shared-memory layout of one CTA (kernel and launch).
#pragma once

#include <type_traits>

#include "col.cuh"
#include "sums.cuh"

namespace gw {
namespace col {

// Threads of a CTA (640 for lengths where that makes the rounds of the x passes
// even, 768 and 1024 were no faster: 48^3 mixed 1.65 against 1.67, 1.69, 1.8 ms)
constexpr int kTPB = 512;
constexpr int kNW = kTPB / 32;
constexpr size_t kSmemMax = 226 * 1024;
// Sums over entries, as exact as those of the solvers they stand for (sums.cuh).
// FP64 throughout in FP64.  FP32 CG: scalars in two floats, projector
// coefficients in one, as the persistent CG.  FP32 SQMR: scalars in three floats
// (the launches per step sum in FP64), coefficients in plain FP32 over 8 entries
// of a lane, then two floats (launches per step: FP32 within a tile of 16
// pencils, FP64 over the tiles; the FP32 part decides).
template <typename T, int KIND>
using ScalarAcc = typename std::conditional<KIND == COL_CG_PAIR, Acc<T>, Acc3<T>>::type;
template <typename T, int KIND> using CoefAcc = typename std::conditional<KIND == COL_CG_PAIR, T, Acc<T>>::type;

// Shared memory of one CTA (byte offsets)
struct Lay {
  size_t Z, R, T, X, C, V, K, kin, hpos, rt, own, zm, zs, tw, cp, coefp, coef, part, sc, total;
};
__host__ __device__ inline size_t up16(size_t x) { return (x + 15) & ~(size_t)15; }
// Projector rows a warp takes at a time (their products with one load of the
// vectors), and the parts the entries are cut into so that all warps work.
__host__ __device__ inline int row_group(int nproj, bool f32) {
  if (nproj < 8) return nproj < 4 ? 1 : 2;
  if (!f32 || nproj <= 4 * kNW) return 4;
  return nproj <= 5 * kNW ? 5 : nproj <= 6 * kNW ? 6 : 4;
}
__host__ __device__ inline int splits(int nproj, int rg, int nhl) {
  const int g = (nproj + rg - 1) / rg, s = g > 0 ? kNW / g : 1, m = (nhl + 31) / 32;
  return s < 1 ? 1 : s > m ? m : s;
}

template <typename T>
__host__ __device__ inline Lay layout(int kind, const ColShape& sh, int N, int P, int npair, int ldz, int nhl,
                                      int nproj) {
  const size_t sv = sizeof(cpx<T>), s4 = 4 * sizeof(T);
  const int Q = 1 << sh.lq, nzl = (N + Q - 1) / Q, nv = kind == COL_CG_PAIR ? 4 : 2;
  const int rg = row_group(nproj, sizeof(T) == 4);
  const bool cg = kind == COL_CG_PAIR;
  const size_t sc = cg ? sizeof(CoefAcc<T, COL_CG_PAIR>) : sizeof(CoefAcc<T, COL_QMR>);
  const size_t ss = cg ? sizeof(ScalarAcc<T, COL_CG_PAIR>) : sizeof(ScalarAcc<T, COL_QMR>);
  const size_t tile = (size_t)sh.nsb * N * (N | 1) * sv, temp = (size_t)nhl * s4 * (kind == COL_CG_PAIR ? 2 : 1);
  Lay L;
  L.Z = 0;
  L.R = up16(L.Z + (size_t)N * ldz * sv);
  L.T = up16(L.R + (Q > 1 ? (size_t)nzl * (2 * npair) * sv : 0));
  L.X = up16(L.T + (tile > temp ? tile : temp));
  L.C = up16(L.X + (sh.vec_smem ? 4 * (size_t)nhl * s4 : 0));
  L.V = up16(L.C + (sh.c_smem ? (size_t)nproj * nhl * sv : 0));
  L.K = up16(L.V + (sh.v_smem ? (size_t)nzl * N * N * sizeof(T) : 0));
  L.kin = up16(L.K + (size_t)nhl * 2 * sizeof(T));
  L.hpos = up16(L.kin + (size_t)nhl * sizeof(T));
  L.rt = up16(L.hpos + (size_t)nhl * sizeof(unsigned));
  L.own = up16(L.rt + (size_t)N * P * sizeof(unsigned short));
  L.zm = up16(L.own + (size_t)2 * npair);
  L.zs = up16(L.zm + (size_t)ldz);
  L.tw = up16(L.zs + (size_t)N);
  L.cp = up16(L.tw + (size_t)N * sv);
  L.coefp = up16(L.cp + (size_t)splits(nproj, rg, nhl) * nproj * nv * sc);
  L.coef = up16(L.coefp + (size_t)Q * nproj * nv * sc);
  L.part = up16(L.coef + (size_t)nproj * nv * sizeof(T));
  L.sc = up16(L.part + (size_t)kNW * 4 * ss);
  L.total = up16(L.sc + (size_t)3 * Q * 4 * ss);
  return L;
}

// The kernel of transform length A B (one translation unit per few lengths).
template <typename T, int A, int B> const void* kernel_ptr(int kind);

}  // namespace col
}  // namespace gw
