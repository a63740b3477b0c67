// Column solver (Eq. P2 inside the FP64 refinement): one thread-block cluster
// of Q = 1, 2, 4, 8 or 16 CTAs runs the whole inner pass of one unit,
//   COL_CG_PAIR   two columns that are real in real space, conjugate gradients
//   COL_QMR       one complex column, simplified QMR (bilinear form)
//   COL_QMR_PAIR  two real columns with real shifts, simplified QMR
// with everything an iteration exchanges in (distributed) shared memory; units
// do not wait for one another, and no iteration returns to the host.
//
// Work split.  The CTA of rank r owns a contiguous range of mirror pairs of
// disc pencils {(i0, i1), (-i0, -i1)} -- so G and -G live in the same CTA --
// and the slabs i2 = r nzl .. (r + 1) nzl.  One application of H:
//   scatter, z-IFFT of the own pencils, values sent to the slab owners
//   per slab: y-IFFT of the planes |n0| <= nm, x-IFFT, * V(r)/N_g, x-FFT,
//     y-FFT, the disc values sent back to the pencil owners
//   z-FFT, gather, kinetic part
// so that only the disc's values (npen N) cross the cluster, twice.
//
// Transforms.  N = N1 N2, both radices in registers: step 1 takes
// x[n1 N2 + n2] over n1 and leaves k1 in its place (times w_N^(k1 n2)), step 2
// takes n2 over N2 contiguous slots and leaves X[k1 + N1 k2] at slot
// k1 N2 + k2.  The way back runs the transposed steps from that slot order to
// natural order, so every pass is in place, no pass only reorders, and the
// second x step, the product with V and the first step back are one pass.
//
// Half-sphere storage.  A half entry h stands for G and -G (h = 0: G = 0).
// A real column has c(-G) = conj c(G): one complex value per half entry and
// real projector coefficients; a pair shares the transform as u_0 + i u_1.  A
// complex column keeps both values.  The projector rows are real in real space
// too, so <C|y> = sum_h conj(c) y(G) + c y(-G) takes 4 real products per row
// and half entry for either kind, half of what the full sphere takes, and half
// of the rows' bytes.
//
// Preconditioner.  The diagonal of H - E at the column's own shift, kept away
// from zero: with V0 the level below which V lies in two thirds of the cell and
// d = |G|^2/2 + V0 - Re E,
//   real shift     K = 1 / sqrt(d^2 + 0.03^2)   (positive, as CG needs)
//   complex shift  K = 1 / (d - i (Im E + 0.2 sgn Im E))
// V0 because a constant in V and the energies changes nothing (without it 16^3,
// 179 plane waves, V + 3 Ha: static 20 -> 166 iterations, 0.957 + 0.1 i 32 ->
// 174); not the mean, the diagonal's own, because P_c takes away the states of
// the wells (mean: 24^3, 619 plane waves, static 18 -> 25 iterations).
// K(-G) = K(G), so it is symmetric in the bilinear form too.  The
// Teter-Payne-Allan form of the other kernels knows the kinetic energy of the
// occupied state but not the shift.  Iterations to 1e-5 (FP64), then and now:
// 32^3, 2109 plane waves, 0.957 + 0.1 i: 170 -> 46 for the slow sign, 11 -> 7
// for the other; 45^3, 0.3 + 0.1 i 55 -> 35 and 15 -> 10; static 32^3 10 -> 7,
// 48^3 29 -> 25 (slowest column) and 10 -> 7 (fastest).
//
// Scalars of the recurrences come from ordered sums that every CTA of the
// cluster forms from the same partial sums: all CTAs decide alike.
//
// What bounds it: FP32 the latency of one unit's iteration (48^3, 16 rows, Q =
// 16: 39k cycles, of which the slabs' seven passes 13k, z passes 4k, update 4k,
// projector 5k, three cluster barriers and scalar steps the rest), and the
// occupied rows where they don't fit beside the vectors: 69 rows of 1055
// entries, read twice an iteration by every SM at about 12 TB/s out of L2, 31k
// of 110k cycles.  FP64 the FP64 pipe, which takes one warp instruction in 64
// cycles and scheduler here: sums are halved across the lanes instead of
// repeated in them, scalar steps share one division, products are accumulated
// in chains of fused multiply-adds (a += x y + z w is three instructions, not
// two) and the transforms keep the fewest operations (dft in fft.cuh).
// Measured on a GB300, one application, before (launches per step, or the
// grid-wide task queue of kernels_cg.cu, with the Teter-Payne-Allan form) and
// after, both sides in one run: 48^3 grid, 12053 plane waves, 16 CG columns, FP32
// 3.69 -> 1.58 ms, FP64 15.8 -> 8.9 ms; 45^3, 2007 plane waves, 22 complex columns
// 11.7 -> 2.29 ms; 32^3, 2109 plane waves, 69 rows, 1104 complex columns 398 ->
// 29.9 ms; 64^3, 38401 plane waves, 64 rows, 256 complex columns 1044 -> 111 ms
// (of the last two, columns that stalled on the rounding floor took 120 .. 400 ms
// before, more or fewer by the input: 232 and 837 ms at least).  What the scaling
// of the columns costs of that: a second read of b and one barrier a pass, 0.5 to
// 1%; the exact sums of FP32 SQMR: 2 to 3%.
#pragma once

#include <cooperative_groups.h>

#include "col_layout.cuh"
#include "fft.cuh"
#include "linalg.cuh"

namespace gw {
namespace col {

namespace cgr = cooperative_groups;

// Smoothing of the preconditioner's denominators (Ha), by scans of 0.02 .. 0.8
// over static, real, imaginary and complex frequencies on 16^3 .. 48^3 cells, wells
// and barriers, dense and sparse (mean of V -0.76 .. +0.14 Ha).  Of the levels of V
// tried there (mean, 1/2, 3/5, 2/3, 3/4, 9/10, largest) that of 2/3 is the best or
// within a tenth of it everywhere: higher ones cost barriers (3/4: 108 -> 145
// iterations), lower ones dense wells (1/2: 110 -> 125).
constexpr double kPreReal = 0.03, kPreImag = 0.2;
// SQMR stagnation: iterations without a halving of the quasi-residual norm tau.
// FP32: rounding errors scale with the largest residual of the pass (it peaks
// in the first steps), so tau goes no further than some 30 ulp of that, now and
// then 1.5 to 10 times the target; past it the recurrence comes apart, |r|
// grows to 1e2 .. 1e5 times tau and tau stays (kApartWait: within 10 of it).
constexpr int kQmrWindow = 1000;     // anywhere (as the multi-launch solver's)
constexpr int kQmrWindowFloor = 48;  // FP32, tau below 1e-4 |b| or 2e-6 max |r|
constexpr int kApartWait = 16;       // FP32, iterations in a row with |r| > 100 tau
constexpr int kNearWait = 32;        // iterations granted within a factor 2 of the target norm

template <typename T> struct alignas(16) V4 { T x, y, z, w; };

// Warp sums of M values per lane (M a power of 2, at most 32) by recursive
// halving: M - 1 + log2(32 / M) additions instead of 5 M.  Lane l returns the
// sum of value l / (32 / M), the same bits in all its lanes.
template <int M, typename A> __device__ __forceinline__ A warp_sums(A* v) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = M / 2; n >= 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const A keep = up ? v[n + k] : v[k], give = up ? v[k] : v[n + k];
      v[k] = acc_add(keep, acc_shfl(give, o));
    }
  }
#pragma unroll
  for (int q = 16 / M; q >= 1; q >>= 1) v[0] = acc_add(v[0], acc_shfl(v[0], q));
  return v[0];
}
__host__ __device__ constexpr int pow2_up(int n) { int p = 1; while (p < n) p *= 2; return p; }

// --- R-point transforms in registers: dft (fft.cuh)
// v[k] *= w_N^(S k m)  (stw holds exp(-2 pi i k / N); k m < N)
template <typename T, int S, int R> __device__ __forceinline__ void twid(cpx<T>* v, const cpx<T>* stw, int m) {
#pragma unroll
  for (int k = 1; k < R; ++k) {
    cpx<T> w = stw[k * m];
    if (S > 0) w.y = -w.y;
    v[k] = cmul(v[k], w);
  }
}
template <int R> struct IC { static constexpr int value = R; };

// Per-column state of the recurrences (every CTA keeps its own equal copy).
template <typename T> struct CgCol {
  T gam, gdiv, alpha, stop, rmin, rbest, al, bt;
  int it, itb, active, flag;
};
struct QmrCol {
  double2 rho, alpha, beta, qc;
  double dc, theta2, tau2, stop, qbest, rr0, rmax;         // theta^2, tau^2
  int it, itb, near, apart, active, flag, upd;
};

template <typename T, int KIND, int N1, int N2>
__global__ void __launch_bounds__(kTPB, 1) k_col_solve(ColArgs<T> a) {
  using V = cpx<T>;
  using W4 = V4<T>;
  using SA = ScalarAcc<T, KIND>;
  using CA = CoefAcc<T, KIND>;
  constexpr bool PAIR = KIND != COL_QMR;
  constexpr bool CG = KIND == COL_CG_PAIR;
  constexpr int NV = CG ? 4 : 2;
  constexpr int NC = PAIR ? 2 : 1;
  constexpr int N = N1 * N2, LD = N | 1;
  constexpr IC<N1> R1_{};
  constexpr IC<N2> R2_{};
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int s_pb[kColMaxQ + 1];
  __shared__ CgCol<T> s_cg[2];
  __shared__ QmrCol s_q[2];
  __shared__ int s_any;
  __shared__ int s_top[2], s_xtop[2];             // high words of the columns' largest components: b, x
  cgr::cluster_group cl = cgr::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int Q = 1 << a.sh.lq, rank = Q > 1 ? (int)cl.block_rank() : 0;
  const int unit = blockIdx.x >> a.sh.lq;
  const int c0 = PAIR ? 2 * unit : unit, nc = min(NC, a.ncol - c0);
  bool on[2] = {false, false};
  for (int c = 0; c < nc; ++c) on[c] = !a.outer_active || a.outer_active[c0 + c];
  if (!on[0] && !on[1]) {                         // the whole cluster leaves together
    if (rank == 0 && tid < nc) { a.iters[c0 + tid] = 0; a.flags[c0 + tid] = 0; }
    return;
  }
  const int P = a.P, nm = a.nm, ldz = a.ldz, ldr = 2 * a.npair;
  const int nproj = a.nproj, rgrp = row_group(nproj, sizeof(T) == 4), nsplit = splits(nproj, rgrp, a.nhl);
  const Lay L = layout<T>(KIND, a.sh, N, P, a.npair, ldz, a.nhl, nproj);
  V* Z = reinterpret_cast<V*>(sm + L.Z);          // [N][ldz] own pencils
  V* R = reinterpret_cast<V*>(sm + L.R);          // [nzl][ldr] own slabs, disc values
  V* Tt = reinterpret_cast<V*>(sm + L.T);         // [nsb][N][LD] slab tiles
  W4* Tm = reinterpret_cast<W4*>(sm + L.T);       // [nhl] A u, CG then u (share the tiles' place)
  T* Vs = reinterpret_cast<T*>(sm + L.V);         // [nzl][N][N] V / N_g of the own slabs (v_smem)
  T* Kt = reinterpret_cast<T*>(sm + L.K);         // preconditioner: one real value per column,
  V* KC = reinterpret_cast<V*>(sm + L.K);         // COL_QMR one complex value
  T* kin = reinterpret_cast<T*>(sm + L.kin);
  unsigned* hpos = reinterpret_cast<unsigned*>(sm + L.hpos);
  unsigned short* rt = reinterpret_cast<unsigned short*>(sm + L.rt);
  unsigned char* own = sm + L.own;
  signed char* zm = reinterpret_cast<signed char*>(sm + L.zm);
  unsigned char* zs = sm + L.zs;
  V* stw = reinterpret_cast<V*>(sm + L.tw);
  CA* cp = reinterpret_cast<CA*>(sm + L.cp);      // [nsplit][nproj][NV] this CTA's coefficients in parts
  CA* coefp = reinterpret_cast<CA*>(sm + L.coefp);   // [Q][nproj][NV]
  T* coef = reinterpret_cast<T*>(sm + L.coef);    // [nproj][NV]
  SA* part = reinterpret_cast<SA*>(sm + L.part);  // [kNW][4] scalar sums of the warps
  SA* sc = reinterpret_cast<SA*>(sm + L.sc);      // [3][Q][4] of the CTAs

  auto at = [&](auto* p, int q) { return Q > 1 ? cl.map_shared_rank(p, q) : p; };
  auto csync = [&]() { if (Q > 1) cl.sync(); else __syncthreads(); };

  // ---- tables
  if (tid <= Q) s_pb[tid] = a.split[a.sh.lq * (kColMaxQ + 1) + tid];
  if (tid < 2) s_top[tid] = s_xtop[tid] = 0;
  __syncthreads();
  const int p0 = s_pb[rank], npl = s_pb[rank + 1] - p0, nrl = 2 * npl;
  const int h0 = a.hstart[p0], nh = a.hstart[p0 + npl] - h0;
  const int nzl = (N + Q - 1) >> a.sh.lq, z0 = rank * nzl, nsl = max(0, min(nzl, N - z0));
  FastDiv dnr;
  dnr.set((unsigned)max(nrl, 1));
  auto owner = [&](int j) { int o = 0; while (o + 1 < Q && j >= s_pb[o + 1]) ++o; return o; };
  for (int k = tid; k < N; k += kTPB) {
    stw[k] = a.tw[k];
    zs[k] = (unsigned char)((k % N1) * N2 + k / N1);
  }
  for (int k = tid; k < 2 * a.npair; k += kTPB) {
    const int j = k >> 1, m = k & 1, o = owner(j);
    own[2 * s_pb[o] + (m ? s_pb[o + 1] - s_pb[o] : 0) + (j - s_pb[o])] = (unsigned char)o;
  }
  for (int k = tid; k < N * P; k += kTPB) {
    const unsigned d = a.disc[k];
    unsigned v = 0xffffu;
    if (d != 0xffffu) {
      const int j = d >> 1, o = owner(j);
      v = (unsigned)(2 * s_pb[o] + ((d & 1) ? s_pb[o + 1] - s_pb[o] : 0) + (j - s_pb[o]));
    }
    rt[k] = (unsigned short)v;
  }
  for (int k = tid; k < nrl; k += kTPB) {
    const int j = p0 + (k < npl ? k : k - npl);
    zm[k] = (signed char)((j == 0 && k >= npl) ? -1 : (int)a.zmax[j]);
  }
  bool pre[2] = {false, false};
  T Ex[2] = {(T)0, (T)0}, Ep[2] = {(T)0, (T)0}, Ey = (T)0;   // Ep: of the preconditioner
  for (int c = 0; c < nc; ++c) {
    pre[c] = a.tk && a.tk[c0 + c] != 0.0;
    Ex[c] = (T)a.E[c0 + c].x;
    Ep[c] = (T)(a.E[c0 + c].x - a.v0);
    if (!PAIR) Ey = (T)a.E[c0].y;
  }
  auto precond_real = [](T d) { return (T)1 / sqrt(d * d + (T)(kPreReal * kPreReal)); };
  // solver vectors: CG r, p, s, x; SQMR r, q, d, x
  const size_t xs = a.sh.vec_smem ? (size_t)a.nhl : (size_t)a.nh;
  W4* X = a.sh.vec_smem ? reinterpret_cast<W4*>(sm + L.X)
                        : reinterpret_cast<W4*>(a.vecs + (size_t)unit * a.sh.vec_elems) + h0;
  const V* C = a.Ch + h0;
  size_t ldc = (size_t)a.nh;
  if (a.sh.c_smem) {
    V* Cs = reinterpret_cast<V*>(sm + L.C);
    for (int v = warp; v < nproj; v += kNW)
      for (int e = lane; e < nh; e += 32) Cs[(size_t)v * a.nhl + e] = C[(size_t)v * ldc + e];
    C = Cs;
    ldc = (size_t)a.nhl;
  }
  if (a.sh.v_smem) {
    const T* v = a.Vp + (size_t)z0 * N * N;
    for (int k = tid; k < nsl * N * N; k += kTPB) Vs[k] = v[k];
  }
  // FP32 passes and pairs run on the right-hand side times the power of two that
  // brings its largest component to 1 .. 2 (exact; nothing else depends on the
  // size of b).  Unscaled, products of FP32 entries leave the range below 1e-22
  // and their rounding errors below 3e-16, where a refinement's later passes
  // arrive; and the rounding errors of one column of a pair land in the other.
  constexpr bool SCALED = sizeof(T) == 4 || PAIR;
  auto hi = [](double x) { return __double2hiint(x) & 0x7fffffff; };
  int ex[2] = {0, 0};
  if constexpr (SCALED) {
    int top[2] = {0, 0};
    for (int e = tid; e < nh; e += kTPB) {
      const int g = a.gp[h0 + e], m = a.gm[h0 + e];
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (on[c]) {
          const double2 u = a.b64[(size_t)(c0 + c) * a.npw + g], w = a.b64[(size_t)(c0 + c) * a.npw + m];
          top[c] = max(max(top[c], max(hi(u.x), hi(u.y))), max(hi(w.x), hi(w.y)));
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      top[c] = __reduce_max_sync(0xffffffffu, top[c]);
      if (lane == 0) atomicMax(&s_top[c], top[c]);
    }
    csync();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      int t = 0;
      for (int q = 0; q < Q; ++q) t = max(t, *at(&s_top[c], q));
      ex[c] = pow2_exp(__hiloint2double(t, 0));
    }
  }
  // 2^-ex of column c, and back
  auto scale_in = [&](int c) { return SCALED ? pow2_in(c ? ex[1] : ex[0]) : 1.0; };
  auto scale_out = [&](int c) { return SCALED ? pow2_out(c ? ex[1] : ex[0]) : 1.0; };
  auto stop_abs = [&](int c) { return a.rr_abs ? a.rr_abs[c0 + c] * scale_in(c) * scale_in(c) : 0.0; };
  for (int e = tid; e < nh; e += kTPB) {
    const int h = h0 + e;
    const T k = a.kin[h];
    kin[e] = k;
    hpos[e] = a.hpos[h];
    if (PAIR) {
      Kt[2 * e] = pre[0] ? precond_real(k - Ep[0]) : (T)1;
      Kt[2 * e + 1] = pre[1] ? precond_real(k - Ep[1]) : (T)1;
    } else {
      const T dr = k - Ep[0], di = Ey > (T)0 ? Ey + (T)kPreImag : Ey - (T)kPreImag;
      V kc = mk<T>((T)1, (T)0);
      if (pre[0]) {
        if (Ey == (T)0) kc.x = precond_real(dr);
        else { const T d = (T)1 / (dr * dr + di * di); kc = mk<T>(dr * d, di * d); }
      }
      KC[e] = kc;
    }
    const int g = a.gp[h], m = a.gm[h];
    W4 r = {(T)0, (T)0, (T)0, (T)0};
    if (PAIR) {
      double2 b[2] = {make_double2(0, 0), make_double2(0, 0)};
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (on[c]) {
          const double2 u = a.b64[(size_t)(c0 + c) * a.npw + g], w = a.b64[(size_t)(c0 + c) * a.npw + m];
          b[c] = make_double2(0.5 * scale_in(c) * (u.x + w.x), 0.5 * scale_in(c) * (u.y - w.y));
        }
      r = {(T)b[0].x, (T)b[0].y, (T)b[1].x, (T)b[1].y};
    } else {
      const double2 u = a.b64[(size_t)c0 * a.npw + g], w = a.b64[(size_t)c0 * a.npw + m];
      const double f = scale_in(0);
      r = {(T)(f * u.x), (T)(f * u.y), (T)(f * w.x), (T)(f * w.y)};
      if (h == 0) r.z = r.w = (T)0;
    }
    const W4 zero = {(T)0, (T)0, (T)0, (T)0};
    X[e] = r;
    X[xs + e] = zero;
    X[2 * xs + e] = zero;
    X[3 * xs + e] = zero;
  }
  if (tid < 2) {
    s_cg[tid] = CgCol<T>{};
    s_q[tid] = QmrCol{};
  }
  csync();                                        // every CTA of the cluster has started

  const T one = (T)1, two = (T)2;
  auto of = [](T x) { return AccFrom<SA>::of(x); };
  // |n| <= m for index k of N (one comparison; m = -1: none)
  auto inside = [&](int k, int m) { return (unsigned)(k - m - 1) >= (unsigned)(N - 2 * m - 1); };
  auto present = [&](int x) { return inside(x, nm); };
  auto mirror_row = [&](int j) { return j == 0 ? 0 : npl + (j - p0); };   // local row of a pair's second pencil

  // u (both halves of the pair, or the complex column) into the own pencils
  auto scatter = [&](int e, const W4& u) {
    const unsigned hp = hpos[e];
    const int j = (int)(hp >> 8), z = (int)(hp & 255u);
    V g, m;
    if (PAIR) {
      g = mk<T>(u.x - u.w, u.y + u.z);
      m = mk<T>(u.x + u.w, u.z - u.y);
    } else {
      g = mk<T>(u.x, u.y);
      m = mk<T>(u.z, u.w);
    }
    Z[z * ldz + (j - p0)] = g;
    if (h0 + e != 0) Z[(N - z) % N * ldz + mirror_row(j)] = m;
  };

  // z-IFFT of the own pencils, sent to the slab owners
  auto z_step1 = [&]() {
    ([&](auto RR) {
      constexpr int R1 = decltype(RR)::value;
      for (int t = tid; t < nrl * N2; t += kTPB) {
        const int n2 = dnr.div(t), row = t - n2 * nrl;
        const int zmx = zm[row];
        V v[R1];
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) {
          const int z = n1 * N2 + n2;
          v[n1] = inside(z, zmx) ? Z[z * ldz + row] : mk<T>(0, 0);
        }
        dft<T, 1, R1>(v);
        twid<T, 1, R1>(v, stw, n2);
#pragma unroll
        for (int k = 0; k < R1; ++k) Z[(k * N2 + n2) * ldz + row] = v[k];
      }
    })(R1_);
  };
  auto z_inverse_send = [&]() {
    z_step1();
    __syncthreads();
    ([&](auto RR) {
      constexpr int R2 = decltype(RR)::value;
      for (int t = tid; t < nrl * N1; t += kTPB) {
        const int k1 = dnr.div(t), row = t - k1 * nrl;
        V v[R2];
#pragma unroll
        for (int k = 0; k < R2; ++k) v[k] = Z[(k1 * R2 + k) * ldz + row];
        dft<T, 1, R2>(v);
#pragma unroll
        for (int k = 0; k < R2; ++k) {
          const int z = k1 + N1 * k;
          const int o = a.dnz.div(z);
          at(R, o)[(z - o * nzl) * ldr + 2 * p0 + row] = v[k];
        }
      }
    })(R2_);
  };
  // Q = 1: the same, left in the pencils (i2 at slot zs[i2])
  auto z_inverse_local = [&]() {
    z_step1();
    __syncthreads();
    ([&](auto RR) {
      constexpr int R2 = decltype(RR)::value;
      for (int t = tid; t < nrl * N1; t += kTPB) {
        const int k1 = dnr.div(t), row = t - k1 * nrl;
        V v[R2];
#pragma unroll
        for (int k = 0; k < R2; ++k) v[k] = Z[(k1 * R2 + k) * ldz + row];
        dft<T, 1, R2>(v);
#pragma unroll
        for (int k = 0; k < R2; ++k) Z[(k1 * R2 + k) * ldz + row] = v[k];
      }
    })(R2_);
  };

  auto z_inverse = [&]() { if (Q > 1) z_inverse_send(); else z_inverse_local(); };

  // the slabs: returns true when the unit has stopped (CG: decided while the
  // first step runs)
  auto slabs = [&](bool check) {
    const int absent = N - P;                     // planes without entries: nm < i0 < N - nm
    for (int sb = 0; sb < max(nsl, 1); sb += a.sh.nsb) {
      const int ns = min(a.sh.nsb, nsl - sb);
      ([&](auto RR) {
        constexpr int R1 = decltype(RR)::value;
        for (int t = tid; t < ns * N2 * P; t += kTPB) {
          const int q = a.dP.div(t), p = t - q * P, s = (int)((unsigned)q / N2), n2 = q - s * N2;
          const V* src = Q > 1 ? R + (size_t)(sb + s) * ldr : Z + zs[sb + s] * ldz;
          V v[R1];
#pragma unroll
          for (int n1 = 0; n1 < R1; ++n1) {
            const unsigned row = rt[(n1 * N2 + n2) * P + p];
            v[n1] = row != 0xffffu ? src[row] : mk<T>(0, 0);
          }
          dft<T, 1, R1>(v);
          twid<T, 1, R1>(v, stw, n2);
          V* d = Tt + (s * N + (p <= nm ? p : p + absent)) * LD + n2;
#pragma unroll
          for (int k = 0; k < R1; ++k) d[k * N2] = v[k];
        }
      })(R1_);
      __syncthreads();
      if (check && sb == 0 && !s_any) return true;
      ([&](auto RR) {
        constexpr int R2 = decltype(RR)::value;
        for (int t = tid; t < ns * N1 * P; t += kTPB) {
          const int q = a.dP.div(t), p = t - q * P, s = (int)((unsigned)q / N1), k1 = q - s * N1;
          V* d = Tt + (s * N + (p <= nm ? p : p + absent)) * LD + k1 * R2;
          V v[R2];
#pragma unroll
          for (int k = 0; k < R2; ++k) v[k] = d[k];
          dft<T, 1, R2>(v);
#pragma unroll
          for (int k = 0; k < R2; ++k) d[k] = v[k];
        }
      })(R2_);
      __syncthreads();
      ([&](auto RR) {
        constexpr int R1 = decltype(RR)::value;
        for (int t = tid; t < ns * N2 * N; t += kTPB) {
          const int q = (int)((unsigned)t / N), y = t - q * N, s = (int)((unsigned)q / N2), n2 = q - s * N2;
          V* d = Tt + (s * N + n2) * LD + y;
          V v[R1];
#pragma unroll
          for (int n1 = 0; n1 < R1; ++n1) {
            const int x = n1 * N2 + n2;
            v[n1] = present(x) ? d[n1 * N2 * LD] : mk<T>(0, 0);
          }
          dft<T, 1, R1>(v);
          twid<T, 1, R1>(v, stw, n2);
#pragma unroll
          for (int k = 0; k < R1; ++k) d[k * N2 * LD] = v[k];
        }
      })(R1_);
      ([&](auto RR) {
        constexpr int R2 = decltype(RR)::value;
        // FP32: the potential of a thread's next task is loaded ahead, of the
        // first before the barrier, of the others before the second transform
        // of the last (in FP64 the registers would spill, and the FP64 pipe,
        // not latency, is the bound)
        constexpr bool ahead = sizeof(T) == 4;
        const int tasks = ns * N1 * N;
        T pot[R2];
        auto load = [&](int t) {
          if (t >= tasks) return;
          const int q = (int)((unsigned)t / N), y = t - q * N, s = (int)((unsigned)q / N1), k1 = q - s * N1;
          if (a.sh.v_smem) {
            const T* vp = Vs + ((sb + s) * N + k1) * N + y;
#pragma unroll
            for (int k = 0; k < R2; ++k) pot[k] = vp[k * N1 * N];
          } else {
            const T* vp = a.Vp + ((size_t)(z0 + sb + s) * N + k1) * N + y;
#pragma unroll
            for (int k = 0; k < R2; ++k) pot[k] = __ldg(vp + k * N1 * N);
          }
        };
        if (ahead) load(tid);
        __syncthreads();
        for (int t = tid; t < tasks; t += kTPB) {
          const int q = (int)((unsigned)t / N), y = t - q * N, s = (int)((unsigned)q / N1), k1 = q - s * N1;
          V* d = Tt + (s * N + k1 * R2) * LD + y;
          V v[R2];
#pragma unroll
          for (int k = 0; k < R2; ++k) v[k] = d[k * LD];
          dft<T, 1, R2>(v);
          if (!ahead) load(t);
#pragma unroll
          for (int k = 0; k < R2; ++k) v[k] = mk<T>(v[k].x * pot[k], v[k].y * pot[k]);
          if (ahead) load(t + kTPB);
          dft<T, -1, R2>(v);
          twid<T, -1, R2>(v, stw, k1);
#pragma unroll
          for (int k = 0; k < R2; ++k) d[k * LD] = v[k];
        }
      })(R2_);
      __syncthreads();
      ([&](auto RR) {
        constexpr int R1 = decltype(RR)::value;
        for (int t = tid; t < ns * N2 * N; t += kTPB) {
          const int q = (int)((unsigned)t / N), y = t - q * N, s = (int)((unsigned)q / N2), n2 = q - s * N2;
          V* d = Tt + (s * N + n2) * LD + y;
          V v[R1];
#pragma unroll
          for (int k = 0; k < R1; ++k) v[k] = d[k * N2 * LD];
          dft<T, -1, R1>(v);
#pragma unroll
          for (int n1 = 0; n1 < R1; ++n1) {
            const int x = n1 * N2 + n2;
            if (present(x)) d[n1 * N2 * LD] = v[n1];
          }
        }
      })(R1_);
      __syncthreads();
      ([&](auto RR) {
        constexpr int R2 = decltype(RR)::value;
        for (int t = tid; t < ns * N1 * P; t += kTPB) {
          const int q = a.dP.div(t), p = t - q * P, s = (int)((unsigned)q / N1), k1 = q - s * N1;
          V* d = Tt + (s * N + (p <= nm ? p : p + absent)) * LD + k1 * R2;
          V v[R2];
#pragma unroll
          for (int k = 0; k < R2; ++k) v[k] = d[k];
          dft<T, -1, R2>(v);
          twid<T, -1, R2>(v, stw, k1);
#pragma unroll
          for (int k = 0; k < R2; ++k) d[k] = v[k];
        }
      })(R2_);
      __syncthreads();
      ([&](auto RR) {
        constexpr int R1 = decltype(RR)::value;
        for (int t = tid; t < ns * N2 * P; t += kTPB) {
          const int q = a.dP.div(t), p = t - q * P, s = (int)((unsigned)q / N2), n2 = q - s * N2;
          const V* d = Tt + (s * N + (p <= nm ? p : p + absent)) * LD + n2;
          V v[R1];
#pragma unroll
          for (int k = 0; k < R1; ++k) v[k] = d[k * N2];
          dft<T, -1, R1>(v);
          const int z = zs[z0 + sb + s];
#pragma unroll
          for (int n1 = 0; n1 < R1; ++n1) {
            const unsigned row = rt[(n1 * N2 + n2) * P + p];
            if (row != 0xffffu) {
              const int o = own[row];
              at(Z, o)[z * ldz + ((int)row - 2 * s_pb[o])] = v[n1];
            }
          }
        }
      })(R1_);
      __syncthreads();
    }
    return false;
  };

  // z-FFT of the own pencils, from slot order to natural order, in place
  auto z_forward = [&]() {
    ([&](auto RR) {
      constexpr int R2 = decltype(RR)::value;
      for (int t = tid; t < nrl * N1; t += kTPB) {
        const int k1 = dnr.div(t), row = t - k1 * nrl;
        V v[R2];
#pragma unroll
        for (int k = 0; k < R2; ++k) v[k] = Z[(k1 * R2 + k) * ldz + row];
        dft<T, -1, R2>(v);
        twid<T, -1, R2>(v, stw, k1);
#pragma unroll
        for (int k = 0; k < R2; ++k) Z[(k1 * R2 + k) * ldz + row] = v[k];
      }
    })(R2_);
    __syncthreads();
    ([&](auto RR) {
      constexpr int R1 = decltype(RR)::value;
      for (int t = tid; t < nrl * N2; t += kTPB) {
        const int n2 = dnr.div(t), row = t - n2 * nrl;
        const int zmx = zm[row];
        V v[R1];
#pragma unroll
        for (int k = 0; k < R1; ++k) v[k] = Z[(k * N2 + n2) * ldz + row];
        dft<T, -1, R1>(v);
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) {
          const int z = n1 * N2 + n2;
          if (inside(z, zmx)) Z[z * ldz + row] = v[n1];
        }
      }
    })(R1_);
    __syncthreads();
  };

  // (V u) + (kin - E) u at one half entry
  auto gather = [&](int e, const W4& u) {
    const unsigned hp = hpos[e];
    const int j = (int)(hp >> 8), z = (int)(hp & 255u);
    const V y1 = Z[z * ldz + (j - p0)], y2 = Z[(N - z) % N * ldz + mirror_row(j)];
    const T k = kin[e];
    W4 t;
    if (PAIR) {
      t.x = (T)0.5 * (y1.x + y2.x) + (k - Ex[0]) * u.x;
      t.y = (T)0.5 * (y1.y - y2.y) + (k - Ex[0]) * u.y;
      t.z = (T)0.5 * (y1.y + y2.y) + (k - Ex[1]) * u.z;
      t.w = (T)0.5 * (y2.x - y1.x) + (k - Ex[1]) * u.w;
    } else {
      const T dr = k - Ex[0], di = -Ey;
      t.x = y1.x + dr * u.x - di * u.y;
      t.y = y1.y + dr * u.y + di * u.x;
      t.z = y2.x + dr * u.z - di * u.w;
      t.w = y2.y + dr * u.w + di * u.z;
      if (h0 + e == 0) t.z = t.w = (T)0;
    }
    return t;
  };
  // Projector coefficients of Tm (and, CG, of u): a warp takes RG rows and one
  // of the nsplit parts of the own entries.  PAIR: sum_h f Re conj(c) y with
  // f = 2, 1 at G = 0 (summed with 1 and 1/2, doubled at the end); complex:
  // sum_h conj(c) y(G) + c y(-G) = Re c (y + y') + i Im c (y' - y).
  auto dots_rows = [&](auto RR) {
    constexpr int RG = decltype(RR)::value;
    constexpr int M = pow2_up(RG * NV);
    const int ngr = (nproj + RG - 1) / RG;
    for (int w = warp; w < ngr * nsplit; w += kNW) {
      const int gr = w / nsplit, prt = w - gr * nsplit, v0 = gr * RG;
      unsigned row[RG];
#pragma unroll
      for (int q = 0; q < RG; ++q) row[q] = (unsigned)min(v0 + q, nproj - 1) * (unsigned)ldc;
      T acc[M];
      CA sum[M];
#pragma unroll
      for (int k = 0; k < M; ++k) {
        acc[k] = (T)0;
        sum[k] = AccFrom<CA>::of((T)0);
      }
      auto entry = [&](int e) {
        V c[RG];
#pragma unroll
        for (int q = 0; q < RG; ++q) c[q] = C[row[q] + (unsigned)e];
        W4 y = Tm[e];
        if (PAIR) {
          if (h0 + e == 0) { y.x *= (T)0.5; y.z *= (T)0.5; }
        } else {
          y = W4{y.x + y.z, y.y - y.w, y.y + y.w, y.z - y.x};
        }
#pragma unroll
        for (int q = 0; q < RG; ++q) {
          acc[q * NV] = fma(c[q].y, y.y, fma(c[q].x, y.x, acc[q * NV]));
          acc[q * NV + 1] = fma(c[q].y, y.w, fma(c[q].x, y.z, acc[q * NV + 1]));
        }
        if (CG) {
          W4 u = Tm[a.nhl + e];
          if (h0 + e == 0) { u.x *= (T)0.5; u.z *= (T)0.5; }
#pragma unroll
          for (int q = 0; q < RG; ++q) {
            acc[q * NV + NV - 2] = fma(c[q].y, u.y, fma(c[q].x, u.x, acc[q * NV + NV - 2]));
            acc[q * NV + NV - 1] = fma(c[q].y, u.w, fma(c[q].x, u.z, acc[q * NV + NV - 1]));
          }
        }
      };
      if constexpr (std::is_same<CA, T>::value) {
#pragma unroll 2
        for (int e = lane + 32 * prt; e < nh; e += 32 * nsplit) entry(e);
#pragma unroll
        for (int k = 0; k < M; ++k) sum[k] = acc[k];
      } else {
        // 8 entries (16 products) in plain FP32
        auto take = [&]() {
#pragma unroll
          for (int k = 0; k < RG * NV; ++k) {
            acc_in(sum[k], acc[k]);
            acc[k] = (T)0;
          }
        };
        const int st = 32 * nsplit;
        int e = lane + 32 * prt;
        for (; e + 7 * st < nh; e += 8 * st) {
#pragma unroll 2
          for (int k = 0; k < 8; ++k) entry(e + k * st);
          take();
        }
#pragma unroll 2
        for (; e < nh; e += st) entry(e);
        take();
      }
      CA t = warp_sums<M, CA>(sum);
      if (PAIR) t = acc_add(t, t);
      const int k = lane / (32 / M), q = k / NV;
      if (lane % (32 / M) == 0 && q < RG && v0 + q < nproj)
        cp[((size_t)prt * nproj + v0 + q) * NV + (k - q * NV)] = t;
    }
  };
  auto dots = [&]() {
    switch (rgrp) {
      case 1: dots_rows(IC<1>()); break;
      case 2: dots_rows(IC<2>()); break;
      case 5: if constexpr (sizeof(T) == 4) dots_rows(IC<5>()); break;
      case 6: if constexpr (sizeof(T) == 4) dots_rows(IC<6>()); break;
      default: dots_rows(IC<4>());
    }
  };
  // the parts added, to every CTA
  auto send_coef = [&]() {
    const int n = nproj * NV;
    for (int t = tid; t < (n << a.sh.lq); t += kTPB) {
      const int q = t / n, j = t - q * n;
      CA v = cp[j];
      for (int p = 1; p < nsplit; ++p) v = acc_add(v, cp[p * n + j]);
      at(coefp, q)[rank * n + j] = v;
    }
  };
  auto coef_of = [&](int j) {
    CA v = coefp[j];
    for (int q = 1; q < Q; ++q) v = acc_add(v, coefp[q * nproj * NV + j]);
    return acc_val(v);
  };
  auto coef_sum = [&]() {
    for (int j = tid; j < nproj * NV; j += kTPB) coef[j] = coef_of(j);
  };
  // Up to four scalar sums.  put: this thread's values into the warp's part;
  // after a barrier one warp adds the parts and sends them to every CTA (slot);
  // after the cluster barrier take gives value (lane & 3) in every lane.
  auto put_sums = [&](auto NN, SA* v) {
    constexpr int NS = decltype(NN)::value;
    const SA t = warp_sums<NS, SA>(v);
    if (lane % (32 / NS) == 0) part[warp * 4 + lane / (32 / NS)] = t;
  };
  auto send_sums = [&](int ns, int slot) {        // one warp
    const int k = lane & 3;
    SA t = of((T)0);
    if (k < ns)
      for (int w = lane >> 2; w < kNW; w += 8) t = acc_add(t, part[w * 4 + k]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) t = acc_add(t, acc_shfl(t, o));
    if (k < ns)
      for (int q = lane >> 2; q < Q; q += 8) at(sc, q)[((slot << a.sh.lq) + rank) * 4 + k] = t;
  };
  auto take_sums = [&](int slot) {                // one warp
    SA t = of((T)0);
    for (int q = lane >> 2; q < Q; q += 8) t = acc_add(t, sc[((slot << a.sh.lq) + q) * 4 + (lane & 3)]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) t = acc_add(t, acc_shfl(t, o));
    return t;
  };
  // y - sum_v C_v coef_v at one half entry
  auto project = [&](int e, W4 y) {
    T a1 = (T)0, a2 = (T)0, a3 = (T)0, a4 = (T)0;
    constexpr int U = sizeof(T) == 4 ? 16 : 8;    // rows in flight
    int v = 0;
    for (; v + U <= nproj; v += U) {
      V c[U];
#pragma unroll
      for (int q = 0; q < U; ++q) c[q] = C[(unsigned)(v + q) * (unsigned)ldc + (unsigned)e];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        const T k0 = coef[(v + q) * NV], k1 = coef[(v + q) * NV + 1];
        a1 += c[q].x * k0;
        a4 += c[q].y * k0;
        a3 += c[q].x * k1;
        a2 += c[q].y * k1;
      }
    }
    for (; v < nproj; ++v) {
      const V c = C[(size_t)v * ldc + e];
      const T k0 = coef[v * NV], k1 = coef[v * NV + 1];
      a1 += c.x * k0;
      a4 += c.y * k0;
      a3 += c.x * k1;
      a2 += c.y * k1;
    }
    if (PAIR) {
      y.x -= a1; y.y -= a4; y.z -= a3; y.w -= a2;
    } else {
      y.x -= a1 - a2; y.y -= a3 + a4;
      if (h0 + e != 0) { y.z -= a1 + a2; y.w -= a3 - a4; }
    }
    return y;
  };

  if constexpr (CG) {
    // Chronopoulos and Gear's one-reduction form (see kernels_cg.cu): u = K r,
    // w = P_c (H - E) u, gamma = r^H u, delta = u^H w.  The four real
    // components of a half entry (Re, Im of both columns) are independent but
    // for the packing: one thread each while that fills no more than the CTA
    // (latency counts: 16^3 FP64, update 9.6k -> 4.0k cycles), else one thread
    // per entry (a quarter of the loads: 48^3 FP32, 7.4k -> 3.2k cycles).
    T* XT = reinterpret_cast<T*>(X);
    T* TT = reinterpret_cast<T*>(Tm);
    T* ZT = reinterpret_cast<T*>(Z);
    const T* CT = reinterpret_cast<const T*>(C);
    const bool quads = 4 * a.nhl <= kTPB;
    // r after k updates: u into the pencils, gamma and |r|^2
    auto update1 = [&](int k, SA* v4) {
      T g0 = (T)0, r0 = (T)0, g1 = (T)0, r1 = (T)0;
      const T al0 = s_cg[0].al, al1 = s_cg[1].al, bt0 = s_cg[0].bt, bt1 = s_cg[1].bt;
      const bool a0 = k == 0 || s_cg[0].active, a1 = k == 0 || s_cg[1].active;
      for (int e = tid; e < nh; e += kTPB) {
        const T k0 = Kt[2 * e], k1 = Kt[2 * e + 1];
        W4 r = X[e];
        if (k > 0) {
          W4 p = X[xs + e], sv = X[2 * xs + e], x = X[3 * xs + e];
          const W4 w = project(e, Tm[e]);
          if (a0) {
            p.x = k0 * r.x + bt0 * p.x; p.y = k0 * r.y + bt0 * p.y;
            sv.x = w.x + bt0 * sv.x;    sv.y = w.y + bt0 * sv.y;
            x.x += al0 * p.x;           x.y += al0 * p.y;
            r.x -= al0 * sv.x;          r.y -= al0 * sv.y;
          }
          if (a1) {
            p.z = k1 * r.z + bt1 * p.z; p.w = k1 * r.w + bt1 * p.w;
            sv.z = w.z + bt1 * sv.z;    sv.w = w.w + bt1 * sv.w;
            x.z += al1 * p.z;           x.w += al1 * p.w;
            r.z -= al1 * sv.z;          r.w -= al1 * sv.w;
          }
          X[e] = r;
          X[xs + e] = p;
          X[2 * xs + e] = sv;
          X[3 * xs + e] = x;
        }
        const T f = (h0 + e == 0) ? one : two;
        const T n0 = f * (r.x * r.x + r.y * r.y), n1 = f * (r.z * r.z + r.w * r.w);
        r0 += n0;
        g0 += k0 * n0;
        r1 += n1;
        g1 += k1 * n1;
        W4 u = {(T)0, (T)0, (T)0, (T)0};
        if (a0) { u.x = k0 * r.x; u.y = k0 * r.y; }
        if (a1) { u.z = k1 * r.z; u.w = k1 * r.w; }
        scatter(e, u);
      }
      v4[0] = of(g0); v4[1] = of(r0); v4[2] = of(g1); v4[3] = of(r1);
    };
    const int cmp = tid & 3, cc = cmp >> 1;       // component x, y (column 0), z, w (column 1)
    const int im = (cmp == 1 || cmp == 2) ? 1 : 0;
    auto update4 = [&](int k, SA* v4) {
      T gs = (T)0, rs = (T)0, u = (T)0;
      const int t = tid, e = t >> 2;              // 4 nh <= kTPB: one round
      if (e < nh) {
        const T kc = Kt[2 * e + cc];
        T r = XT[t];
        const bool act = k == 0 || s_cg[cc].active;
        if (k > 0 && act) {
          const T al = s_cg[cc].al, bt = s_cg[cc].bt;
          T w = TT[t], p = XT[4 * xs + t], sv = XT[8 * xs + t], x = XT[12 * xs + t];
          const T* c = CT + 2 * e + (cmp & 1);
          const T* kf = coef + cc;
          T acc = (T)0;
          int v = 0;
          for (; v + 8 <= nproj; v += 8) {
            T cv[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) cv[q] = c[2 * (size_t)(v + q) * ldc];
#pragma unroll
            for (int q = 0; q < 8; ++q) acc += cv[q] * kf[(v + q) * NV];
          }
          for (; v < nproj; ++v) acc += c[2 * (size_t)v * ldc] * kf[v * NV];
          w -= acc;
          p = kc * r + bt * p;
          sv = w + bt * sv;
          x += al * p;
          r -= al * sv;
          XT[t] = r;
          XT[4 * xs + t] = p;
          XT[8 * xs + t] = sv;
          XT[12 * xs + t] = x;
        }
        rs = (h0 + e == 0) ? r * r : two * r * r;
        gs = kc * rs;
        if (act) u = kc * r;
      }
      // pair packing: x - w, y + z at G; x + w, z - y at -G
      const T o = acc_shfl(u, 3);
      if (e < nh) {
        const unsigned hp = hpos[e];
        const int j = (int)(hp >> 8), z = (int)(hp & 255u);
        if (cmp < 2) ZT[2 * (z * ldz + (j - p0)) + im] = cmp ? u + o : u - o;
        else if (h0 + e != 0) ZT[2 * ((N - z) % N * ldz + mirror_row(j)) + im] = cmp == 2 ? u - o : u + o;
      }
      v4[0] = of(cc ? (T)0 : gs); v4[1] = of(cc ? (T)0 : rs);
      v4[2] = of(cc ? gs : (T)0); v4[3] = of(cc ? rs : (T)0);
    };
    // w and u, and u^H w before the projector
    auto gather1 = [&](SA* v2) {
      T d0 = (T)0, d1 = (T)0;
      for (int e = tid; e < nh; e += kTPB) {
        const T k0 = Kt[2 * e], k1 = Kt[2 * e + 1];
        const W4 r = X[e];
        const W4 u = {k0 * r.x, k0 * r.y, k1 * r.z, k1 * r.w};
        const W4 w = gather(e, u);
        Tm[e] = w;
        Tm[a.nhl + e] = u;
        const T f = (h0 + e == 0) ? one : two;
        d0 += f * (u.x * w.x + u.y * w.y);
        d1 += f * (u.z * w.z + u.w * w.w);
      }
      v2[0] = of(d0);
      v2[1] = of(d1);
    };
    auto gather4 = [&](SA* v2) {
      T ds = (T)0;
      const int t = tid, e = t >> 2;
      if (e < nh) {
        const unsigned hp = hpos[e];
        const int j = (int)(hp >> 8), z = (int)(hp & 255u);
        const T y1 = ZT[2 * (z * ldz + (j - p0)) + im], y2 = ZT[2 * ((N - z) % N * ldz + mirror_row(j)) + im];
        const T u = Kt[2 * e + cc] * XT[t];
        const T fv = (T)0.5 * (cmp == 1 ? y1 - y2 : cmp == 3 ? y2 - y1 : y1 + y2);
        const T w = fv + (kin[e] - Ex[cc]) * u;
        TT[t] = w;
        TT[4 * a.nhl + t] = u;
        ds = ((h0 + e == 0) ? one : two) * u * w;
      }
      v2[0] = of(cc ? (T)0 : ds);
      v2[1] = of(cc ? ds : (T)0);
    };
    const bool decide = warp == kNW - 1;
    for (int k = 0;; ++k) {
      {
        SA v4[4];
        if (quads) update4(k, v4);
        else update1(k, v4);
        put_sums(IC<4>(), v4);
      }
      __syncthreads();
      if (decide) send_sums(4, 0);
      z_inverse();
      csync();
      // while the slabs' first step runs: gamma, |r|^2 and the stopping tests
      if (decide) {
        const SA tot = take_sums(0);
        const SA g = acc_lane(tot, (2 * lane) & 3), q = acc_lane(tot, (2 * lane + 1) & 3);
        int act = 0;
        if (lane < 2) {
          CgCol<T>& st = s_cg[lane];
          const T gam = acc_val(g), rr = acc_val(q);
          if (k == 0) {
            const T s1 = (T)a.tol2 * rr, s2 = lane < nc ? (T)stop_abs(lane) : (T)0;
            st.stop = s1 > s2 ? s1 : s2;
            st.rmin = rr;
            st.rbest = rr;
            st.active = (lane < nc && on[lane] && rr > (T)0) ? 1 : 0;
          }
          if (st.active) {
            st.rmin = rr < st.rmin ? rr : st.rmin;
            if (rr < (T)0.25 * st.rbest) { st.rbest = rr; st.itb = k; }
            int stop = 0;
            if (!isfinite(rr)) { st.flag = 2; stop = 1; }
            else if (rr <= st.stop) { st.flag = 0; stop = 1; }
            else if (rr > (T)1e4 * st.rmin) { st.flag = 3; stop = 1; }
            else if (k >= a.maxit) { st.flag = 1; stop = 1; }
            else if (k - st.itb > max(kCgStagWindow, 2 * st.itb)) { st.flag = 4; stop = 1; }
            st.it = k;
            // beta, and gamma / alpha_prev for the denominator of alpha
            st.bt = k > 0 ? gam / st.gam : (T)0;
            st.gdiv = k > 0 ? gam / st.alpha : (T)0;
            st.gam = gam;
            if (stop) st.active = 0;
          }
          act = st.active;
        }
        const unsigned any = __ballot_sync(0xffffffffu, act != 0);
        if (lane == 0) s_any = any != 0u;
      }
      if (slabs(true)) break;
      csync();
      z_forward();
      {
        SA v2[2];
        if (quads) gather4(v2);
        else gather1(v2);
        put_sums(IC<2>(), v2);
      }
      __syncthreads();
      dots();
      __syncthreads();
      send_coef();
      if (decide) send_sums(2, 1);
      csync();
      coef_sum();
      if (decide) {
        // delta = u^H w - sum_v <C_v|u> <C_v|w>, alpha
        const SA tot = take_sums(1);
        SA t2[2] = {of((T)0), of((T)0)};
        for (int v = lane; v < nproj; v += 32) {
          const W4* c4 = reinterpret_cast<const W4*>(coefp) + v;
          W4 c = c4[0];
          for (int q = 1; q < Q; ++q) {
            const W4 d = c4[q * nproj];
            c.x += d.x; c.y += d.y; c.z += d.z; c.w += d.w;
          }
          t2[0] = acc_add(t2[0], of(c.x * c.z));
          t2[1] = acc_add(t2[1], of(c.y * c.w));
        }
        const SA tv = warp_sums<2, SA>(t2);
        const SA t = acc_lane(tv, (lane & 1) * 16), uw = acc_lane(tot, lane & 1);
        int act = 0;
        if (lane < 2) {
          CgCol<T>& st = s_cg[lane];
          if (st.active) {
            const T delta = acc_val(acc_add(uw, acc_scale(t, (T)-1)));
            const T den = k > 0 ? delta - st.bt * st.gdiv : delta;
            if (!(den > (T)0) || !isfinite(den) || !(st.gam > (T)0)) {
              st.flag = 2;
              st.active = 0;
            } else {
              st.alpha = st.gam / den;
              st.al = st.alpha;
            }
          }
          act = st.active;
        }
        const unsigned any = __ballot_sync(0xffffffffu, act != 0);
        if (lane == 0) s_any = any != 0u;
      }
      __syncthreads();
      if (!s_any) break;
    }
  } else {
    // simplified QMR (kernels_linalg.cu has the recurrences):
    //   t = P_c (H - E) q; alpha = rho / [q, t]; r -= alpha t;
    //   theta, tau from |r|; d = dc d + qc q; x += d; rho' = [r, K r]; q = K r + beta q
    // K r
    auto apply_k = [&](int e, const W4& r) {
      if (PAIR) {
        const T k0 = Kt[2 * e], k1 = Kt[2 * e + 1];
        return W4{k0 * r.x, k0 * r.y, k1 * r.z, k1 * r.w};
      }
      const V k = KC[e];
      return W4{k.x * r.x - k.y * r.y, k.x * r.y + k.y * r.x, k.x * r.z - k.y * r.w, k.x * r.w + k.y * r.z};
    };
    // r^H r and [r, K r] of one entry into v (PAIR: rr0, rr1, rho0, rho1; else rr, rho)
    auto norms = [&](int e, const W4& r, SA* v) {
      if (PAIR) {
        const T f = (h0 + e == 0) ? one : two;
        const T k0 = f * Kt[2 * e], k1 = f * Kt[2 * e + 1];
        acc_fma(v[0], f * r.x, r.x); acc_fma(v[0], f * r.y, r.y);
        acc_fma(v[1], f * r.z, r.z); acc_fma(v[1], f * r.w, r.w);
        acc_fma(v[2], k0 * r.x, r.x); acc_fma(v[2], k0 * r.y, r.y);
        acc_fma(v[3], k1 * r.z, r.z); acc_fma(v[3], k1 * r.w, r.w);
      } else {
        const W4 u = apply_k(e, r);
        acc_fma(v[0], r.x, r.x); acc_fma(v[0], r.y, r.y); acc_fma(v[0], r.z, r.z); acc_fma(v[0], r.w, r.w);
        if (h0 + e == 0) {
          acc_fma(v[1], u.x, r.x); acc_fma(v[1], -u.y, r.y);
          acc_fma(v[2], u.x, r.y); acc_fma(v[2], u.y, r.x);
        } else {
          acc_fma(v[1], two * u.x, r.z); acc_fma(v[1], -two * u.y, r.w);
          acc_fma(v[2], two * u.x, r.w); acc_fma(v[2], two * u.y, r.z);
        }
      }
    };
    const bool decide = warp == kNW - 1;
    {
      SA v[4] = {of((T)0), of((T)0), of((T)0), of((T)0)};
      for (int e = tid; e < nh; e += kTPB) {
        const W4 r = X[e];
        norms(e, r, v);
        const W4 q = apply_k(e, r);
        X[xs + e] = q;
        scatter(e, q);
      }
      put_sums(IC<4>(), v);
      __syncthreads();
      if (decide) send_sums(4, 0);
      csync();
      if (decide) {
        const double t = acc_dbl(take_sums(0));
        const double rr = acc_lane(t, PAIR ? lane & 1 : 0), rx = acc_lane(t, PAIR ? 2 + (lane & 1) : 1), ry = acc_lane(t, 2);
        int act = 0;
        if (lane < nc) {
          QmrCol& st = s_q[lane];
          st.tau2 = rr;
          st.rho = make_double2(rx, PAIR ? 0.0 : ry);
          st.stop = fmax(a.tol2 * rr, stop_abs(lane));
          st.qbest = rr;
          st.rr0 = rr;
          st.rmax = rr;
          st.near = -1;
          st.active = act = (on[lane] && rr > 0.0) ? 1 : 0;
        }
        const unsigned any = __ballot_sync(0xffffffffu, act != 0);
        if (lane == 0) s_any = any != 0u;
      }
      __syncthreads();
    }
    while (s_any) {
      z_inverse();
      csync();
      slabs(false);
      csync();
      z_forward();
      for (int e = tid; e < nh; e += kTPB) Tm[e] = gather(e, X[xs + e]);
      __syncthreads();
      dots();
      __syncthreads();
      send_coef();
      csync();
      coef_sum();
      __syncthreads();
      // t = P_c t and [q, t]
      SA v[4] = {of((T)0), of((T)0), of((T)0), of((T)0)};
      for (int e = tid; e < nh; e += kTPB) {
        const W4 t = project(e, Tm[e]);
        Tm[e] = t;
        const W4 q = X[xs + e];
        if (PAIR) {
          const T f = (h0 + e == 0) ? one : two;
          acc_fma(v[0], f * q.x, t.x); acc_fma(v[0], f * q.y, t.y);
          acc_fma(v[1], f * q.z, t.z); acc_fma(v[1], f * q.w, t.w);
        } else if (h0 + e == 0) {
          acc_fma(v[0], q.x, t.x); acc_fma(v[0], -q.y, t.y);
          acc_fma(v[1], q.x, t.y); acc_fma(v[1], q.y, t.x);
        } else {
          acc_fma(v[0], q.z, t.x); acc_fma(v[0], -q.w, t.y); acc_fma(v[0], q.x, t.z); acc_fma(v[0], -q.y, t.w);
          acc_fma(v[1], q.z, t.y); acc_fma(v[1], q.w, t.x); acc_fma(v[1], q.x, t.w); acc_fma(v[1], q.y, t.z);
        }
      }
      put_sums(IC<2>(), v);
      __syncthreads();
      if (decide) send_sums(2, 1);
      csync();
      if (decide) {
        // alpha = rho / [q, t]: one division in the lanes of Re and Im (PAIR: of the columns)
        const double t = acc_dbl(take_sums(1));
        const double sx = acc_lane(t, PAIR ? lane & 1 : 0), sy = PAIR ? 0.0 : acc_lane(t, 1);
        QmrCol& st = s_q[PAIR ? lane & 1 : 0];
        const double2 rho = st.rho;
        const double num = PAIR ? rho.x : (lane & 1) ? rho.y * sx - rho.x * sy : rho.x * sx + rho.y * sy;
        const double s2 = sx * sx + sy * sy;
        const double al = num / (PAIR ? sx : s2);
        const bool bad = !(s2 > 1e-300 * (rho.x * rho.x + rho.y * rho.y)) || !isfinite(sx) || !isfinite(sy);
        __syncwarp();
        // a stopped column of a pair has q = 0 and keeps its flag
        if (lane < 2 && (!PAIR || (lane < nc && st.active))) {
          if (bad) st.flag = 2;                   // serious breakdown: [q, A q] = 0
          double* d = &st.alpha.x + (PAIR ? 0 : lane);
          *d = bad ? 0.0 : al;
        }
      }
      __syncthreads();
      // r -= alpha t
      {
        const bool a0 = s_q[0].active, a1 = PAIR ? s_q[1].active : a0;
        const T ax = (T)s_q[0].alpha.x, ay = (T)(PAIR ? s_q[1].alpha.x : s_q[0].alpha.y);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = of((T)0);
        for (int e = tid; e < nh; e += kTPB) {
          W4 r = X[e];
          const W4 t = Tm[e];
          if (PAIR) {
            if (a0) { r.x -= ax * t.x; r.y -= ax * t.y; }
            if (a1) { r.z -= ay * t.z; r.w -= ay * t.w; }
          } else {
            r.x = fma(ay, t.y, fma(-ax, t.x, r.x));
            r.y = fma(-ay, t.x, fma(-ax, t.y, r.y));
            r.z = fma(ay, t.w, fma(-ax, t.z, r.z));
            r.w = fma(-ay, t.z, fma(-ax, t.w, r.w));
          }
          X[e] = r;
          norms(e, r, v);
        }
      }
      put_sums(IC<4>(), v);
      __syncthreads();
      if (decide) send_sums(4, 2);
      csync();
      if (decide) {
        // theta^2 = |r|^2 / tau^2, c^2 = 1 / (1 + theta^2) = tau^2 / (tau^2 + |r|^2),
        // tau'^2 = tau^2 theta^2 c^2 = |r|^2 c^2, beta = rho' / rho: one division,
        // the quotients in lanes 0, 1 .. (PAIR: two lanes each)
        const double t = acc_dbl(take_sums(2));
        const int c = PAIR ? lane & 1 : 0, w = PAIR ? lane >> 1 : lane;
        const double rr = acc_lane(t, PAIR ? c : 0), rx = acc_lane(t, PAIR ? 2 + c : 1), ry = PAIR ? 0.0 : acc_lane(t, 2);
        const double tau2 = s_q[c].tau2;
        const double2 rho = s_q[c].rho;
        const double rho2 = PAIR ? rho.x : rho.x * rho.x + rho.y * rho.y;
        double num = w == 0 ? rr : w == 1 ? tau2 : rx, den = w == 0 ? tau2 : w == 1 ? tau2 + rr : rho2;
        if (!PAIR && w == 2) num = rx * rho.x + ry * rho.y;
        if (!PAIR && w == 3) num = ry * rho.x - rx * rho.y;
        const double quo = num / den;
        const double th2 = acc_lane(quo, c), c2 = acc_lane(quo, PAIR ? 2 + c : 1);
        const double bx = acc_lane(quo, PAIR ? 4 + c : 2), by = PAIR ? 0.0 : acc_lane(quo, 3);
        __syncwarp();
        int act = 0;
        if (lane < nc) {
          QmrCol& st = s_q[lane];
          const double2 rn = make_double2(rx, ry);
          st.upd = st.active;
          if (st.active) {
            st.dc = c2 * st.theta2;
            st.qc = make_double2(c2 * st.alpha.x, c2 * st.alpha.y);
            st.tau2 = rr * c2;
            st.theta2 = th2;
            st.beta = rho2 != 0.0 ? make_double2(bx, by) : make_double2(0.0, 0.0);
            st.rho = rn;
            const int it = ++st.it;
            const double qb = st.tau2;
            if (qb < 0.25 * st.qbest) { st.qbest = qb; st.itb = it; }
            if (st.near < 0 && qb <= 4.0 * st.stop) st.near = it;
            st.rmax = fmax(st.rmax, rr);
            // (a large |r| over a flat tau is ordinary far from the floor: an
            // eigenvalue close to the shift)
            const double floor2 = fmax(1e-8 * st.rr0, 4e-12 * st.rmax);
            st.apart = rr > 1e4 * qb && qb <= 100.0 * floor2 ? st.apart + 1 : 0;
            bool stop = false;
            if (st.flag == 2 || !isfinite(st.tau2)) { st.flag = 2; stop = true; }
            else if (qb <= st.stop) { st.flag = 0; stop = true; }
            else if (!(rn.x * rn.x + rn.y * rn.y > 0.0)) { st.flag = 2; stop = true; }
            else if (it >= a.maxit) { st.flag = 1; stop = true; }
            else if (it - st.itb > max(kQmrWindow, 2 * st.itb)) { st.flag = 4; stop = true; }
            else if (sizeof(T) == 4 && qb <= floor2 && it - st.itb > kQmrWindowFloor) {
              st.flag = 4;
              stop = true;
            } else if (sizeof(T) == 4 && st.apart > kApartWait) { st.flag = 4; stop = true; }
            // tau never grows: short of the target after this, the FP64 residual of
            // the refinement decides (1104 columns on 32^3, 256 on 64^3: one or two
            // kept the pass going for 1000 iterations after the others' 80)
            else if (st.near >= 0 && it - st.near > kNearWait) { st.flag = 4; stop = true; }
            if (stop) st.active = 0;
          }
          act = st.active;
        }
        const unsigned any = __ballot_sync(0xffffffffu, act != 0);
        if (lane == 0) s_any = any != 0u;
      }
      __syncthreads();
      // d = dc d + qc q; x += d; q = K r + beta q, into the pencils
      {
        const int l = PAIR ? 1 : 0;
        const bool u0 = s_q[0].upd, u1 = s_q[l].upd, a0 = s_q[0].active, a1 = s_q[l].active, any = s_any;
        const T d0 = (T)s_q[0].dc, d1 = (T)s_q[l].dc;
        const T qx = (T)s_q[0].qc.x, qy = (T)(PAIR ? s_q[1].qc.x : s_q[0].qc.y);
        const T bx = (T)s_q[0].beta.x, by = (T)(PAIR ? s_q[1].beta.x : s_q[0].beta.y);
        for (int e = tid; e < nh; e += kTPB) {
          W4 q = X[xs + e], d = X[2 * xs + e], x = X[3 * xs + e];
          if (PAIR) {
            if (u0) { d.x = d0 * d.x + qx * q.x; d.y = d0 * d.y + qx * q.y; x.x += d.x; x.y += d.y; }
            if (u1) { d.z = d1 * d.z + qy * q.z; d.w = d1 * d.w + qy * q.w; x.z += d.z; x.w += d.w; }
          } else {
            d.x = d0 * d.x + (qx * q.x - qy * q.y);
            d.y = d0 * d.y + (qx * q.y + qy * q.x);
            d.z = d0 * d.z + (qx * q.z - qy * q.w);
            d.w = d0 * d.w + (qx * q.w + qy * q.z);
            x.x += d.x; x.y += d.y; x.z += d.z; x.w += d.w;
          }
          X[2 * xs + e] = d;
          X[3 * xs + e] = x;
          if (!any) continue;
          const W4 z = apply_k(e, X[e]);
          if (PAIR) {
            q.x = a0 ? z.x + bx * q.x : (T)0;
            q.y = a0 ? z.y + bx * q.y : (T)0;
            q.z = a1 ? z.z + by * q.z : (T)0;
            q.w = a1 ? z.w + by * q.w : (T)0;
          } else {
            q = W4{z.x + bx * q.x - by * q.y, z.y + bx * q.y + by * q.x,
                   z.z + bx * q.z - by * q.w, z.w + bx * q.w + by * q.z};
          }
          X[xs + e] = q;
          scatter(e, q);
        }
        __syncthreads();
      }
    }
  }

  // ---- the solution of the pass, added to x64 (own entries)
  int xt[2] = {0, 0};
  for (int e = tid; e < nh; e += kTPB) {
    const int h = h0 + e, g = a.gp[h], m = a.gm[h];
    const W4 x = X[3 * xs + e];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (c >= nc || !on[c]) continue;
      double2* o = a.x64 + (size_t)(c0 + c) * a.npw;
      const double f = scale_out(c);
      const double ux = f * (c ? (double)x.z : (double)x.x), uy = f * (c ? (double)x.w : (double)x.y);
      double2 y = o[g];
      y = make_double2(y.x + ux, y.y + uy);
      o[g] = y;
      xt[c] = max(xt[c], max(hi(y.x), hi(y.y)));
      if (h == 0) continue;
      y = o[m];
      o[m] = PAIR ? make_double2(y.x + ux, y.y - uy) : make_double2(y.x + f * (double)x.z, y.y + f * (double)x.w);
    }
  }
  if (rank == 0 && tid < nc) {
    a.iters[c0 + tid] = CG ? s_cg[tid].it : s_q[tid].it;
    a.flags[c0 + tid] = CG ? s_cg[tid].flag : s_q[tid].flag;
  }
  if (PAIR) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      xt[c] = __reduce_max_sync(0xffffffffu, xt[c]);
      if (lane == 0) atomicMax(at(&s_xtop[c], 0), xt[c]);
    }
  }
  csync();                                        // no CTA leaves while others may reach its memory
  if (PAIR && rank == 0 && tid < nc && (tid ? on[1] : on[0])) a.xmax[c0 + tid] = __hiloint2double(s_xtop[tid], 0);
}

template <typename T, int A, int B> const void* kernel_ptr(int kind) {
  if (kind == COL_CG_PAIR) return (const void*)k_col_solve<T, COL_CG_PAIR, A, B>;
  if (kind == COL_QMR) return (const void*)k_col_solve<T, COL_QMR, A, B>;
  return (const void*)k_col_solve<T, COL_QMR_PAIR, A, B>;
}

}  // namespace col
}  // namespace gw

#define GW_COL_SIZE(A, B)                                       \
  template const void* gw::col::kernel_ptr<float, A, B>(int);   \
  template const void* gw::col::kernel_ptr<double, A, B>(int);
