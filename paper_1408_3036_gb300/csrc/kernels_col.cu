// Column solver: launch shapes, launches, and the data in its orders
// (col_kernel.cuh has the kernel; kernels_col_*.cu its instances).
#include <algorithm>
#include <cmath>
#include <tuple>

#include "col_layout.cuh"
#include "device_cache.h"
#include "linalg.cuh"

namespace gw {
namespace col {

// lengths with kernels, N1 <= N2 as near as they go
#define GW_COL_SIZES(X)                                                                                          \
  X(3, 4) X(3, 5) X(4, 4) X(3, 6) X(4, 5) X(4, 6) X(5, 5) X(3, 9) X(5, 6) X(4, 8) X(6, 6) X(5, 8) X(5, 9) X(6, 8) \
  X(5, 10) X(6, 9) X(6, 10) X(8, 8) X(8, 9) X(8, 10)

template <typename T> const void* kernel_of(int N, int kind) {
  switch (N) {
#define GW_COL_CASE(A, B) case A * B: return kernel_ptr<T, A, B>(kind);
    GW_COL_SIZES(GW_COL_CASE)
#undef GW_COL_CASE
    default: return nullptr;
  }
}

inline cudaLaunchConfig_t config(cudaLaunchAttribute* at, int q, int grid, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(kTPB);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = q;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return c;
}

// Kernel attributes (once per function and device) and the clusters of size q
// that run at once on the current device (0: this size does not run here).
int active_clusters(const void* f, int lq, size_t smem) {
  static DeviceCache<const void*, bool> ready;
  static DeviceCache<std::tuple<const void*, int, size_t>, int> known;
  int dev = 0, n = 0;
  bool set = false;
  const bool ok =
      cudaGetDevice(&dev) == cudaSuccess && ready.get(dev, f, &set, [&](bool* s) {
        return *s = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) == cudaSuccess &&
                    cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
      }) && known.get(dev, {f, lq, smem}, &n, [&](int* c) {
        cudaLaunchAttribute at;
        const cudaLaunchConfig_t cfg = config(&at, 1 << lq, 1 << lq, smem, nullptr);
        return cudaOccupancyMaxActiveClusters(c, f, &cfg) == cudaSuccess;
      });
  if (!ok) cudaGetLastError();
  return ok ? n : 0;
}

}  // namespace col

template <typename T>
bool col_shape(const ColPlan& p, int kind, int N, int nproj, int nunit, int cta_div, ColShape* out) {
  if (!p.ok || nunit < 1 || nproj > kMaxOcc) return false;
  const void* f = col::kernel_of<T>(N, kind);
  if (!f) return false;
  // An iteration of one unit takes a fixed time (barriers, reductions, scalar
  // steps) and its work over Q CTAs; microseconds, fitted to sweeps over Q
  // (45^3 grid, 11 rows, FP32 SQMR: 107, 57, 38, 26, 25 for Q = 1 .. 16; 48^3,
  // 16 rows, CG pair: 55, 30, 22 for Q = 4 .. 16, FP64 424, 222 for Q = 8, 16;
  // 16^3, 4 rows, FP64: 88, 57, 42, 35, 36).  Units beyond the clusters that
  // run at once wait for a free one: whole rounds for CG (columns alike, but the
  // last few pairs of a cell are its fastest); for SQMR the slowest columns,
  // which start first, take about twice the mean.  The order of the sums, and
  // with it the last bits, depends on Q: FP64 results do not depend on how many
  // contexts share the GPU, so there Q does not either.
  const bool f32 = sizeof(T) == 4;
  // (contexts that share the GPU keep it busy about half the time each)
  const double share = f32 ? std::max(0.5 * cta_div, 1.0) : 1.0;
  const double fixed = f32 ? 11.0 : 27.0;
  const double work = (f32 ? 1.0e-3 : 1.5e-2) * N * N * N + (f32 ? 0.9e-3 : 1.66e-2) * nproj * p.nh;
  double best = 1e300;
  for (int lq = 0; lq < kColNQ; ++lq) {
    const int Q = 1 << lq, ldz = 2 * p.maxpair[lq], nhl = p.maxh[lq];
    if (Q > N || Q > p.npair) continue;
    ColShape s;
    s.lq = lq;
    const int nzl = (N + Q - 1) / Q;
    auto fits = [&](int nsb, bool vec, bool c, bool v = false) {
      s.nsb = nsb;
      s.vec_smem = vec;
      s.c_smem = c;
      s.v_smem = v;
      s.smem = col::layout<T>(kind, s, N, p.P, p.npair, ldz, nhl, nproj).total;
      return s.smem <= col::kSmemMax;
    };
    // slabs together: the fewest rounds of the CTA's threads (FP64: of a warp
    // per scheduler) over the passes of all batches; then the rows and the
    // potential where room is left
    auto rounds_of = [&](int nsb) {
      const int unit = sizeof(T) == 4 ? col::kTPB : 128;
      auto r = [&](long tasks) { return (double)((tasks + unit - 1) / unit); };
      double t = 0.0;
      for (int sb = 0; sb < nzl; sb += nsb) {
        const long ns = std::min(nsb, nzl - sb);
        t += 2.0 * (r(ns * p.N2 * p.P) + r(ns * p.N1 * p.P) + r(ns * p.N2 * N)) + 1.6 * r(ns * p.N1 * N) + 2.0;
      }
      return t;
    };
    // the projector rows (read twice an iteration) before the vectors (read
    // and written once) where the rows are the larger traffic
    const bool rows_first = 2 * nproj * sizeof(cpx<T>) > 9 * 4 * sizeof(T);
    int nsb = 0;
    bool vec = false, c = false, v = false;
    for (int pass = 0; pass < 4 && nsb == 0; ++pass) {
      vec = pass == 0 || pass == (rows_first ? 2 : 1);
      c = pass == 0 || pass == (rows_first ? 1 : 2);
      for (int n = 1; n <= nzl; ++n)
        if (fits(n, vec, c) && (nsb == 0 || rounds_of(n) < rounds_of(nsb))) nsb = n;
    }
    if (nsb == 0) continue;
    v = fits(nsb, vec, c, true);
    fits(nsb, vec, c, v);
    s.vec_elems = vec ? 0 : 16 * (size_t)p.nh;
    const int act = col::active_clusters(f, lq, s.smem);
    if (act < 1) continue;
    const double load = (double)nunit * share / act;
    const double rounds = kind != COL_CG_PAIR ? std::max(1.0, 0.5 * load)
                                              : load <= 1.25 ? std::max(1.0, load) : std::ceil(load);
    const double t = rounds * (fixed + lq + work / Q);
    if (t < best) { best = t; *out = s; }
  }
  return best < 1e300;
}

template <typename T>
cudaError_t launch_col_solve(cudaStream_t s, int kind, const ColArgs<T>& a) {
  const int Q = 1 << a.sh.lq;
  const void* f = col::kernel_of<T>(a.N, kind);
  if (!f || col::active_clusters(f, a.sh.lq, a.sh.smem) < 1) return cudaErrorNotSupported;
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t c = col::config(&at, Q, a.nunit * Q, a.sh.smem, s);
  ColArgs<T> arg = a;
  void* args[] = {&arg};
  ++g_launches;
  return cudaLaunchKernelExC(&c, f, args);
}

namespace col {
template <typename T>
__global__ void k_col_perm_v(int N, int N1, int N2, const T* __restrict__ v, T* __restrict__ out) {
  const int n = N * N * N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int c = i % N, x = (i / N) % N, z = i / (N * N);
    const int y = c / N2 + N1 * (c % N2);
    out[i] = v[((size_t)x * N + y) * N + z];
  }
}
template <typename T>
__global__ void k_col_perm_rows(int nh, int npw, int rows, const int* __restrict__ gp, const cpx<T>* __restrict__ C,
                                cpx<T>* __restrict__ out) {
  const size_t n = (size_t)nh * rows;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const size_t v = i / nh;
    out[i] = C[v * npw + gp[i - v * nh]];
  }
}
template <typename T>
__global__ void k_col_perm_kin(int nh, const int* __restrict__ gp, const T* __restrict__ kin, T* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nh; i += gridDim.x * blockDim.x) out[i] = kin[gp[i]];
}
}  // namespace col

// vloc_s / kin (fixed per cell) and C (per occupied block) in the solver's
// orders; a null input leaves that part alone.
template <typename T>
cudaError_t launch_col_permute(cudaStream_t s, const ColPlan& p, int N, int npw, const T* vloc_s, const cpx<T>* C,
                               int nproj, const T* kin, ColPrec<T>& out) {
  if (vloc_s) {
    ++g_launches;
    col::k_col_perm_v<T><<<std::min((N * N * N + 255) / 256, 152 * 8), 256, 0, s>>>(N, p.N1, p.N2, vloc_s, out.Vp);
  }
  if (kin) {
    ++g_launches;
    col::k_col_perm_kin<T><<<(p.nh + 255) / 256, 256, 0, s>>>(p.nh, p.gp, kin, out.kin);
  }
  if (C && nproj > 0) {
    const size_t n = (size_t)p.nh * nproj;
    ++g_launches;
    col::k_col_perm_rows<T><<<(int)std::min<size_t>((n + 255) / 256, 152 * 16), 256, 0, s>>>(p.nh, npw, nproj, p.gp, C,
                                                                                              out.Ch);
  }
  return cudaGetLastError();
}

bool col_radices(int N, int* N1, int* N2) {
  switch (N) {
#define GW_COL_CASE(A, B) case A * B: *N1 = A; *N2 = B; return true;
    GW_COL_SIZES(GW_COL_CASE)
#undef GW_COL_CASE
    default: return false;
  }
}

#define GW_COL_INST(T)                                                                                     \
  template bool col_shape<T>(const ColPlan&, int, int, int, int, int, ColShape*);                               \
  template cudaError_t launch_col_solve<T>(cudaStream_t, int, const ColArgs<T>&);                          \
  template cudaError_t launch_col_permute<T>(cudaStream_t, const ColPlan&, int, int, const T*, const cpx<T>*, int, \
                                             const T*, ColPrec<T>&);


GW_COL_INST(float)
GW_COL_INST(double)

}  // namespace gw
