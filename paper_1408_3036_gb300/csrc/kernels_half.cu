// FP64 projector and residual on half the sphere.
//
// The projector rows are real in real space (c(-G) = conj c(G)), so with the
// half entries h of ColPlan (G and -G; h = 0: G = 0)
//   <C|y> = sum_h conj(c) y(G) + c y(-G)
// takes two real products per row and half entry for a column that is real in
// real space and four for a complex one, half of what the sums over the whole
// sphere take; the update y -= C k forms Re c k and Im c k once for G and -G.
// FP64 instructions are what these kernels cost on this GPU (a warp-wide one
// holds a scheduler's FP64 unit for about 64 cycles): a warp keeps a tile of
// rows x columns in registers, its lane sums are reduced by recursive halving,
// and the partial sums over chunks of entries are added by the kernel that
// uses the coefficients (no ticket, no serial tail).
// 16 rows, 16 columns, 12053 plane waves: coefficients and update 61 + 31 us
// with one warp per row and shuffle sums per value, now 15 + 14 (19 + 14 before
// the products became chains of fused multiply-adds; 64 rows, 256 complex
// columns, 38401 plane waves 5.0 -> 3.3 ms, its multiply-adds alone 2.1).
#include <algorithm>

#include "col.cuh"
#include "gw_common.cuh"
#include "linalg.cuh"

namespace gw {
namespace {

constexpr int kRT = 4;              // rows of a warp's tile
constexpr int kGramWarps = 4;       // warps per CTA

template <int M> __device__ __forceinline__ double lane_sums(double* v) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = M / 2; n >= 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < n; ++k) {
      const double keep = up ? v[n + k] : v[k], give = up ? v[k] : v[n + k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
#pragma unroll
  for (int q = 16 / M; q >= 1; q >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], q);
  return v[0];
}

// part[chunk][col][row] (REAL) or [chunk][col][row][2]: one warp per (chunk,
// tile of CT columns, tile of kRT rows)
template <bool REAL>
__global__ void __launch_bounds__(32 * kGramWarps)
k_gram_half(const double2* __restrict__ C, int nrow, int nh, const int* __restrict__ gp, const int* __restrict__ gm,
            const double2* __restrict__ Y, int npw, int ncol, const int* __restrict__ active, int nchunk, int chunk,
            double* __restrict__ part) {
  constexpr int CT = REAL ? 4 : 2, NV = REAL ? 1 : 2;
  const int lane = threadIdx.x & 31;
  const int nrt = (nrow + kRT - 1) / kRT, nct = (ncol + CT - 1) / CT;
  const long w = (long)blockIdx.x * kGramWarps + (threadIdx.x >> 5);
  if (w >= (long)nchunk * nct * nrt) return;
  const int rt = (int)(w % nrt), ct = (int)((w / nrt) % nct), ck = (int)(w / ((long)nrt * nct));
  const int v0 = rt * kRT, c0 = ct * CT;
  if (active) {
    bool any = false;
    for (int c = 0; c < CT; ++c) any |= (c0 + c < ncol) && active[c0 + c];
    if (!any) return;
  }
  double acc[kRT * CT * NV];
#pragma unroll
  for (int k = 0; k < kRT * CT * NV; ++k) acc[k] = 0.0;
  const int h1 = min(nh, (ck + 1) * chunk);
  for (int h = ck * chunk + lane; h < h1; h += 32) {
    double2 c[kRT];
#pragma unroll
    for (int r = 0; r < kRT; ++r) c[r] = C[(size_t)min(v0 + r, nrow - 1) * nh + h];
    const int g = gp[h], m = REAL ? 0 : gm[h];
    double2 y[CT], z[CT];
#pragma unroll
    for (int k = 0; k < CT; ++k) {
      const double2* col = Y + (size_t)min(c0 + k, ncol - 1) * npw;
      y[k] = col[g];
      if (!REAL) z[k] = col[m];
    }
#pragma unroll
    for (int k = 0; k < CT; ++k) {
      if (REAL) {
        if (h == 0) y[k] = make_double2(0.5 * y[k].x, 0.5 * y[k].y);
#pragma unroll
        for (int r = 0; r < kRT; ++r) {
          double& t = acc[r * CT + k];
          t = fma(c[r].y, y[k].y, fma(c[r].x, y[k].x, t));
        }
      } else {
        if (h == 0) z[k] = make_double2(0.0, 0.0);
        const double a = y[k].x + z[k].x, b = y[k].y - z[k].y, d = y[k].y + z[k].y, e = z[k].x - y[k].x;
#pragma unroll
        for (int r = 0; r < kRT; ++r) {
          double& t = acc[(r * CT + k) * 2];
          double& u = acc[(r * CT + k) * 2 + 1];
          t = fma(c[r].y, b, fma(c[r].x, a, t));
          u = fma(c[r].y, e, fma(c[r].x, d, u));
        }
      }
    }
  }
  constexpr int M = kRT * CT * NV;       // 16
  const double t = lane_sums<M>(acc);
  const int q = lane / (32 / M), k = q / NV, r = k / CT, col = c0 + k % CT;
  if (lane % (32 / M) == 0 && v0 + r < nrow && col < ncol)
    part[(((size_t)ck * ncol + col) * nrow + v0 + r) * NV + q % NV] = REAL ? 2.0 * t : t;
}

constexpr int kHT = 256;

// coefficients of one column into sc[nrow][NV]: groups of threads over the chunks, then over the groups in order
template <int NV>
__device__ __forceinline__ void take_coef(const double* __restrict__ part, int nchunk, int ncol, int col, int nrow,
                                          double* sc, double* tmp) {
  const int n = nrow * NV;
  const int grp = max(1, min(min(kHT / n, nchunk), 16));
  if (grp == 1) {
    for (int j = threadIdx.x; j < n; j += kHT) {
      double s = 0.0;
      for (int k = 0; k < nchunk; ++k) s += part[((size_t)k * ncol + col) * n + j];
      sc[j] = s;
    }
  } else {
    const int g = threadIdx.x / n, j = threadIdx.x - g * n;
    if (g < grp) {
      double s = 0.0;
      for (int k = g; k < nchunk; k += grp) s += part[((size_t)k * ncol + col) * n + j];
      tmp[g * n + j] = s;
    }
    __syncthreads();
    if (threadIdx.x < n) {
      double s = tmp[threadIdx.x];
      for (int k = 1; k < grp; ++k) s += tmp[k * n + threadIdx.x];
      sc[threadIdx.x] = s;
    }
  }
  __syncthreads();
}

// y(G), y(-G) minus sum_v C_v coef_v at half entry h
template <bool REAL>
__device__ __forceinline__ void sub_rows(const double2* __restrict__ C, int nrow, int nh, int h, const double* sc,
                                         double2& y, double2& z) {
  double a1 = 0.0, a2 = 0.0, a3 = 0.0, a4 = 0.0;
  int v = 0;
  for (; v + 4 <= nrow; v += 4) {
    double2 c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = C[(size_t)(v + q) * nh + h];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double k0 = sc[(v + q) * (REAL ? 1 : 2)];
      a1 += c[q].x * k0;
      a4 += c[q].y * k0;
      if (!REAL) {
        const double k1 = sc[(v + q) * 2 + 1];
        a3 += c[q].x * k1;
        a2 += c[q].y * k1;
      }
    }
  }
  for (; v < nrow; ++v) {
    const double2 c = C[(size_t)v * nh + h];
    const double k0 = sc[v * (REAL ? 1 : 2)];
    a1 += c.x * k0;
    a4 += c.y * k0;
    if (!REAL) {
      const double k1 = sc[v * 2 + 1];
      a3 += c.x * k1;
      a2 += c.y * k1;
    }
  }
  if (REAL) {                       // c k at G, conj(c) k at -G
    y.x -= a1; y.y -= a4;
    z.x -= a1; z.y += a4;
  } else {
    y.x -= a1 - a2; y.y -= a3 + a4;
    z.x -= a1 + a2; z.y -= a3 - a4;
  }
}

// Y -= C coef; grid (chunks of kHT half entries, ncol)
template <bool REAL>
__global__ void __launch_bounds__(kHT)
k_proj_half(const double2* __restrict__ C, int nrow, int nh, const int* __restrict__ gp, const int* __restrict__ gm,
            double2* __restrict__ Y, int npw, int ncol, const int* __restrict__ active, int nchunk,
            const double* __restrict__ part) {
  __shared__ double sc[2 * kMaxOcc], tmp[kHT];
  const int col = blockIdx.y;
  if (active && !active[col]) return;
  take_coef<REAL ? 1 : 2>(part, nchunk, ncol, col, nrow, sc, tmp);
  const int h = blockIdx.x * kHT + threadIdx.x;
  if (h >= nh) return;
  double2* y = Y + (size_t)col * npw;
  const int g = gp[h], m = gm[h];
  double2 a = y[g], b = y[m];
  sub_rows<REAL>(C, nrow, nh, h, sc, a, b);
  y[g] = a;
  if (h > 0) y[m] = b;
}

// r -= C coef (r = b - A x on entry), then |r|^2, |b|^2, |x|^2 per column
template <bool REAL>
__global__ void __launch_bounds__(kHT)
k_residual_half(const double2* __restrict__ C, int nrow, int nh, const int* __restrict__ gp,
                const int* __restrict__ gm, double2* __restrict__ r, const double2* __restrict__ b,
                const double2* __restrict__ x, int npw, int ncol, const int* __restrict__ active, int nchunk,
                const double* __restrict__ part, double* __restrict__ sums, unsigned* __restrict__ cnt,
                double* __restrict__ out) {
  __shared__ double sc[2 * kMaxOcc], tmp[kHT];
  const int col = blockIdx.y;
  if (active && !active[col]) return;
  take_coef<REAL ? 1 : 2>(part, nchunk, ncol, col, nrow, sc, tmp);
  const int h = blockIdx.x * kHT + threadIdx.x;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (h < nh) {
    const size_t o = (size_t)col * npw;
    const int g = gp[h], m = gm[h];
    double2 p = r[o + g], q = r[o + m];
    const double2 bp = b[o + g], bq = b[o + m], xp = x[o + g], xq = x[o + m];
    sub_rows<REAL>(C, nrow, nh, h, sc, p, q);
    r[o + g] = p;
    v[0] = p.x * p.x + p.y * p.y;
    v[1] = bp.x * bp.x + bp.y * bp.y;
    v[2] = xp.x * xp.x + xp.y * xp.y;
    if (h > 0) {
      r[o + m] = q;
      v[0] += q.x * q.x + q.y * q.y;
      v[1] += bq.x * bq.x + bq.y * bq.y;
      v[2] += xq.x * xq.x + xq.y * xq.y;
    }
  }
  const double t = lane_sums<4>(v);
  __syncthreads();
  if ((threadIdx.x & 7) == 0) tmp[(threadIdx.x >> 5) * 4 + ((threadIdx.x & 31) >> 3)] = t;
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
    for (int k = 0; k < kHT / 32; ++k) s += tmp[k * 4 + threadIdx.x];
    sums[((size_t)blockIdx.x * ncol + col) * 3 + threadIdx.x] = s;
  }
  if (!last_block(&cnt[col], gridDim.x)) return;
  if (threadIdx.x < 3) {
    double s;
    sum_records<1>(sums + (size_t)col * 3 + threadIdx.x, gridDim.x, 3 * (size_t)ncol, &s);
    out[(size_t)threadIdx.x * ncol + col] = s;
  }
}

// Chunks of entries of the coefficient sums: enough warps for two per
// scheduler, at least 64 entries each.
int half_chunks(bool real, int nrow, int nh, int ncol, int* chunk) {
  const long tiles = (long)((nrow + kRT - 1) / kRT) * ((ncol + (real ? 3 : 1)) / (real ? 4 : 2));
  const int want = (int)std::min<long>(std::max<long>((1216 + tiles - 1) / tiles, 1), (nh + 63) / 64);
  *chunk = ((nh + want - 1) / want + 31) / 32 * 32;
  return (nh + *chunk - 1) / *chunk;
}

}  // namespace

size_t half_part_elems(int nrow, int nh, int ncol) {
  int c;
  const size_t a = (size_t)half_chunks(true, nrow, nh, ncol, &c) * ncol * nrow;
  const size_t b = (size_t)half_chunks(false, nrow, nh, ncol, &c) * ncol * nrow * 2;
  return std::max(a, b);
}
size_t half_sum_elems(int nh, int ncol) { return (size_t)((nh + kHT - 1) / kHT) * ncol * 3; }

int launch_gram_half(cudaStream_t s, bool real, const ColPlan& p, const double2* Ch, int nrow, const double2* Y,
                     int npw, int ncol, const int* active, double* part) {
  int chunk = 0;
  const int n = half_chunks(real, nrow, p.nh, ncol, &chunk), ct = real ? 4 : 2;
  const long warps = (long)n * ((nrow + kRT - 1) / kRT) * ((ncol + ct - 1) / ct);
  const unsigned grid = (unsigned)((warps + kGramWarps - 1) / kGramWarps);
  ++g_launches;
  if (real)
    k_gram_half<true><<<grid, 32 * kGramWarps, 0, s>>>(Ch, nrow, p.nh, p.gp, p.gm, Y, npw, ncol, active, n, chunk, part);
  else
    k_gram_half<false><<<grid, 32 * kGramWarps, 0, s>>>(Ch, nrow, p.nh, p.gp, p.gm, Y, npw, ncol, active, n, chunk, part);
  return n;
}

void launch_proj_half(cudaStream_t s, bool real, const ColPlan& p, const double2* Ch, int nrow, double2* Y, int npw,
                      int ncol, const int* active, int nchunk, const double* part) {
  dim3 g((p.nh + kHT - 1) / kHT, ncol);
  ++g_launches;
  if (real) k_proj_half<true><<<g, kHT, 0, s>>>(Ch, nrow, p.nh, p.gp, p.gm, Y, npw, ncol, active, nchunk, part);
  else k_proj_half<false><<<g, kHT, 0, s>>>(Ch, nrow, p.nh, p.gp, p.gm, Y, npw, ncol, active, nchunk, part);
}

void launch_residual_half(cudaStream_t s, bool real, const ColPlan& p, const double2* Ch, int nrow, double2* r,
                          const double2* b, const double2* x, int npw, int ncol, const int* active, int nchunk,
                          const double* part, double* sums, unsigned* cnt, double* out) {
  dim3 g((p.nh + kHT - 1) / kHT, ncol);
  ++g_launches;
  if (real)
    k_residual_half<true><<<g, kHT, 0, s>>>(Ch, nrow, p.nh, p.gp, p.gm, r, b, x, npw, ncol, active, nchunk, part, sums,
                                            cnt, out);
  else
    k_residual_half<false><<<g, kHT, 0, s>>>(Ch, nrow, p.nh, p.gp, p.gm, r, b, x, npw, ncol, active, nchunk, part, sums,
                                             cnt, out);
}

}  // namespace gw
