// Sums of the one-launch solvers in FP32 instructions (this GPU runs FP64 at 1/64
// of that rate): unevaluated sums of two or three floats whose additions are
// error-free (Knuth's TwoSum, 6 instructions; the error of a product by one
// multiply-add).  The types of CUDA are all this file needs, so that its
// arithmetic can be compiled for the host and compared with exact sums.
//   float2  hi + lo, renormalised after each addition: about 47 bits.
//   F3      the errors of the sum are summed the same way and theirs in a third
//           float (Ogita, Rump and Oishi, Accurate sum and dot product, SIAM J.
//           Sci. Comput. 26, 2005: SumK, K = 3): as exact as FP64 sums of exact
//           products.  24 instructions a product, against one of FP64 that takes
//           as long as 64 and two conversions that take as long each.
#pragma once

namespace gw {

// by precision: FP64, or two floats
template <typename T> struct AccOf { using type = double; };
template <> struct AccOf<float> { using type = float2; };
template <typename T> using Acc = typename AccOf<T>::type;
struct F3 { float x, y, z; };
// FP64, or three floats
template <typename T> struct Acc3Of { using type = double; };
template <> struct Acc3Of<float> { using type = F3; };
template <typename T> using Acc3 = typename Acc3Of<T>::type;

__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

__device__ __forceinline__ float acc_add(float a, float b) { return a + b; }
__device__ __forceinline__ double acc_add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 acc_add(float2 a, float2 b) {
  float e;
  const float s = two_sum(a.x, b.x, e);
  const float t = __fadd_rn(e, __fadd_rn(a.y, b.y));
  const float h = __fadd_rn(s, t);
  return make_float2(h, __fsub_rn(t, __fsub_rn(h, s)));
}
__device__ __forceinline__ F3 acc_add(F3 a, F3 b) {
  float e, f, g;
  const float s = two_sum(a.x, b.x, e);
  const float t = two_sum(a.y, b.y, f);
  const float u = two_sum(t, e, g);
  return F3{s, u, __fadd_rn(__fadd_rn(a.z, b.z), __fadd_rn(f, g))};
}
// acc += a, without renormalising (7 instructions)
__device__ __forceinline__ void acc_in(float2& acc, float a) {
  float e;
  acc.x = two_sum(acc.x, a, e);
  acc.y = __fadd_rn(acc.y, e);
}
// acc += a b
__device__ __forceinline__ void acc_fma(double& acc, double a, double b) { acc += a * b; }
__device__ __forceinline__ void acc_fma(F3& acc, float a, float b) {
  const float p = __fmul_rn(a, b);
  acc = acc_add(acc, F3{p, fmaf(a, b, -p), 0.f});
}
__device__ __forceinline__ double acc_scale(double a, double c) { return a * c; }
__device__ __forceinline__ float2 acc_scale(float2 a, float c) {
  const float p = __fmul_rn(a.x, c);
  const float e = fmaf(a.y, c, fmaf(a.x, c, -p));
  const float h = __fadd_rn(p, e);
  return make_float2(h, __fsub_rn(e, __fsub_rn(h, p)));
}

// a scalar as a sum (A: the type), and back: rounded to the scalar, and in FP64
template <typename A> struct AccFrom;
template <> struct AccFrom<float> { static __device__ __forceinline__ float of(float x) { return x; } };
template <> struct AccFrom<double> { static __device__ __forceinline__ double of(double x) { return x; } };
template <> struct AccFrom<float2> {
  static __device__ __forceinline__ float2 of(float x) { return make_float2(x, 0.f); }
};
template <> struct AccFrom<F3> { static __device__ __forceinline__ F3 of(float x) { return F3{x, 0.f, 0.f}; } };
__device__ __forceinline__ float acc_val(float a) { return a; }
__device__ __forceinline__ double acc_val(double a) { return a; }
__device__ __forceinline__ float acc_val(float2 a) { return __fadd_rn(a.x, a.y); }
__device__ __forceinline__ double acc_dbl(double a) { return a; }
__device__ __forceinline__ double acc_dbl(F3 a) { return (double)a.x + ((double)a.y + (double)a.z); }

// from another lane: lane ^ o, lane l
__device__ __forceinline__ float acc_shfl(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double acc_shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ float2 acc_shfl(float2 a, int o) { return make_float2(acc_shfl(a.x, o), acc_shfl(a.y, o)); }
__device__ __forceinline__ F3 acc_shfl(F3 a, int o) {
  return F3{acc_shfl(a.x, o), acc_shfl(a.y, o), acc_shfl(a.z, o)};
}
__device__ __forceinline__ double acc_lane(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }
__device__ __forceinline__ float2 acc_lane(float2 a, int l) {
  return make_float2(__shfl_sync(0xffffffffu, a.x, l), __shfl_sync(0xffffffffu, a.y, l));
}

}  // namespace gw
