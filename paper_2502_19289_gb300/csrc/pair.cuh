// pair.cuh -- arithmetic of the divide and conquer solver: FP64, or pairs of
// FP32 numbers.
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cfloat>

#include "numeric.cuh"

namespace ctebd {

// ---------------------------------------------------------------------------
// Arithmetic of the tridiagonal problem: FP64 in the FP64 mode, pairs of FP32
// numbers (Dekker, Numer. Math. 18, 224 (1971); about 46 bits) in the FP32
// mode.  One warp's FP64 instruction takes its FP64 unit 64 cycles on this
// chip (measured, dependent or not), a pair operation 7 to 20 cycles.  46 bits
// are far more than the FP32 matrix carries: weights are resolved to 1e-13 of
// the total, and the smallest cutoff that FP32 resolves is 1e-11.  T is scaled
// to a largest entry of order one first, for the FP32 exponent range.
//
// Reciprocal and root of a pair are one Newton step from the FP32 ones, whose
// relative error is 2^-24: the step squares it and adds a few roundings of
// 2^-47, in all below 2^-44 for arguments from 1e-25 to 1e25 (beyond, the low
// halves leave the normal range).
// ---------------------------------------------------------------------------
struct Pair {
  float h, l;
};
__device__ __forceinline__ Pair quick_sum(float a, float b) {   // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Pair two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair operator+(Pair a, Pair b) {
  Pair s = two_sum(a.h, b.h);
  const Pair t = two_sum(a.l, b.l);
  s = quick_sum(s.h, __fadd_rn(s.l, t.h));
  return quick_sum(s.h, __fadd_rn(s.l, t.l));
}
__device__ __forceinline__ Pair operator-(Pair a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Pair operator-(Pair a, Pair b) { return a + (-b); }
__device__ __forceinline__ Pair operator*(Pair a, Pair b) {
  const float p = __fmul_rn(a.h, b.h), e = fmaf(a.h, b.h, -p);
  return quick_sum(p, fmaf(a.h, b.l, fmaf(a.l, b.h, e)));
}
__device__ __forceinline__ bool operator<(Pair a, Pair b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }
__device__ __forceinline__ bool operator>(Pair a, Pair b) { return b < a; }
__device__ __forceinline__ bool operator==(Pair a, Pair b) { return a.h == b.h && a.l == b.l; }

// the operations that differ by type; R: run precision
template <typename R> struct Real;
template <> struct Real<double> {
  using T = double;
  static constexpr double kEps = DBL_EPSILON, kFloor = 1e-30;
  static __device__ __forceinline__ bool is_zero(double x) { return x == 0.0; }
  static __device__ __forceinline__ double of(double x) { return x; }
  static __device__ __forceinline__ double inf() { return CUDART_INF; }
  static __device__ __forceinline__ double rcp(double x) { return rcp_nr(x); }
  static __device__ __forceinline__ double root(double x) { return x > 1e-290 ? sqrt_nr(x) : 0.0; }
  static __device__ __forceinline__ double mag(double x) { return fabs(x); }
  static __device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
  static __device__ __forceinline__ float f(double x) { return (float)x; }
  static __device__ __forceinline__ double run(double x) { return x; }
  static __device__ __forceinline__ double shfl(double x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); }
};
template <> struct Real<float> {
  using T = Pair;
  static constexpr double kEps = 1.4e-14, kFloor = 1e-20;   // 2^-46
  static __device__ __forceinline__ bool is_zero(Pair x) { return x.h == 0.f; }
  static __device__ __forceinline__ Pair of(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
  }
  static __device__ __forceinline__ Pair of(float x) { return {x, 0.f}; }
  static __device__ __forceinline__ Pair inf() { return {CUDART_INF_F, 0.f}; }
  static __device__ __forceinline__ Pair rcp(Pair b) {   // one Newton step from the FP32 estimate
    const float r = rcp_nr(b.h), p = __fmul_rn(b.h, r);
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.f, p), fmaf(b.h, r, -p)), __fmul_rn(b.l, r));
    return quick_sum(r, __fmul_rn(e, r));
  }
  static __device__ __forceinline__ Pair root(Pair a) {
    if (!(a.h > 1e-36f)) return {0.f, 0.f};
    const float s = sqrt_nr(a.h), p = __fmul_rn(s, s);
    const float e = __fadd_rn(__fsub_rn(__fsub_rn(a.h, p), fmaf(s, s, -p)), a.l);   // a - s^2
    return quick_sum(s, __fmul_rn(0.5f * e, rcp_nr(s)));
  }
  static __device__ __forceinline__ Pair mag(Pair a) { return a.h < 0 ? -a : a; }
  static __device__ __forceinline__ Pair mad(Pair a, Pair b, Pair c) { return a * b + c; }
  static __device__ __forceinline__ float f(Pair a) { return a.h; }
  static __device__ __forceinline__ float run(Pair a) { return a.h; }
  static __device__ __forceinline__ Pair shfl(Pair a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
  }
};

}  // namespace ctebd
