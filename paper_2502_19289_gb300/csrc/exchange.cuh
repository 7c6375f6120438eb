// exchange.cuh -- values passed between the CTAs of one cooperative launch.
#pragma once
#include <cuda_runtime.h>

#include "waits.h"

namespace ctebd {

// ---- exchange between the CTAs of a group ------------------------------------
// Every exchanged value travels in one 128-bit store together with its
// sequence number, and the reader polls the value itself: one trip through L2
// instead of data, fence, flag and data again.  A slot's value is valid when
// its sequence number is the step's; the slots are zeroed before the launch
// and numbers start at 1.  Polls are bounded: one that runs out sets *err to the
// caller's code (waits.h); the first one's stays.
constexpr int kSpinLimit = 1 << 21;

__device__ __forceinline__ void st128(void* p, unsigned long long lo, unsigned long long hi) {
  asm volatile("{\n.reg .b128 q;\nmov.b128 q, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], q;\n}\n" ::"l"(p), "l"(lo),
               "l"(hi)
               : "memory");
}
__device__ __forceinline__ void ld128(const void* p, unsigned long long& lo, unsigned long long& hi) {
  asm volatile("{\n.reg .b128 q;\nld.relaxed.gpu.global.b128 q, [%2];\nmov.b128 {%0, %1}, q;\n}\n"
               : "=l"(lo), "=l"(hi)
               : "l"(p)
               : "memory");
}
template <typename CT> struct Slot;
template <> struct Slot<float2> {
  static constexpr int kBytes = 16;
  static __device__ __forceinline__ void put(unsigned char* p, float2 v, unsigned seq) {
    st128(p, (unsigned long long)__float_as_uint(v.x) | ((unsigned long long)__float_as_uint(v.y) << 32), seq);
  }
  static __device__ __forceinline__ bool get(const unsigned char* p, unsigned seq, float2& v) {
    unsigned long long lo, hi;
    ld128(p, lo, hi);
    v = make_float2(__uint_as_float((unsigned)lo), __uint_as_float((unsigned)(lo >> 32)));
    return (unsigned)hi == seq;
  }
};
template <> struct Slot<double2> {
  static constexpr int kBytes = 32;
  static __device__ __forceinline__ void put(unsigned char* p, double2 v, unsigned seq) {
    st128(p, (unsigned long long)__double_as_longlong(v.x), seq);
    st128(p + 16, (unsigned long long)__double_as_longlong(v.y), seq);
  }
  static __device__ __forceinline__ bool get(const unsigned char* p, unsigned seq, double2& v) {
    unsigned long long a, b, c, d;
    ld128(p, a, b);
    ld128(p + 16, c, d);
    v = make_double2(__longlong_as_double((long long)a), __longlong_as_double((long long)c));
    return (unsigned)b == seq && (unsigned)d == seq;
  }
};

// Poll N slots (those with a non-null address) until all carry seq.  (All of
// them from the first poll on: waiting for one and then reading the others
// costs another trip, 28.1 -> 29.5 ms for two 2048-wide problems.)
template <int N, typename CT>
__device__ __forceinline__ bool poll(const unsigned char* const (&p)[N], unsigned seq, CT (&v)[N], int* err,
                                     int code) {
  bool have[N];
#pragma unroll
  for (int i = 0; i < N; i++) { have[i] = p[i] == nullptr; v[i] = CT{0, 0}; }
  for (int it = 0; it < kSpinLimit; it++) {
    bool all = true;
#pragma unroll
    for (int i = 0; i < N; i++)
      if (!have[i]) have[i] = Slot<CT>::get(p[i], seq, v[i]);
#pragma unroll
    for (int i = 0; i < N; i++) all = all && have[i];
    if (all) return true;
    if ((it & 1023) == 1023 && *(volatile int*)err) break;
  }
  atomicCAS(err, kWaitNone, code);
  return false;
}

}  // namespace ctebd
