// amplitude.cu -- <bits|psi> of the MPS: a chain of vector-matrix products,
// one per site, in FP64 (products of the run precision's values).
//
// The left half of the chain runs left to right, the right half right to left,
// each by its own CTAs of one launch.  A CTA computes a slice of the next
// vector and passes it on (exchange.cuh); what bounds it is the chain: one
// exchange of 1.2 us and one slice per site, so a site's values are read
// before its vector is complete.  A launch per site in which one thread summed
// a whole column took 88 us a site at chi = 256.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "exchange.cuh"
#include "internal.h"

namespace ctebd {

namespace {

// four warps: one per FP64 unit of an SM
constexpr int kAmpThreads = 128, kAmpAhead = 16;   // values of a site read ahead, per thread

template <typename R> struct C2;
template <> struct C2<float> { using T = float2; };
template <> struct C2<double> { using T = double2; };

template <typename R>
__global__ void __launch_bounds__(kAmpThreads, 1)
    k_amp_half(const AmpSite* __restrict__ sites, int n, int G, int max_chi, unsigned char* __restrict__ slots,
               double2* __restrict__ ends, int* err) {
  using CT = typename C2<R>::T;
  constexpr int SB = Slot<double2>::kBytes;
  extern __shared__ __align__(16) unsigned char smraw[];
  double2* vs = reinterpret_cast<double2*>(smraw);          // the vector so far
  double2* red = vs + max_chi;                              // partial sums, one per thread
  __shared__ int bad;
  const int half = blockIdx.x / G, c = blockIdx.x % G, tid = threadIdx.x, mid = n / 2;
  const int count = half == 0 ? mid : n - mid;
  unsigned char* ex = slots + (size_t)half * 2 * max_chi * SB;
  if (tid == 0) { vs[0] = make_double2(1.0, 0.0); bad = 0; }
  // slice of a site: outputs [o0, o0 + no) of this CTA, `len` terms each;
  // thread -> output oi, terms t0, t0 + nt, ...
  struct Slice {
    int outs, o0, no, len, oi, t0, nt;
    long long so, st;                                       // strides of an output and of a term
    const CT* S;
  };
  auto site_at = [&](int k) { return sites[half == 0 ? k : n - 1 - k]; };
  auto open_site = [&](const AmpSite& a, Slice& z, CT (&ahead)[kAmpAhead]) {
    z.outs = half == 0 ? a.cr : a.cl;
    z.len = half == 0 ? a.cl : a.cr;
    const int per = G > 1 ? (z.outs + G - 1) / G : z.outs;
    z.o0 = c * per;
    z.no = max(0, min(per, z.outs - z.o0));
    int lg = 0;                                             // threads per output: a power of two
    while ((1 << lg) < per && (1 << lg) < kAmpThreads) lg++;
    const int p2 = 1 << lg;
    z.nt = kAmpThreads >> lg;
    // neighbouring threads read neighbouring elements of a row
    z.oi = half == 0 ? tid & (p2 - 1) : tid / z.nt;
    z.t0 = half == 0 ? tid >> lg : tid & (z.nt - 1);
    z.so = half == 0 ? 1 : 2LL * a.cr;
    z.st = half == 0 ? 2LL * a.cr : 1;
    z.S = reinterpret_cast<const CT*>(a.S) + (long long)a.bit * a.cr;
#pragma unroll
    for (int i = 0; i < kAmpAhead; i++) {
      const int t = z.t0 + i * z.nt;
      if (z.oi < z.no && t < z.len) ahead[i] = z.S[(z.o0 + z.oi) * z.so + t * z.st];
    }
  };
  // a site's values are on their way while the site before it is worked on,
  // its description one site earlier
  Slice cur{}, nxt{};
  CT now[kAmpAhead], ahead[kAmpAhead];
  AmpSite desc{};
  if (count > 0) open_site(site_at(0), cur, now);
  if (count > 1) desc = site_at(1);
  __syncthreads();
  for (int k = 0; k < count; k++) {
    const unsigned seq = k + 1;
    unsigned char* buf = ex + (size_t)(seq & 1u) * max_chi * SB;
    const bool more = k + 1 < count;
    if (more) open_site(desc, nxt, ahead);
    if (k + 2 < count) desc = site_at(k + 2);
    const int p2 = kAmpThreads / cur.nt;
    for (int ob = 0; ob < cur.no; ob += p2) {               // one turn unless a lone CTA has more outputs than threads
      double2 acc = make_double2(0, 0);
      auto term = [&](int t, CT s) {
        const double2 v = vs[t];
        acc.x = fma(v.x, (double)s.x, acc.x); acc.x = fma(-v.y, (double)s.y, acc.x);
        acc.y = fma(v.x, (double)s.y, acc.y); acc.y = fma(v.y, (double)s.x, acc.y);
      };
      if (ob + cur.oi < cur.no) {
        if (ob == 0) {
#pragma unroll
          for (int i = 0; i < kAmpAhead; i++) {
            if (i * cur.nt >= cur.len) break;               // for all threads alike
            if (cur.t0 + i * cur.nt < cur.len) term(cur.t0 + i * cur.nt, now[i]);
          }
        }
        for (int t = cur.t0 + (ob == 0 ? kAmpAhead * cur.nt : 0); t < cur.len; t += cur.nt)
          term(t, cur.S[(cur.o0 + ob + cur.oi) * cur.so + t * cur.st]);
      }
      // sum over the nt threads of an output
      const int at = cur.oi * cur.nt + cur.t0;
      red[at] = acc;
      __syncthreads();
      for (int s = cur.nt >> 1; s > 0; s >>= 1) {
        if (cur.t0 < s) {
          red[at].x += red[at + s].x;
          red[at].y += red[at + s].y;
        }
        __syncthreads();
      }
      if (tid < p2 && ob + tid < cur.no) {
        const double2 v = red[tid * cur.nt];
        if (G > 1) Slot<double2>::put(buf + (size_t)(cur.o0 + ob + tid) * SB, v, seq);
        else vs[max_chi + kAmpThreads + ob + tid] = v;      // the next vector (a lone CTA)
      }
      __syncthreads();
    }
    if (G > 1) {
      // A CTA without a slice of the next site skips this vector.  (One that
      // has a slice holds up the vector after the next, so the slots it still
      // has to read are not written again before.)
      const bool need = more ? nxt.no > 0 : c == 0;
      for (int j = tid; need && j < cur.outs; j += kAmpThreads) {
        const unsigned char* ad[1] = {buf + (size_t)j * SB};
        double2 v[1];
        if (!poll(ad, seq, v, err, kWaitAmplitude)) bad = 1;
        vs[j] = v[0];
      }
    } else {
      for (int j = tid; j < cur.outs; j += kAmpThreads) vs[j] = vs[max_chi + kAmpThreads + j];
    }
    __syncthreads();
    if (bad) return;
    if (more) {
      cur = nxt;
#pragma unroll
      for (int i = 0; i < kAmpAhead; i++) now[i] = ahead[i];
    }
  }
  if (c == 0) {
    const int m = count > 0 ? cur.outs : 1;
    for (int j = tid; j < m; j += kAmpThreads) ends[(size_t)half * max_chi + j] = vs[j];
  }
}

// the two halves' vectors meet at the middle bond
__global__ void __launch_bounds__(kAmpThreads) k_amp_dot(const double2* __restrict__ ends, int len, int max_chi,
                                                         double2* __restrict__ out) {
  __shared__ double2 red[kAmpThreads];
  double2 acc = make_double2(0, 0);
  for (int j = threadIdx.x; j < len; j += kAmpThreads) {
    const double2 a = ends[j], b = ends[max_chi + j];
    acc.x = fma(a.x, b.x, acc.x); acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y); acc.y = fma(a.y, b.x, acc.y);
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int s = kAmpThreads / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      red[threadIdx.x].x += red[threadIdx.x + s].x;
      red[threadIdx.x].y += red[threadIdx.x + s].y;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = red[0];
}

}  // namespace

// CTAs per half: about 1024 complex products per CTA and site, whose FP64
// arithmetic then takes about the time of the exchange
int amp_ctas(int max_chi, int n_sm) {
  const long long e = (long long)max_chi * max_chi;
  return (int)std::max<long long>(1, std::min<long long>(n_sm / 2, e / 1024));
}

// exchange slots, the halves' vectors, the result
size_t amp_scratch_bytes(int max_chi) {
  return (size_t)4 * max_chi * Slot<double2>::kBytes + ((size_t)2 * max_chi + 1) * sizeof(double2);
}

template <typename R>
cudaError_t launch_amplitude(const AmpSite* d_sites, int n, int mid_chi, int max_chi, int ctas, unsigned char* scratch,
                             double2* out, int* err, cudaStream_t s) {
  const size_t slot_bytes = (size_t)4 * max_chi * Slot<double2>::kBytes;
  double2* ends = reinterpret_cast<double2*>(scratch + slot_bytes);
  // vector, partial sums, and the next vector of a lone CTA
  const size_t sm = sizeof(double2) * (max_chi + kAmpThreads + (ctas == 1 ? max_chi : 0));
  static bool attr = false;
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(k_amp_half<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(double2) * (2 * 2048 + kAmpThreads));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  cudaError_t e;
  if (ctas > 1) {
    e = cudaMemsetAsync(scratch, 0, slot_bytes, s);
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&d_sites, (void*)&n, (void*)&ctas, (void*)&max_chi, (void*)&scratch, (void*)&ends, (void*)&err};
    e = cudaLaunchCooperativeKernel((const void*)k_amp_half<R>, dim3(2 * ctas), dim3(kAmpThreads), args, sm, s);
  } else {
    k_amp_half<R><<<2, kAmpThreads, sm, s>>>(d_sites, n, 1, max_chi, scratch, ends, err);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  k_amp_dot<<<1, kAmpThreads, 0, s>>>(ends, mid_chi, max_chi, out);
  return cudaGetLastError();
}
template cudaError_t launch_amplitude<float>(const AmpSite*, int, int, int, int, unsigned char*, double2*, int*,
                                              cudaStream_t);
template cudaError_t launch_amplitude<double>(const AmpSite*, int, int, int, int, unsigned char*, double2*, int*,
                                              cudaStream_t);

}  // namespace ctebd
