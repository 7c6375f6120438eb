// small_split.cu -- all k - 1 splits of a narrow cluster in one CTA and one
// launch (Fig. 2 / Fig. 3 with the truncation of Sec. II.B).
//
// Narrow splits are bound by launches, host reads of the ranks and the latency
// of a dozen short kernels per split, not by arithmetic.  Here a CTA keeps the
// split matrix in shared memory and, level by level,
//   - reduces M = diag(lambda_L) Mbar, where it has more rows than columns, to
//     its triangular factor R by Householder reflectors (a barrier per column),
//   - makes the columns of R^H (of M^H) orthogonal by one-sided Jacobi rotations; they
//     are then sigma_i v_i, so no rotations are accumulated (the scheme of
//     Drmac and Veselic, SIAM J. Matrix Anal. Appl. 29, 1322 (2008), which
//     keeps small singular values to relative accuracy),
//   - forms Z = Mbar V and its FP64 column weights, sorts and truncates them by
//     the rule of k_select,
//   - writes the new site and the remainder, which is the next level's matrix.
// Bound by the FP64 units' issue rate within one CTA (a warp's FP64 instruction
// holds its unit for 64 cycles): so four warps, one per unit, a half warp per
// pair of vectors, and the rotation angles in FP32, normalised in FP64 (a
// 16 x 16 split 0.56 -> 0.27 ms); no QR where it would not shorten the vectors
// (0.27 -> 0.20).  Splits of a few columns are bound by instruction fetch: 12 us
// each.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "numeric.cuh"

namespace ctebd {

namespace {

constexpr int kSmThreads = 128, kSmMaxN = 16, kSmSmem = 200 * 1024;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// sums over each half warp, known to all of its lanes
__device__ __forceinline__ double hsum(double v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ void hsum2(double& a, double& b) {
  const int lane = threadIdx.x & 31, base = lane & 16;
  double u = ((lane & 1) ? b : a) + __shfl_xor_sync(0xffffffffu, (lane & 1) ? a : b, 1);
  u += __shfl_xor_sync(0xffffffffu, u, 2);
  u += __shfl_xor_sync(0xffffffffu, u, 4);
  u += __shfl_xor_sync(0xffffffffu, u, 8);
  a = __shfl_sync(0xffffffffu, u, base);
  b = __shfl_sync(0xffffffffu, u, base + 1);
}

// four sums over each half warp, known to all of its lanes
__device__ __forceinline__ void hsum4(double& a, double& b, double& c, double& d) {
  const int lane = threadIdx.x & 31, base = lane & 16;
  double u = ((lane & 2) ? c : a) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? a : c, 2);
  double v = ((lane & 2) ? d : b) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? b : d, 2);
  u = ((lane & 1) ? v : u) + __shfl_xor_sync(0xffffffffu, (lane & 1) ? u : v, 1);
  u += __shfl_xor_sync(0xffffffffu, u, 4);
  u += __shfl_xor_sync(0xffffffffu, u, 8);
  a = __shfl_sync(0xffffffffu, u, base);
  b = __shfl_sync(0xffffffffu, u, base + 1);
  c = __shfl_sync(0xffffffffu, u, base + 2);
  d = __shfl_sync(0xffffffffu, u, base + 3);
}

// largest of K numbers that are not negative, compared as integers
__device__ __forceinline__ double largest(const double* v, int K) {
  long long t = 0;
  for (int i = 0; i < K; i++) t = max(t, __double_as_longlong(v[i]));
  return __longlong_as_double(t);
}

__device__ __forceinline__ double2 wide(float2 v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ double2 wide(double2 v) { return v; }

// S: the tensors' type; the arithmetic is FP64 in both (sigma_i v_i of a rank-deficient matrix then leaves its row
// space by the inputs' rounding only, and a width of 16 keeps the cost of FP64 small).
template <typename S>
__global__ void __launch_bounds__(kSmThreads, 1)
    k_small_chain(const SmallProb* __restrict__ probs, int chi_max, double cutoff, double floor2, int max_sweeps) {
  using CS = typename CplxOf<S>::T;
  using CT = double2;
  const SmallProb P = probs[blockIdx.x];
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double key[kSmMaxN], nrm[kSmMaxN + 1], vinv[kSmMaxN], head[2];
  __shared__ int order[kSmMaxN], sig, r_s;
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, w = tid >> 5, nw = NT >> 5;
  const int c0 = lane & 15;
  // Vectors far below the largest one are what rounding left of a rank-deficient matrix.  They are not rotated
  // (kQuiet, of the squared norm), and all below the truncation's numerical-zero floor are dropped: the weights of
  // their directions, taken from Z, would be their overlap with the large ones.
  // Couplings (squared, relative) up to kLow are left: far below the tensors' rounding, or in FP64 at the level of
  // the sums' own; up to kSkip, ten times the rotations' rounding, only small turns are made (between equal norms
  // noise would turn by 45 degrees for ever).  A sweep with a rotation by more than sqrt(kAgain), or at a coupling
  // above it, is followed by another; what is left after one without is far smaller (of second order, and 1e-7 of
  // it, the angles' rounding).  The angle counts as well as the coupling: between equal norms a tiny coupling turns
  // the two by 45 degrees, and with them their couplings to others, from pairs still to come to pairs already done.
  constexpr double kTiny = 1e-290;
  constexpr float kQuiet = 1e-29f, kLow = sizeof(S) == 4 ? 1e-20f : 3e-31f, kSkip = sizeof(S) == 4 ? 1e-20f : 3.2e-30f;
  constexpr float kAgain = sizeof(S) == 4 ? 1e-10f : 1e-18f;
  const CS* src = reinterpret_cast<const CS*>(P.theta);
  int rdim = P.chiR;
  for (int lev = 1; lev < P.k; lev++) {
    const int j = P.k - lev, m = P.chiL << j, n = 2 * rdim, K = min(m, n);
    const int ld = m | 1, ldx = n | 1;
    CT* A = reinterpret_cast<CT*>(smraw);            // n columns of m (stride ld), then Z
    CT* X = A + (size_t)n * ld;                      // K vectors of n (stride ldx): columns of R^H
    // ---- M = diag(lambda) Mbar, column by column; with no more rows than columns the rows are the vectors
    const bool tall = m > n;
    if (tall)
      for (int e = tid; e < K * ldx; e += NT) X[e] = make_double2(0, 0);
    for (int e = tid; e < m * n; e += NT) {
      const int r = e / n, c = e - r * n;
      const CT v = wide(src[e]);
      const double l = P.lam[r >> j];
      if (tall) A[c * ld + r] = make_double2(v.x * l, v.y * l);
      else X[r * ldx + c] = make_double2(v.x * l, -v.y * l);
    }
    __syncthreads();
    // ---- R: every half warp reflects column c alike and takes its share of the columns behind it
    for (int c = 0; tall && c < K; c++) {
      const CT* a = A + c * ld;
      double s = 0;
      for (int r = c + 1 + c0; r < m; r += 16) s = fma(a[r].x, a[r].x, fma(a[r].y, a[r].y, s));
      s = hsum(s);
      double beta;
      CT tau, inv;
      reflector<double, CT>(a[c], s, beta, tau, inv);
      if (tid == 0) X[c * ldx + c] = make_double2(beta, 0);
      const CT ctau = make_double2(tau.x, -tau.y), cinv = make_double2(inv.x, -inv.y);
      for (int q2 = c + 1 + 2 * w; q2 < n; q2 += 2 * nw) {   // the halves of a warp stay together
        const int q = q2 + (lane >> 4);
        const bool have = q < n;
        CT* b = A + (have ? q : c) * ld;
        // u^H b = b_c + conj(inv) sum conj(a_r) b_r
        CT t = make_double2(0, 0);
        if (have)
          for (int r = c + 1 + c0; r < m; r += 16) addcjmul(t, a[r], b[r]);
        hsum2(t.x, t.y);
        CT y = b[c];
        addmul(y, t, cinv);
        y = mulc(ctau, y);
        if (have) {
          const CT yi = mulc(y, inv);
          for (int r = c + 1 + c0; r < m; r += 16) {
            CT v = b[r];
            submul(v, a[r], yi);
            b[r] = v;
          }
          if (c0 == 0) X[c * ldx + q] = make_double2(b[c].x - y.x, -(b[c].y - y.y));   // conj(R[c][q])
        }
        __syncwarp();
      }
      __syncthreads();
    }
    // ---- the vectors scaled to a largest norm of one (only their directions and ratios are used below)
    for (int i = 2 * w + (lane >> 4); i < 2 * ((K + 1) / 2); i += 2 * nw) {
      const CT x = i < K && c0 < n ? X[i * ldx + c0] : make_double2(0, 0);
      const double s = hsum(fma(x.x, x.x, x.y * x.y));
      if (c0 == 0) nrm[i] = s;
    }
    __syncthreads();
    double top = largest(nrm, K);                    // largest squared norm
    const double unit = top > kTiny ? rcp_nr(sqrt_nr(top)) : 0.0;
    for (int e = tid; e < K * ldx; e += NT) X[e] = make_double2(X[e].x * unit, X[e].y * unit);
    __syncthreads();
    // ---- one-sided Jacobi on the K vectors, circle schedule, a half warp per pair and a lane per element
    const int Kp = (K + 1) & ~1;
    int sweep = 0;
    for (; sweep < max_sweeps; sweep++) {
      if (tid == 0) sig = 0;
      __syncthreads();
      for (int t = 0; t < Kp - 1; t++) {
        for (int i2 = w; 2 * i2 < Kp / 2; i2 += nw) {
          const int i = 2 * i2 + (lane >> 4);
          int p = i == 0 ? t : t + i, q = i == 0 ? Kp - 1 : t - i;
          if (p >= Kp - 1) p -= Kp - 1;
          if (q < 0) q += Kp - 1;
          if (p > q) { const int z = p; p = q; q = z; }
          const bool have = i < Kp / 2 && q < K && c0 < n;
          CT u = make_double2(0, 0), v = u;
          if (have) { u = X[p * ldx + c0]; v = X[q * ldx + c0]; }
          // both norms anew for every pair: updated ones lose what cancels, and small vectors are decided by them
          double a = fma(u.x, u.x, u.y * u.y), d = fma(v.x, v.x, v.y * v.y);
          CT g = make_double2(0, 0);
          addcjmul(g, u, v);
          hsum4(a, d, g.x, g.y);
          // The angle in FP32 (a few 1e-7 of it leave that much of the coupling to the next sweep); the rotation
          // is then normalised in FP64.  rf = 1 / (|u| |v|); couplings are taken relative to the norms.
          const float af = (float)a, df = (float)d;
          const bool big = fminf(af, df) > kQuiet;
          const float rf = big ? rsqrtf(af) * rsqrtf(df) : 0.f;
          const float gx = (float)(g.x * (double)rf), gy = (float)(g.y * (double)rf);
          const float g2 = fmaf(gx, gx, gy * gy);
          if (g2 > kLow) {
            const float ig = rsqrtf(g2), zeta = (float)(d - a) * 0.5f * rf * ig, az = fabsf(zeta);
            const float tt = az < 1e9f ? 1.f / (az + sqrtf(fmaf(az, az, 1.f))) : 0.5f / az, st = (zeta >= 0.f ? tt : -tt) * ig;
            const bool turn = g2 > kSkip || tt * tt < 1e-6f;
            const double tx = (double)(st * gx), ty = -(double)(st * gy);
            const double n2 = fma(tx, tx, fma(ty, ty, 1.0));
            double co = (double)rsqrtf((float)n2);   // 1e-7, cubed by one step of third order
            const double er = fma(-n2 * co, co, 1.0);
            co = fma(co * er, fma(er, 0.375, 0.5), co);
            const double sx = co * tx, sy = co * ty;
            if (have && turn) {    // u' = co u - s v, v' = co v + conj(s) u
              X[p * ldx + c0] = make_double2(fma(co, u.x, fma(-sx, v.x, sy * v.y)), fma(co, u.y, fma(-sx, v.y, -sy * v.x)));
              X[q * ldx + c0] = make_double2(fma(co, v.x, fma(sx, u.x, sy * u.y)), fma(co, v.y, fma(sx, u.y, -sy * u.x)));
            }
            if (c0 == 0 && turn && fmaxf(g2, tt * tt) > kAgain) sig = 1;
          }
          __syncwarp();
        }
        __syncthreads();
      }
      const int again = sig;
      __syncthreads();
      if (!again) break;
    }
    // ---- v_i = x_i / |x_i|.  Norms and spectra by the general division and root, a few of each per split: with the
    // Newton routines of numeric.cuh the states of exact runs of 12 qubits were off by 5.6e-16 and 5.0e-16 on average
    // (two families of 60 circuits), now by 3.7e-16 and 4.2e-16 (block Jacobi: 3.5e-16 and 4.5e-16), in the same time.
    for (int i = 2 * w + (lane >> 4); i < 2 * ((K + 1) / 2); i += 2 * nw) {
      const CT x = i < K && c0 < n ? X[i * ldx + c0] : make_double2(0, 0);
      const double s = hsum(fma(x.x, x.x, x.y * x.y));
      if (c0 == 0) nrm[i] = s;
    }
    __syncthreads();
    if (tid < K) {
      top = largest(nrm, K);
      vinv[tid] = nrm[tid] > fmax(floor2 * top, kTiny) ? 1.0 / sqrt(nrm[tid]) : 0.0;
    }
    __syncthreads();
    // ---- Z = Mbar V: thread -> column i, rows in pairs (neighbouring threads share the rows)
    for (int e = tid; e < K * ((m + 1) / 2); e += NT) {
      const int i = e % K, r0 = e / K * 2;
      const CT* x = X + i * ldx;
      const CS* s0 = src + (size_t)r0 * n;
      const CS* s1 = r0 + 1 < m ? s0 + n : s0;
      CT z0 = make_double2(0, 0), z1 = z0;
      for (int c = 0; c < n; c++) {
        const CT v = x[c];
        addmul(z0, wide(s0[c]), v);
        addmul(z1, wide(s1[c]), v);
      }
      const double iv = vinv[i];
      A[i * ld + r0] = make_double2(z0.x * iv, z0.y * iv);
      if (r0 + 1 < m) A[i * ld + r0 + 1] = make_double2(z1.x * iv, z1.y * iv);
    }
    __syncthreads();
    // ---- weights rho_i = sum lambda^2 |z|^2
    for (int i = w; i < K; i += nw) {
      const CT* z = A + i * ld;
      double s = 0;
      for (int r = lane; r < m; r += 32) {
        const double lx = P.lam[r >> j];
        s = fma(lx * lx, fma(z[r].x, z[r].x, z[r].y * z[r].y), s);
      }
      s = wsum(s);
      if (lane == 0) key[i] = s;
    }
    __syncthreads();
    // ---- descending order (ties by index), truncation as in k_select
    if (w == 0) {
      const long long mine = lane < K ? __double_as_longlong(key[lane]) : -1;   // not negative: ordered as integers
      int rank = 0;
      for (int i = 0; i < K; i++) {
        const long long o = __double_as_longlong(key[i]);
        rank += o > mine || (o == mine && i < lane) ? 1 : 0;
      }
      // NaN weights take no rank of their own: keep every slot a valid index
      if (lane < K) order[lane] = lane;
      __syncwarp();
      if (lane < K) order[rank] = lane;
      __syncwarp();
      const double k0 = lane < K ? fmax(key[order[lane]], 0.0) : 0.0;
      double tail = k0;                              // inclusive sum from the smallest weight on
#pragma unroll
      for (int o = 1; o < kSmMaxN; o <<= 1) {
        const double a = __shfl_down_sync(0xffffffffu, tail, o);
        if (lane + o < 32) tail += a;
      }
      const double W = __shfl_sync(0xffffffffu, tail, 0), first = __shfl_sync(0xffffffffu, k0, 0);
      int r = K;
      if (cutoff > 0) {
        const unsigned b = __ballot_sync(0xffffffffu, lane >= 1 && lane < K && tail > cutoff * W);
        r = b ? 32 - __clz(b) : 1;
      }
      r = max(1, min(r, __popc(__ballot_sync(0xffffffffu, lane < K && k0 > floor2 * first))));
      const int rc = r;
      r = min(r, chi_max);
      const double kept = r == K ? W : wsum(lane < r ? k0 : 0.0);
      double* lam = P.lam_out[j];
      if (lane < r) lam[lane] = kept > 0 ? sqrt(k0 / kept) : 0.0;
      if (lane == 0) {
        double* res = P.res + 8 * (lev - 1);
        res[0] = r; res[1] = r == K || !(W > 0) ? 1.0 : fmin(kept / W, 1.0); res[2] = W;
        res[3] = kept; res[4] = rc;
        res[5] = sweep >= max_sweeps ? 1.0 : 0.0;
        r_s = r;
        head[0] = kept > 0 ? 1.0 / sqrt(kept) : 0.0;
      }
    }
    __syncthreads();
    const int r = r_s;
    const double scale = head[0];
    // ---- the new right site (rows v_i^H) and the remainder
    CS* site = reinterpret_cast<CS*>(P.site[j]);
    for (int e = tid; e < r * n; e += NT) {
      const int mu = e / n, c = e - mu * n, i = order[mu];
      const CT v = X[i * ldx + c];
      site[e].x = (S)(v.x * vinv[i]);
      site[e].y = (S)(-v.y * vinv[i]);
    }
    CS* rem = reinterpret_cast<CS*>(lev == P.k - 1 ? P.site[0] : P.rem);
    for (int e = tid; e < r * m; e += NT) {
      const int row = e / r, mu = e - row * r;
      const CT v = A[order[mu] * ld + row];
      rem[e].x = (S)(v.x * scale);
      rem[e].y = (S)(v.y * scale);
    }
    __syncthreads();
    src = rem;
    rdim = r;
  }
}

}  // namespace

size_t small_smem(int m, int n) {
  return 16 * ((size_t)n * (m | 1) + (size_t)std::min(m, n) * (n | 1));
}

// Rule: widths up to 16 (a lane per element) and matrices that fit a CTA's
// shared memory.  Batched kernels / this kernel, whole calls: 10 FP64 clusters
// of 4 sites at chi 8 4.8 / 4.0 ms; a run of 100 qubits at chi 256 (most of
// its bonds narrow) 16.1 ms without, 13.5 with the limit at 8, 10.9 at 16; 12
// exact FP64 qubits 3.4 / 2.2; one 16 x 16 split 0.24 / 0.20 in the kernels.  Wider ones lose: an FP64
// kernel of the same scheme took 3.4 ms in place of 1.7 at width 30.
bool small_fits(int m, int n) { return n <= kSmMaxN && small_smem(m, n) <= kSmSmem; }

template <typename S>
cudaError_t launch_small_chain(const SmallProb* d_probs, int count, size_t smem, int chi_max, double cutoff,
                               double floor2, int max_sweeps, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(k_small_chain<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmSmem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  k_small_chain<S><<<count, kSmThreads, smem, s>>>(d_probs, chi_max, cutoff, floor2, max_sweeps);
  return cudaGetLastError();
}
template cudaError_t launch_small_chain<float>(const SmallProb*, int, size_t, int, double, double, int, cudaStream_t);
template cudaError_t launch_small_chain<double>(const SmallProb*, int, size_t, int, double, double, int, cudaStream_t);

}  // namespace ctebd
