// kernels.cu -- CUDA kernels of the cluster update (sm_103a).
//
// The split of Fig. 2 / Fig. 3 is computed from the Schmidt-weighted Gram
// matrix G = M^H diag(lambda_L^2) M (grouped GEMM), its eigenvectors V from a
// batched block-Jacobi solver, and the weighted column norms of Mbar V, which
// give the kept weights directly from M (Eq. 4 numerator and denominator).
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cfloat>
#include <cstdint>

#include "internal.h"

namespace ctebd {

template <typename R> struct C2;
template <> struct C2<float> { using T = float2; };
template <> struct C2<double> { using T = double2; };

template <typename T> __device__ __forceinline__ T cmk(double re, double im);
template <> __device__ __forceinline__ float2 cmk<float2>(double re, double im) {
  return make_float2((float)re, (float)im);
}
template <> __device__ __forceinline__ double2 cmk<double2>(double re, double im) {
  return make_double2(re, im);
}
template <typename T> __device__ __forceinline__ T cmul(T a, T b) {
  T r; r.x = a.x * b.x - a.y * b.y; r.y = a.x * b.y + a.y * b.x; return r;
}
template <typename T> __device__ __forceinline__ T cconj(T a) { a.y = -a.y; return a; }
template <typename T> __device__ __forceinline__ void cfma(T& acc, T a, T b) {
  acc.x = fma(a.x, b.x, acc.x); acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y); acc.y = fma(a.y, b.x, acc.y);
}
template <typename T> __device__ __forceinline__ T cscale(T a, double s) {
  a.x = (decltype(a.x))(a.x * s); a.y = (decltype(a.y))(a.y * s); return a;
}

// ---------------------------------------------------------------------------
// Grouped complex GEMM: output tiles of 16 TM x 16 TM, 256 threads with TM x TM
// elements each, the next slice of K loaded while the present one is used.
// Merge chain (theta), U application, Gram matrix and Mbar*V all use it.
// Sums run over k in the same order whatever the tile.
// ---------------------------------------------------------------------------
template <typename R, int TM>
__global__ void __launch_bounds__(256) k_gemm(const GemmProb* __restrict__ probs,
                                              const long long* __restrict__ tile_off, int n_probs) {
  using CT = typename C2<R>::T;
  constexpr int BM = 16 * TM, BK = TM == 4 ? (sizeof(R) == 8 ? 8 : 16) : TM == 2 ? (sizeof(R) == 8 ? 16 : 32) : 32;
  constexpr int PER = BM * BK / 256;
  __shared__ CT As[2][BK][BM + 1];
  __shared__ CT Bs[2][BK][BM + 1];
  const long long tid_tile = blockIdx.x;
  int lo = 0, hi = n_probs;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (tile_off[mid] <= tid_tile) lo = mid; else hi = mid;
  }
  const GemmProb P = probs[lo];
  long long t = tid_tile - tile_off[lo];
  const int tilesN = (P.N + BM - 1) / BM, tilesM = (P.M + BM - 1) / BM;
  const int tn = (int)(t % tilesN);
  t /= tilesN;
  const int tm = (int)(t % tilesM);
  const long long bidx = t / tilesM;
  const CT* A = (const CT*)P.A + bidx * P.sA;
  const CT* B = (const CT*)P.B + bidx * P.sB;
  CT* Cm = (CT*)P.C + bidx * P.sC;
  const int m0 = tm * BM, n0 = tn * BM;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  CT acc[TM][TM], ra[PER], rb[PER];
#pragma unroll
  for (int i = 0; i < TM; i++)
#pragma unroll
    for (int j = 0; j < TM; j++) acc[i][j] = cmk<CT>(0, 0);
  // element e of a slice: k fastest where k is contiguous in memory, else the tile's row (column)
  auto fetch = [&](int k0) {
#pragma unroll
    for (int it = 0; it < PER; it++) {
      const int e = threadIdx.x + it * 256;
      const int m = P.opA == 0 ? e / BK : e % BM, ka = k0 + (P.opA == 0 ? e % BK : e / BM);
      CT v = cmk<CT>(0, 0);
      if (m0 + m < P.M && ka < P.K) {
        v = P.opA == 0 ? A[(long long)(m0 + m) * P.lda + ka] : cconj(A[(long long)ka * P.lda + m0 + m]);
        if (P.kw) {
          const double wk = P.kw[ka >> P.kw_shift];
          v = cscale(v, P.kw_pow == 1 ? wk : wk * wk);
        }
      }
      ra[it] = v;
      const int n = P.opB == 0 ? e % BM : e / BK, kb = k0 + (P.opB == 0 ? e / BM : e % BK);
      CT w = cmk<CT>(0, 0);
      if (n0 + n < P.N && kb < P.K)
        w = P.opB == 0 ? B[(long long)kb * P.ldb + n0 + n] : cconj(B[(long long)(n0 + n) * P.ldb + kb]);
      rb[it] = w;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int it = 0; it < PER; it++) {
      const int e = threadIdx.x + it * 256;
      if (P.opA == 0) As[buf][e % BK][e / BK] = ra[it]; else As[buf][e / BM][e % BM] = ra[it];
      if (P.opB == 0) Bs[buf][e / BM][e % BM] = rb[it]; else Bs[buf][e % BK][e / BK] = rb[it];
    }
  };
  fetch(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < P.K; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < P.K;
    if (more) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; kk++) {
      CT a[TM], b[TM];
#pragma unroll
      for (int i = 0; i < TM; i++) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TM; j++) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < TM; j++) cfma(acc[i][j], a[i], b[j]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TM; i++) {
    const int m = m0 + ty + 16 * i;
    if (m >= P.M) continue;
#pragma unroll
    for (int j = 0; j < TM; j++) {
      const int n = n0 + tx + 16 * j;
      if (n < P.N) Cm[(long long)m * P.ldc + n] = cscale(acc[i][j], P.alpha);
    }
  }
}

long long gemm_tiles(const GemmProb& p, int tm) {
  const int bm = 16 * tm;
  return (long long)((p.M + bm - 1) / bm) * ((p.N + bm - 1) / bm) * p.batch;
}

// Rule: the tile whose waves over the SMs cost least, a wave of 16 TM costing
// TM^2 (FP32: times 1.3 and 2 for the two smaller ones, which read shared
// memory more often per product).  Products of the splits are small next to
// the chip -- FP64 runs at 2 lanes a clock and SM, so every idle SM counts.
// Merge and projection kernels of a step, tile 64 / 32 / 16: four FP64
// clusters of 128-wide splits 0.55 + 1.08 / 0.16 + 0.29 / 0.13 + 0.23 ms; eight
// FP64 30-wide 0.074 + 0.143 / 0.027 + 0.047 / 0.019 + 0.023; sixteen FP32
// 48-wide 0.065 + 0.092 / 0.051 + 0.058 / 0.038 + 0.058; eight FP32 200-wide
// 0.087 + 0.147 / 0.074 + 0.138 / 0.092 + 0.162.
int gemm_tile(const GemmProb* probs, int n, bool fp64, int n_sm) {
  int best = 4;
  double cost = 0;
  for (int tm = 4; tm >= 1; tm >>= 1) {
    long long tiles = 0;
    for (int i = 0; i < n; i++) tiles += gemm_tiles(probs[i], tm);
    const double c = (double)((tiles + n_sm - 1) / n_sm) * tm * tm * (fp64 || tm == 4 ? 1.0 : tm == 2 ? 1.3 : 2.0);
    if (tm == 4 || c < cost) { best = tm; cost = c; }
  }
  return best;
}

template <typename R>
cudaError_t launch_gemm(const GemmProb* d_probs, const long long* d_tile_off, int n_probs,
                        long long total_tiles, int tm, cudaStream_t s) {
  if (total_tiles <= 0) return cudaSuccess;
  if (total_tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)total_tiles;
  if (tm == 4) k_gemm<R, 4><<<grid, 256, 0, s>>>(d_probs, d_tile_off, n_probs);
  else if (tm == 2) k_gemm<R, 2><<<grid, 256, 0, s>>>(d_probs, d_tile_off, n_probs);
  else k_gemm<R, 1><<<grid, 256, 0, s>>>(d_probs, d_tile_off, n_probs);
  return cudaGetLastError();
}
template cudaError_t launch_gemm<float>(const GemmProb*, const long long*, int, long long, int, cudaStream_t);
template cudaError_t launch_gemm<double>(const GemmProb*, const long long*, int, long long, int, cudaStream_t);

// ---------------------------------------------------------------------------
// Batched block-Jacobi eigensolver for Hermitian G (two-sided, parallel
// round-robin ordering of JB-blocks).  Per round: (1) every block pair's
// 2JB x 2JB sub-matrix is diagonalised in shared memory by cyclic Jacobi,
// giving a unitary J_p; (2) G <- J^H G J and V <- V J tile by tile.
// ---------------------------------------------------------------------------
template <typename R> struct EigCfg;
// MAXS: inner sweeps when the whole matrix is one block pair (nb == 2);
// with several block pairs one inner sweep per round is enough, the outer
// sweeps converge the rest.
template <> struct EigCfg<float> { static constexpr int JB = 32; static constexpr int MAXS = 10; };
template <> struct EigCfg<double> { static constexpr int JB = 16; static constexpr int MAXS = 12; };
int eig_block(bool fp64) { return fp64 ? EigCfg<double>::JB : EigCfg<float>::JB; }

// Round-robin (circle method) schedule: N players, round t in [0, N-1), slot i.
__device__ __forceinline__ void circle(int t, int i, int N, int& a, int& b) {
  const int M = N - 1;
  if (i == 0) { a = t; b = N - 1; }
  else { a = (t + i) % M; b = (t - i + M) % M; }
  if (a > b) { int x = a; a = b; b = x; }
}

// 2x2 Hermitian Jacobi rotation [[a, g], [g*, d]] -> diagonal.  Rotations
// whose coupling is below the rounding level (relative 4 eps sqrt(a d), or
// absolute eps * trace(G)) are skipped; a rotation is "significant" (keeps the
// sweep loop going) when the relative coupling |g| / sqrt(a d) exceeds
// sqrt(eps) and |g| is well above the absolute noise floor.
template <typename R>
__device__ __forceinline__ void jrot_params(R a, R d, typename C2<R>::T g, R floor_abs, R rel_skip, R& c,
                                            R& s, typename C2<R>::T& ph, bool& skip, bool& signif) {
  using CT = typename C2<R>::T;
  const R eps = sizeof(R) == 4 ? (R)FLT_EPSILON : (R)DBL_EPSILON;
  const R ag = sqrt(g.x * g.x + g.y * g.y);
  const R rad = sqrt(fabs(a * d));
  skip = !(ag > rel_skip * eps * rad) || !(ag > floor_abs) || ag == (R)0;
  signif = !skip && ag > sqrt(eps) * rad && ag > (R)8 * floor_abs;
  if (skip) { c = 1; s = 0; ph = cmk<CT>(1, 0); return; }
  const R zeta = (d - a) / ((R)2 * ag);
  R t;
  if (fabs(zeta) > (R)1e15) t = (R)0.5 / zeta;
  else t = (zeta >= 0 ? (R)1 : (R)-1) / (fabs(zeta) + sqrt((R)1 + zeta * zeta));
  c = (R)1 / sqrt((R)1 + t * t);
  s = c * t;
  ph.x = g.x / ag;
  ph.y = -g.y / ag;  // e^{-i phi}
}

template <typename R, bool ONE_PAIR>
__global__ void __launch_bounds__(256, ONE_PAIR ? 2 : 3) k_eig_inner(const EigProb* __restrict__ probs, int round) {
  using CT = typename C2<R>::T;
  constexpr int JB = EigCfg<R>::JB, D = 2 * JB, LD = D + 1, NBLK = JB * (JB + 1) / 2;
  // per thread: A blocks; Q rows row0 + j QSTEP (one rotation per thread)
  constexpr int NB_T = (NBLK + 255) / 256, QSTEP = 256 / JB, QROWS = D / QSTEP;
  constexpr unsigned PMASK = JB == 32 ? 0xffffffffu : ((1u << JB) - 1u);   // lanes of the parameter phase
  static_assert(256 % JB == 0 && D % QSTEP == 0, "inner kernel: 256 threads");
  const EigProb P = probs[blockIdx.y];
  // each problem takes one variant whatever else shares the launch
  if (!P.active || round >= P.nb - 1 || (int)blockIdx.x >= P.nb / 2 || ONE_PAIR != (P.nb == 2)) return;
  extern __shared__ unsigned char smraw[];
  CT* A = reinterpret_cast<CT*>(smraw);
  CT* Q = A + D * LD;
  // rotation parameters of the round: tan(theta / 2), sin(theta), phase, and
  // the pair (p, q) of each of the JB rotations
  R* tu = reinterpret_cast<R*>(Q + D * LD);
  R* sn = tu + JB;
  CT* ph = reinterpret_cast<CT*>(sn + JB);
  int* pp = reinterpret_cast<int*>(ph + JB);
  int* pq = pp + JB;
  unsigned short* blk = reinterpret_cast<unsigned short*>(pq + JB);   // pair blocks a <= b: a | b << 8
  __shared__ int nrot, nsig;
  __shared__ R nmove;   // weight moved by this sweep's significant rotations
  int I, J;
  circle(round, blockIdx.x, P.nb, I, J);
  const bool cut = P.cut_hi > 0 && P.jflag;
  if (cut && (((I + 1) * JB <= P.cut_lo && (J + 1) * JB <= P.cut_lo) ||
              (I * JB >= P.cut_hi && J * JB >= P.cut_hi))) {
    if (threadIdx.x == 0) P.jflag[blockIdx.x] = 0;   // both blocks on one side of the cut
    return;
  }
  const CT* G = (const CT*)P.G;
  for (int e = threadIdx.x; e < D * D; e += blockDim.x) {
    const int li = e / D, lj = e % D;
    const long long gi = li < JB ? (long long)I * JB + li : (long long)J * JB + li - JB;
    const long long gj = lj < JB ? (long long)I * JB + lj : (long long)J * JB + lj - JB;
    A[li * LD + lj] = G[gi * P.npad + gj];
    Q[li * LD + lj] = cmk<CT>(li == lj ? 1 : 0, 0);
  }
  for (int e = threadIdx.x; e < NBLK; e += blockDim.x) {
    int a = 0, t = e;
    while (t >= JB - a) { t -= JB - a; a++; }
    blk[e] = (unsigned short)(a | ((a + t) << 8));
  }
  const R eps_r = sizeof(R) == 4 ? (R)FLT_EPSILON : (R)DBL_EPSILON;
  const R floor_abs = (R)((double)eps_r * (*P.scale) * P.floor_factor);
  const R rel_skip = P.rel_skip > 0 ? (R)P.rel_skip : (R)4;
  const R move_abs = (R)(P.move_rel * (*P.scale));
  const bool track_move = P.move_tol > 0;   // the solve's moved-weight stopping rule
  // ONE_PAIR (problems of one block pair, the whole matrix): past the
  // eigen-dimension every row and column is zero and every rotation there is
  // skipped, so the problem pairs only its first DE indices (DE - 1 rounds
  // per sweep instead of D - 1).  The other pair slots hold identity
  // rotations on disjoint padded pairs, and the blocks and Q columns they
  // touch are left as they are.
  const int DE = (ONE_PAIR && P.nact > 0) ? min(D, max(2, (P.nact + 1) & ~1)) : D, DH = DE / 2;
  __syncthreads();
  int total = 0, total_sig = 0;
  const int max_sweeps = P.nb == 2 ? EigCfg<R>::MAXS : 1;
  // rotations of round r (the first JB lanes of warp 0)
  auto params = [&](int r) {
    if (threadIdx.x < JB) {
      int p, q;
      R c, s; CT e; bool skip, sig;
      if (!ONE_PAIR || (int)threadIdx.x < DH) {
        circle(r, threadIdx.x, DE, p, q);
        jrot_params<R>(A[p * LD + p].x, A[q * LD + q].x, A[p * LD + q], floor_abs, rel_skip, c, s, e, skip, sig);
      } else {
        p = DE + 2 * ((int)threadIdx.x - DH);
        q = p + 1;
        skip = true; sig = false; c = 1; s = 0; e = cmk<CT>(1, 0);
      }
      R mv = 0;   // the weight the rotation moves between p and q, |t g| (t = s / c)
      if (sig && move_abs > 0) {
        const CT g = A[p * LD + q];
        const R sg = fabs(s) * sqrt(g.x * g.x + g.y * g.y);
        if (!(sg > move_abs * c)) sig = false;
        else if (track_move) mv = sg / c;
      }
      if (cut) {
        const int gp = p < JB ? I * JB + p : J * JB + p - JB;
        const int gq = q < JB ? I * JB + q : J * JB + q - JB;
        if ((gp < P.cut_lo && gq < P.cut_lo) || (gp >= P.cut_hi && gq >= P.cut_hi)) {
          skip = true; sig = false; c = 1; s = 0; e = cmk<CT>(1, 0);
        }
      }
      const int o = threadIdx.x;
      pp[o] = p; pq[o] = q;
      tu[o] = s / ((R)1 + c); sn[o] = s; ph[o] = e;
      // rotation counters (and the moved weight): one shared-memory update
      // per round, by lane 0
      const unsigned mr = __ballot_sync(PMASK, !skip), ms = __ballot_sync(PMASK, sig);
      if (track_move) {
        R mw = sig ? mv : (R)0;
#pragma unroll
        for (int o = JB / 2; o > 0; o >>= 1) mw += __shfl_xor_sync(PMASK, mw, o);
        if (threadIdx.x == 0) nmove += mw;
      }
      if (threadIdx.x == 0) { nrot += __popc(mr); nsig += __popc(ms); }
    }
  };
  double last_move = 0.0;
  for (int sweep = 0; sweep < max_sweeps; sweep++) {
    if (threadIdx.x == 0) { nrot = 0; nsig = 0; nmove = 0; }
    __syncthreads();
    for (int r = 0; r < DE - 1; r++) {
      params(r);
      __syncthreads();
      // A <- R^H A R and Q <- Q R, every rotation in Rutishauser's form
      //   x' = x - s (y + tau x),  y' = y + s (x - tau y),  tau = s / (1 + c):
      // for small angles c = 1 - s tau is not rounded to 1, which would grow
      // every vector by (1 + t^2) per rotation in FP32.  The rotations of a
      // round act on disjoint pairs, so the 2 x 2 block of A on pairs (a, b)
      // becomes R_a^H B R_b by itself: one thread per block with a <= b, the
      // block below the diagonal is its conjugate transpose (A stays Hermitian).
      // Every element a thread touches in a round is its own, so all of its
      // loads (A blocks, Q pairs) are issued before any arithmetic or store.
      int bab[NB_T];   // pair slots of the thread's blocks, a | b << 8 (a <= b)
      CT x00[NB_T], x10[NB_T], x01[NB_T], x11[NB_T];
#pragma unroll
      for (int u = 0; u < NB_T; u++) {
        const int e = threadIdx.x + 256 * u;
        bab[u] = e < NBLK ? blk[e] : 0;
        const int a = bab[u] & 0xff, b = bab[u] >> 8;
        if (ONE_PAIR && b >= DH) continue;   // an identity slot: the block stays as it is
        const int pa = pp[a], qa = pq[a], pb = pp[b], qb = pq[b];
        x00[u] = A[pa * LD + pb]; x10[u] = A[qa * LD + pb];
        x01[u] = A[pa * LD + qb]; x11[u] = A[qa * LD + qb];
      }
      const int kq = threadIdx.x % JB, row0 = threadIdx.x / JB;
      const int cp = pp[kq], cq = pq[kq];
      const bool qrot = !ONE_PAIR || kq < DH;
      CT xq[QROWS], yq[QROWS];
#pragma unroll
      for (int j = 0; j < QROWS; j++) {
        const int row = row0 + j * QSTEP;
        if (qrot) {
          xq[j] = Q[row * LD + cp];
          yq[j] = Q[row * LD + cq];
        }
      }
#pragma unroll
      for (int u = 0; u < NB_T; u++) {
        const int a = bab[u] & 0xff, b = bab[u] >> 8;
        if (threadIdx.x + 256 * u >= NBLK || (ONE_PAIR && b >= DH)) continue;
        const int pa = pp[a], qa = pq[a], pb = pp[b], qb = pq[b];
        const R tb = tu[b], sb = sn[b];
        const CT fb = ph[b];
        const CT y0 = cmul(x01[u], fb), y1 = cmul(x11[u], fb);
        const CT n00 = cmk<CT>(x00[u].x - sb * (y0.x + tb * x00[u].x), x00[u].y - sb * (y0.y + tb * x00[u].y));
        const CT n01 = cmk<CT>(y0.x + sb * (x00[u].x - tb * y0.x), y0.y + sb * (x00[u].y - tb * y0.y));
        const CT n10 = cmk<CT>(x10[u].x - sb * (y1.x + tb * x10[u].x), x10[u].y - sb * (y1.y + tb * x10[u].y));
        const CT n11 = cmk<CT>(y1.x + sb * (x10[u].x - tb * y1.x), y1.y + sb * (x10[u].y - tb * y1.y));
        const R ta = tu[a], sa = sn[a];
        const CT fa = cconj(ph[a]);
        const CT z0 = cmul(n10, fa), z1 = cmul(n11, fa);
        const CT m00 = cmk<CT>(n00.x - sa * (z0.x + ta * n00.x), n00.y - sa * (z0.y + ta * n00.y));
        const CT m10 = cmk<CT>(z0.x + sa * (n00.x - ta * z0.x), z0.y + sa * (n00.y - ta * z0.y));
        const CT m01 = cmk<CT>(n01.x - sa * (z1.x + ta * n01.x), n01.y - sa * (z1.y + ta * n01.y));
        const CT m11 = cmk<CT>(z1.x + sa * (n01.x - ta * z1.x), z1.y + sa * (n01.y - ta * z1.y));
        A[pa * LD + pb] = m00; A[pa * LD + qb] = m01;
        A[qa * LD + pb] = m10; A[qa * LD + qb] = m11;
        if (a != b) {
          A[pb * LD + pa] = cconj(m00); A[qb * LD + pa] = cconj(m01);
          A[pb * LD + qa] = cconj(m10); A[qb * LD + qa] = cconj(m11);
        }
      }
      if (qrot) {
        const R t = tu[kq], s = sn[kq];
        const CT f = ph[kq];
#pragma unroll
        for (int j = 0; j < QROWS; j++) {
          const int row = row0 + j * QSTEP;
          const CT x = xq[j], y = cmul(yq[j], f);
          Q[row * LD + cp] = cmk<CT>(x.x - s * (y.x + t * x.x), x.y - s * (y.y + t * x.y));
          Q[row * LD + cq] = cmk<CT>(y.x + s * (x.x - t * y.x), y.y + s * (x.y - t * y.y));
        }
      }
      __syncthreads();
    }
    const int nr = nrot;
    total += nr;
    total_sig += nsig;
    last_move = (double)nmove;
    __syncthreads();
    if (nr == 0) break;
  }
  // no rotation at all leaves Q exactly the identity: flag it so that the
  // apply step skips the multiply (and J need not be written)
  if (P.jflag && threadIdx.x == 0) P.jflag[blockIdx.x] = total > 0;
  if (!P.jflag || total > 0) {
    CT* Jo = (CT*)P.J + (long long)blockIdx.x * D * D;
    for (int e = threadIdx.x; e < D * D; e += blockDim.x) Jo[e] = Q[(e / D) * LD + (e % D)];
  }
  if (threadIdx.x == 0 && total > 0) {
    atomicAdd(P.off, (double)total_sig);
    atomicAdd(P.off + 1, (double)total);
    if (P.mv) P.mv[blockIdx.x] += last_move;   // of the block pair's last inner sweep; one writer per slot
  }
}

template <typename R>
__global__ void __launch_bounds__(256) k_eig_apply(const EigProb* __restrict__ probs, int round) {
  using CT = typename C2<R>::T;
  constexpr int JB = EigCfg<R>::JB, D = 2 * JB, LD = D + 1, PER = D / 16;
  const EigProb P = probs[blockIdx.y];
  if (!P.active || round >= P.nb - 1) return;
  const int h = P.nb / 2, nG = h * (h + 1) / 2, nV = h * h;
  const int tile = blockIdx.x;
  if (tile >= nG + nV) return;
  extern __shared__ unsigned char smraw[];
  CT* S0 = reinterpret_cast<CT*>(smraw);
  CT* S1 = S0 + D * LD;
  const bool isG = tile < nG;
  int Pp, Qp;
  if (isG) {   // upper-triangular pair index (Pp <= Qp); G is Hermitian
    int t = tile, row = 0;
    while (t >= h - row) { t -= h - row; row++; }
    Pp = row;
    Qp = row + t;
  } else {
    Pp = (tile - nG) / h;
    Qp = (tile - nG) % h;
  }
  // tiles whose rotations are all the identity are left as they are
  const bool fq = !P.jflag || P.jflag[Qp], fp = isG && (!P.jflag || P.jflag[Pp]);
  if (!fq && !fp) return;
  if (P.jflag && threadIdx.x == 0)
    atomicAdd(P.off + 2, 8.0 * D * D * D * ((fq ? 1 : 0) + (fp ? 1 : 0)));
  int K1, K2, I1 = 0, I2 = 0;
  circle(round, Qp, P.nb, K1, K2);
  if (isG) circle(round, Pp, P.nb, I1, I2);
  CT* X = (CT*)(isG ? P.G : P.V);
  const CT* Jb = (const CT*)P.J;
  auto grow = [&](int li) -> long long {
    if (!isG) return (long long)Pp * D + li;
    return li < JB ? (long long)I1 * JB + li : (long long)I2 * JB + li - JB;
  };
  auto gcol = [&](int lj) -> long long {
    return lj < JB ? (long long)K1 * JB + lj : (long long)K2 * JB + lj - JB;
  };
  for (int e = threadIdx.x; e < D * D; e += blockDim.x) {
    const int li = e / D, lj = e % D;
    S0[li * LD + lj] = X[grow(li) * P.npad + gcol(lj)];
    if (fq) S1[li * LD + lj] = Jb[(long long)Qp * D * D + e];
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  CT acc[PER][PER];
#pragma unroll
  for (int i = 0; i < PER; i++)
#pragma unroll
    for (int j = 0; j < PER; j++) acc[i][j] = fq ? cmk<CT>(0, 0) : S0[(ty + 16 * i) * LD + tx + 16 * j];
  if (fq) for (int k = 0; k < D; k++) {  // T = X_tile * J_Q
    CT a[PER], b[PER];
#pragma unroll
    for (int i = 0; i < PER; i++) a[i] = S0[(ty + 16 * i) * LD + k];
#pragma unroll
    for (int j = 0; j < PER; j++) b[j] = S1[k * LD + tx + 16 * j];
#pragma unroll
    for (int i = 0; i < PER; i++)
#pragma unroll
      for (int j = 0; j < PER; j++) cfma(acc[i][j], a[i], b[j]);
  }
  if (!isG) {
#pragma unroll
    for (int i = 0; i < PER; i++)
#pragma unroll
      for (int j = 0; j < PER; j++)
        X[grow(ty + 16 * i) * P.npad + gcol(tx + 16 * j)] = acc[i][j];
    return;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < PER; i++)
#pragma unroll
    for (int j = 0; j < PER; j++) S0[(ty + 16 * i) * LD + tx + 16 * j] = acc[i][j];
  if (fp)
    for (int e = threadIdx.x; e < D * D; e += blockDim.x)
      S1[(e / D) * LD + (e % D)] = Jb[(long long)Pp * D * D + e];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < PER; i++)
#pragma unroll
    for (int j = 0; j < PER; j++) acc[i][j] = fp ? cmk<CT>(0, 0) : S0[(ty + 16 * i) * LD + tx + 16 * j];
  if (fp) for (int k = 0; k < D; k++) {  // Y = J_P^H * T
    CT a[PER], b[PER];
#pragma unroll
    for (int i = 0; i < PER; i++) a[i] = cconj(S1[k * LD + ty + 16 * i]);
#pragma unroll
    for (int j = 0; j < PER; j++) b[j] = S0[k * LD + tx + 16 * j];
#pragma unroll
    for (int i = 0; i < PER; i++)
#pragma unroll
      for (int j = 0; j < PER; j++) cfma(acc[i][j], a[i], b[j]);
  }
  __syncthreads();   // all reads of S0 / S1 done
#pragma unroll
  for (int i = 0; i < PER; i++)
#pragma unroll
    for (int j = 0; j < PER; j++) S0[(ty + 16 * i) * LD + tx + 16 * j] = acc[i][j];
  __syncthreads();
  for (int e = threadIdx.x; e < D * D; e += blockDim.x) {
    const int li = e / D, lj = e % D;
    X[grow(li) * P.npad + gcol(lj)] = S0[li * LD + lj];
  }
  if (Pp != Qp) {   // Hermitian mirror tile (Q, P), written row by row
    for (int e = threadIdx.x; e < D * D; e += blockDim.x) {
      const int li = e / D, lj = e % D;
      X[gcol(li) * P.npad + grow(lj)] = cconj(S0[lj * LD + li]);
    }
  }
}

// FP32 apply, one 64 x 64 complex tile per CTA of 128 threads.  Each thread
// owns 8 rows x 4 columns of the tile: rows 16 w + rg + 2 i (warp w, half-warp
// rg, i < 8) and columns 4 cg .. 4 cg + 3 (cg = lane mod 16), so a k step
// reads 8 broadcast values of the left operand and two 16-byte vectors of the
// right one for 32 complex multiply-adds.  Tiles arrive by 16-byte cp.async
// copies into rows padded to 66 elements (16-byte aligned, and the two
// half-warps' rows fall in different banks); J_P is fetched while T is
// written back.  By default (APPLY_GAUSS) each complex multiply-add takes
// three real FMAs (Gauss's product) instead of four, applied to J - I.
#ifndef APPLY_GAUSS
#define APPLY_GAUSS 1
#endif
namespace {
constexpr int AP_D = 64, AP_LD = 66, AP_THREADS = 128;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_all;\n" ::: "memory");
}
}  // namespace

template <bool GAUSS>
__global__ void __launch_bounds__(AP_THREADS, 3) k_eig_apply_f32(const EigProb* __restrict__ probs, int round) {
  constexpr int JB = 32, D = AP_D, LD = AP_LD;
  const EigProb P = probs[blockIdx.y];
  if (!P.active || round >= P.nb - 1) return;
  const int h = P.nb / 2, nG = h * (h + 1) / 2, nV = h * h;
  const int tile = blockIdx.x;
  if (tile >= nG + nV) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* S0 = reinterpret_cast<float2*>(smraw);
  float2* S1 = S0 + D * LD;
  const bool isG = tile < nG;
  int Pp, Qp;
  if (isG) {
    int t = tile, row = 0;
    while (t >= h - row) { t -= h - row; row++; }
    Pp = row;
    Qp = row + t;
  } else {
    Pp = (tile - nG) / h;
    Qp = (tile - nG) % h;
  }
  const bool fq = !P.jflag || P.jflag[Qp], fp = isG && (!P.jflag || P.jflag[Pp]);
  if (!fq && !fp) return;
  if (P.jflag && threadIdx.x == 0)
    atomicAdd(P.off + 2, 8.0 * D * D * D * ((fq ? 1 : 0) + (fp ? 1 : 0)));
  int K1, K2, I1 = 0, I2 = 0;
  circle(round, Qp, P.nb, K1, K2);
  if (isG) circle(round, Pp, P.nb, I1, I2);
  float2* X = reinterpret_cast<float2*>(isG ? P.G : P.V);
  const float2* Jb = reinterpret_cast<const float2*>(P.J);
  const long long np = P.npad;
  auto grow = [&](int li) -> long long {
    if (!isG) return (long long)Pp * D + li;
    return li < JB ? (long long)I1 * JB + li : (long long)I2 * JB + li - JB;
  };
  auto gcol = [&](int lj) -> long long {
    return lj < JB ? (long long)K1 * JB + lj : (long long)K2 * JB + lj - JB;
  };
  const int t = threadIdx.x;
  for (int c = t; c < D * (D / 2); c += AP_THREADS) {   // 16-byte chunks: 2 complex
    const int li = c >> 5, lj = (c & 31) * 2;
    cp_async16(S0 + li * LD + lj, X + grow(li) * np + gcol(lj));
    if (fq) cp_async16(S1 + li * LD + lj, Jb + (long long)Qp * D * D + li * D + lj);
  }
  cp_async_wait_all();
  __syncthreads();
  if (GAUSS && fq) {   // J_Q - I: the product runs in the form X + X (J - I)
    if (t < D) S1[t * LD + t].x -= 1.f;
    __syncthreads();
  }
  const int w = t >> 5, lane = t & 31, rg = lane >> 4, cg = lane & 15;
  const int r0 = 16 * w + rg, c0 = 4 * cg;
  float2 acc[8][4];
  // out = base + A B over k < 64, thread block 8 rows x 4 columns.  GAUSS:
  // three real products per complex multiply-add -- t1 = sum ax bx, t2 =
  // sum ay by, t3 = sum (ax + ay)(bx + by); re = t1 - t2, im = t3 - t1 - t2 --
  // with A B = X (J - I), whose rounding scales with |J - I|; otherwise the
  // four-product complex FMA of A B = X J.
  auto product = [&](auto loadA, auto loadB, const float2* base) {
    if constexpr (GAUSS) {
      float t1[8][4], t2[8][4], t3[8][4];
#pragma unroll
      for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) t1[i][j] = t2[i][j] = t3[i][j] = 0.f;
#pragma unroll 2
      for (int k = 0; k < D; k++) {
        float2 a[8], b[4];
        float as[8], bs[4];
        loadA(k, a);
        loadB(k, b);
#pragma unroll
        for (int i = 0; i < 8; i++) as[i] = a[i].x + a[i].y;
#pragma unroll
        for (int j = 0; j < 4; j++) bs[j] = b[j].x + b[j].y;
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) {
            t1[i][j] = fmaf(a[i].x, b[j].x, t1[i][j]);
            t2[i][j] = fmaf(a[i].y, b[j].y, t2[i][j]);
            t3[i][j] = fmaf(as[i], bs[j], t3[i][j]);
          }
      }
#pragma unroll
      for (int i = 0; i < 8; i++) {            // base row: two 16-byte loads
        const float4 x01 = *reinterpret_cast<const float4*>(base + (r0 + 2 * i) * LD + c0);
        const float4 x23 = *reinterpret_cast<const float4*>(base + (r0 + 2 * i) * LD + c0 + 2);
        const float2 x[4] = {make_float2(x01.x, x01.y), make_float2(x01.z, x01.w), make_float2(x23.x, x23.y),
                             make_float2(x23.z, x23.w)};
#pragma unroll
        for (int j = 0; j < 4; j++)
          acc[i][j] = make_float2(x[j].x + (t1[i][j] - t2[i][j]), x[j].y + ((t3[i][j] - t1[i][j]) - t2[i][j]));
      }
    } else {
      (void)base;
#pragma unroll
      for (int i = 0; i < 8; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 2
      for (int k = 0; k < D; k++) {
        float2 a[8], b[4];
        loadA(k, a);
        loadB(k, b);
#pragma unroll
        for (int i = 0; i < 8; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) cfma(acc[i][j], a[i], b[j]);
      }
    }
  };
  auto rowsB = [&](const float2* Sb) {   // row k of B, columns c0 .. c0 + 3, two 16-byte loads
    return [=](int k, float2 (&b)[4]) {
      const float4 b01 = *reinterpret_cast<const float4*>(Sb + k * LD + c0);
      const float4 b23 = *reinterpret_cast<const float4*>(Sb + k * LD + c0 + 2);
      b[0] = make_float2(b01.x, b01.y); b[1] = make_float2(b01.z, b01.w);
      b[2] = make_float2(b23.x, b23.y); b[3] = make_float2(b23.z, b23.w);
    };
  };
  if (fq) {                                    // T = X_tile J_Q
    product([&](int k, float2 (&a)[8]) {
#pragma unroll
              for (int i = 0; i < 8; i++) a[i] = S0[(r0 + 2 * i) * LD + k];
            },
            rowsB(S1), S0);
  } else {
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) acc[i][j] = S0[(r0 + 2 * i) * LD + c0 + j];
  }
  if (isG) {
    __syncthreads();                           // every read of S0 and S1 is done
    if (fp) {
      for (int c = t; c < D * (D / 2); c += AP_THREADS) {
        const int li = c >> 5, lj = (c & 31) * 2;
        cp_async16(S1 + li * LD + lj, Jb + (long long)Pp * D * D + li * D + lj);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {              // T -> S0
      float4* dst = reinterpret_cast<float4*>(S0 + (r0 + 2 * i) * LD + c0);
      dst[0] = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
      dst[1] = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
    }
    cp_async_wait_all();
    __syncthreads();
    if (GAUSS && fp) {                         // J_P - I
      if (t < D) S1[t * LD + t].x -= 1.f;
      __syncthreads();
    }
    if (fp) {                                  // Y = J_P^H T
      product([&](int k, float2 (&a)[8]) {
#pragma unroll
                for (int i = 0; i < 8; i++) a[i] = cconj(S1[k * LD + r0 + 2 * i]);
              },
              rowsB(S0), S0);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; i++) {                // the tile, 32 bytes per thread and row
    float4* dst = reinterpret_cast<float4*>(X + grow(r0 + 2 * i) * np + gcol(c0));
    dst[0] = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
    dst[1] = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
  }
  if (isG && Pp != Qp) {                       // Hermitian mirror tile (Q, P), row by row
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) S0[(r0 + 2 * i) * LD + c0 + j] = acc[i][j];
    __syncthreads();
    for (int e = t; e < D * D; e += AP_THREADS) {
      const int li = e / D, lj = e % D;
      X[gcol(li) * np + grow(lj)] = cconj(S0[lj * LD + li]);
    }
  }
}

template <typename R>
__global__ void k_eig_init(const EigProb* __restrict__ probs, int max_npad) {
  using CT = typename C2<R>::T;
  const EigProb P = probs[blockIdx.y];
  const long long n2 = (long long)P.npad * P.npad;
  CT* V = (CT*)P.V;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n2;
       e += (long long)gridDim.x * blockDim.x) {
    const long long i = e / P.npad, j = e % P.npad;
    V[e] = cmk<CT>(i == j ? 1 : 0, 0);
  }
}

template <typename R>
__global__ void k_eig_trace(const EigProb* __restrict__ probs) {
  using CT = typename C2<R>::T;
  const EigProb P = probs[blockIdx.x];
  const CT* G = (const CT*)P.G;
  double acc = 0;
  for (int i = threadIdx.x; i < P.npad; i += blockDim.x) acc += fabs((double)G[(long long)i * P.npad + i].x);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += part[w];
    *const_cast<double*>(P.scale) = t;
  }
}

template <typename R>
cudaError_t launch_eig_trace(const EigProb* d_probs, int n_probs, cudaStream_t s) {
  if (n_probs <= 0) return cudaSuccess;
  k_eig_trace<R><<<n_probs, 256, 0, s>>>(d_probs);
  return cudaGetLastError();
}
template cudaError_t launch_eig_trace<float>(const EigProb*, int, cudaStream_t);
template cudaError_t launch_eig_trace<double>(const EigProb*, int, cudaStream_t);

template <typename R>
cudaError_t launch_eig_init(const EigProb* d_probs, int n_probs, int max_npad, cudaStream_t s) {
  if (n_probs <= 0) return cudaSuccess;
  long long n2 = (long long)max_npad * max_npad;
  unsigned gx = (unsigned)((n2 + 255) / 256);
  if (gx > 4096) gx = 4096;
  k_eig_init<R><<<dim3(gx, n_probs), 256, 0, s>>>(d_probs, max_npad);
  return cudaGetLastError();
}

template <typename R>
static void eig_attrs() {
  using CT = typename C2<R>::T;
  constexpr int JB = EigCfg<R>::JB, D = 2 * JB, LD = D + 1;
  static bool attr = false;
  if (attr) return;
  const size_t sm_inner = 2 * sizeof(CT) * D * LD + JB * (2 * sizeof(R) + sizeof(CT) + 2 * sizeof(int)) +
                          sizeof(unsigned short) * JB * (JB + 1) / 2;
  const size_t sm_apply = 2 * sizeof(CT) * D * LD;
  cudaFuncSetAttribute(k_eig_inner<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_inner);
  cudaFuncSetAttribute(k_eig_inner<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_inner);
  cudaFuncSetAttribute(k_eig_apply<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm_apply);
  attr = true;
}

template <typename R>
cudaError_t launch_eig_inner(const EigProb* d_probs, int n_probs, int max_nb, int round, cudaStream_t s) {
  using CT = typename C2<R>::T;
  constexpr int JB = EigCfg<R>::JB, D = 2 * JB, LD = D + 1;
  eig_attrs<R>();
  const size_t sm_inner = 2 * sizeof(CT) * D * LD + JB * (2 * sizeof(R) + sizeof(CT) + 2 * sizeof(int)) +
                          sizeof(unsigned short) * JB * (JB + 1) / 2;
  // problems of one block pair (nb == 2) have a single round, the first; the
  // others run the general variant
  if (max_nb > 2) {
    k_eig_inner<R, false><<<dim3(max_nb / 2, n_probs), 256, sm_inner, s>>>(d_probs, round);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (round == 0) k_eig_inner<R, true><<<dim3(1, n_probs), 256, sm_inner, s>>>(d_probs, round);
  return cudaGetLastError();
}

int eig_inner_launches(int max_nb, int round) { return (max_nb > 2 ? 1 : 0) + (round == 0 ? 1 : 0); }

template <typename R>
cudaError_t launch_eig_apply(const EigProb* d_probs, int n_probs, int max_nb, int round, cudaStream_t s) {
  using CT = typename C2<R>::T;
  constexpr int JB = EigCfg<R>::JB, D = 2 * JB, LD = D + 1;
  eig_attrs<R>();
  const int h = max_nb / 2;
  if constexpr (sizeof(R) == 4) {
    static_assert(D == AP_D, "FP32 apply tile");
    const size_t sm = 2 * sizeof(float2) * AP_D * AP_LD;
    eig_prepare(false);
    k_eig_apply_f32<APPLY_GAUSS != 0><<<dim3(h * (h + 1) / 2 + h * h, n_probs), AP_THREADS, sm, s>>>(d_probs, round);
  } else {
    const size_t sm_apply = 2 * sizeof(CT) * D * LD;
    k_eig_apply<R><<<dim3(h * (h + 1) / 2 + h * h, n_probs), 256, sm_apply, s>>>(d_probs, round);
  }
  return cudaGetLastError();
}

cudaError_t eig_prepare(bool fp64) {
  if (fp64) {
    eig_attrs<double>();
  } else {
    eig_attrs<float>();
    static bool attr = false;
    if (!attr) {
      const size_t sm = 2 * sizeof(float2) * AP_D * AP_LD;
      cudaFuncSetAttribute(k_eig_apply_f32<APPLY_GAUSS != 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      attr = true;
    }
  }
  return cudaGetLastError();
}

// One thread walks the problems (a few hundred at most per batch).  With a
// compact array, the problems still active after the sweep are also copied
// there when they fit (the copies point at the same buffers and counters),
// and *mode tells the next sweep which chain of launches to run.
__global__ void k_sweep_end(EigProb* __restrict__ probs, int n, double* __restrict__ cum,
                            double* __restrict__ n_sweeps, int max_sweeps, cudaGraphConditionalHandle h,
                            EigProb* __restrict__ compact, int compact_cap, int* __restrict__ mode) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  bool any = false;
  int n_active = 0;
  for (int i = 0; i < n; i++) {
    EigProb& P = probs[i];
    if (!P.active) continue;
    cum[4 * i] += P.off[1];
    cum[4 * i + 1] += P.off[2];
    cum[4 * i + 2] += 1.0;
    double mw = 0;   // the sweep's moved weight, summed in slot order
    if (P.mv)
      for (int k = 0; k < P.nb / 2; k++) { mw += P.mv[k]; P.mv[k] = 0.0; }
    const double moved = mw / (*P.scale), before = cum[4 * i + 3];
    cum[4 * i + 3] = moved;   // weight the last sweep moved, relative to the trace
    // skipped rotations inside the cut's classes leave couplings that rotations
    // across the cut keep renewing: where the moved weight stalls, rotate every
    // pair from now on
    if (P.cut_hi > 0 && P.move_tol > 0 && cum[4 * i + 2] >= 6.0 && moved > 0.9 * before) P.cut_hi = 0;
    const bool settled = P.move_tol > 0 && moved <= P.move_tol;
    if (P.off[0] == 0.0 || settled) P.active = 0; else { any = true; n_active++; }
    P.off[0] = 0.0; P.off[1] = 0.0; P.off[2] = 0.0;
  }
  *n_sweeps += 1.0;
  if (compact) {
    const bool fit = n_active <= compact_cap;
    if (fit) {
      int c = 0;
      for (int i = 0; i < n; i++)
        if (probs[i].active) compact[c++] = probs[i];
      for (; c < compact_cap; c++) compact[c].active = 0;
    }
    *mode = fit ? 1 : 0;
  }
  cudaGraphSetConditional(h, (any && *n_sweeps < (double)max_sweeps) ? 1u : 0u);
}

// First node of a device-side sweep: run the compact chain (mode 1) or the
// full one (mode 0).
__global__ void k_sweep_begin(const int* __restrict__ mode, cudaGraphConditionalHandle h_compact,
                              cudaGraphConditionalHandle h_full) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const unsigned m = *mode != 0 ? 1u : 0u;
  cudaGraphSetConditional(h_compact, m);
  cudaGraphSetConditional(h_full, 1u - m);
}

cudaError_t launch_sweep_end(EigProb* d_probs, int n, double* cum, double* n_sweeps, int max_sweeps,
                             cudaGraphConditionalHandle h, EigProb* compact, int compact_cap, int* mode,
                             cudaStream_t s) {
  k_sweep_end<<<1, 32, 0, s>>>(d_probs, n, cum, n_sweeps, max_sweeps, h, compact, compact_cap, mode);
  return cudaGetLastError();
}

cudaError_t launch_sweep_begin(const int* mode, cudaGraphConditionalHandle h_compact,
                               cudaGraphConditionalHandle h_full, cudaStream_t s) {
  k_sweep_begin<<<1, 32, 0, s>>>(mode, h_compact, h_full);
  return cudaGetLastError();
}

template cudaError_t launch_eig_init<float>(const EigProb*, int, int, cudaStream_t);
template cudaError_t launch_eig_init<double>(const EigProb*, int, int, cudaStream_t);
template cudaError_t launch_eig_inner<float>(const EigProb*, int, int, int, cudaStream_t);
template cudaError_t launch_eig_inner<double>(const EigProb*, int, int, int, cudaStream_t);
template cudaError_t launch_eig_apply<float>(const EigProb*, int, int, int, cudaStream_t);
template cudaError_t launch_eig_apply<double>(const EigProb*, int, int, int, cudaStream_t);

// ---------------------------------------------------------------------------
// Weighted column norms rho_i = sum_row lambda_L[row >> shift]^2 |R[row][i]|^2
// in FP64: the Schmidt weight carried by direction i (Eq. 4 terms).
// ---------------------------------------------------------------------------
// One CTA of 256 threads per 32 columns: warp w sums rows w, w + 8, ... of
// its lane's column (a warp reads 32 consecutive elements of a row), then the
// eight partial sums are added in a fixed order -- the result does not depend
// on the order in which CTAs run (ties between weights decide the sort order
// of the directions, so rho must be reproducible bit for bit).
constexpr int CN_COLS = 32, CN_WARPS = 8;

template <typename R>
__global__ void __launch_bounds__(CN_COLS * CN_WARPS) k_colnorm(
    const void* const* __restrict__ Rs, const int* __restrict__ ms, const int* __restrict__ ns,
    const int* __restrict__ lds, const double* const* __restrict__ lams, const int* __restrict__ shifts,
    double* const* __restrict__ rhos) {
  using CT = typename C2<R>::T;
  __shared__ double part[CN_WARPS][CN_COLS];
  const int p = blockIdx.y;
  const int n = ns[p], m = ms[p];
  const int c0 = blockIdx.x * CN_COLS;
  if (c0 >= n) return;
  const long long ld = lds ? lds[p] : n;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = c0 + lane;
  const CT* Rm = (const CT*)Rs[p];
  const double* lam = lams[p];
  const int sh = shifts[p];
  double acc = 0;
  if (c < n)
    for (int r = w; r < m; r += CN_WARPS) {
      const CT v = Rm[(long long)r * ld + c];
      const double wt = lam ? lam[r >> sh] : 1.0;
      acc += wt * wt * ((double)v.x * v.x + (double)v.y * v.y);
    }
  part[w][lane] = acc;
  __syncthreads();
  if (w == 0 && c < n) {
    double t = 0;
#pragma unroll
    for (int k = 0; k < CN_WARPS; k++) t += part[k][lane];
    rhos[p][c] = t;
  }
}

template <typename R>
cudaError_t launch_colnorm_batch(const void* const* d_R, const int* d_m, const int* d_n, const int* d_ld,
                                 const double* const* d_lam, const int* d_shift,
                                 double* const* d_rho, int n_probs, int max_n, int max_m,
                                 cudaStream_t s) {
  if (n_probs <= 0) return cudaSuccess;
  (void)max_m;
  dim3 grid((max_n + CN_COLS - 1) / CN_COLS, n_probs);
  k_colnorm<R><<<grid, CN_COLS * CN_WARPS, 0, s>>>(d_R, d_m, d_n, d_ld, d_lam, d_shift, d_rho);
  return cudaGetLastError();
}
template cudaError_t launch_colnorm_batch<float>(const void* const*, const int*, const int*, const int*,
                                                 const double* const*, const int*,
                                                 double* const*, int, int, int, cudaStream_t);
template cudaError_t launch_colnorm_batch<double>(const void* const*, const int*, const int*, const int*,
                                                  const double* const*, const int*,
                                                  double* const*, int, int, int, cudaStream_t);

// The accumulated rotations V are orthonormal only to rounding: the weight of
// direction i is rho_i / |v_i|^2, and the site row / remainder column it
// yields is scaled by 1 / |v_i|.  rho_i <- rho_i / vn_i, vn_i <- 1 / sqrt(vn_i).
__global__ void k_rho_normalize(double* const* __restrict__ rhos, double* const* __restrict__ vns,
                                const int* __restrict__ ns) {
  const int p = blockIdx.y;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ns[p]) return;
  const double v = vns[p][i];
  if (v > 0) {
    rhos[p][i] /= v;
    vns[p][i] = 1.0 / sqrt(v);
  } else {
    vns[p][i] = 1.0;
  }
}

cudaError_t launch_rho_normalize(double* const* d_rho, double* const* d_vn, const int* d_n, int n_probs,
                                 int max_n, cudaStream_t s) {
  if (n_probs <= 0 || max_n <= 0) return cudaSuccess;
  k_rho_normalize<<<dim3((max_n + 255) / 256, n_probs), 256, 0, s>>>(d_rho, d_vn, d_n);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Truncation (Sec. II.B): sort the weights descending, keep the smallest r
// whose discarded weight is <= cutoff * total, drop numerical zeros
// (rho <= floor2 * rho_max), keep no more than the matrix's rank bound
// (rank_cap) and chi_max; f = kept / total (Eq. 4); the
// kept spectrum is renormalised to unit weight.
// ---------------------------------------------------------------------------
constexpr int SEL_MAX = 4096, SEL_T = 1024;

// doubles as integers of the same order (FP64 compares hold their unit for 64 cycles)
__device__ __forceinline__ unsigned long long sel_enc(double v) {
  const long long b = __double_as_longlong(v + 0.0);   // -0 as 0
  return (unsigned long long)(b < 0 ? ~b : b ^ (long long)0x8000000000000000ull);
}
__device__ __forceinline__ double sel_dec(unsigned long long u) {
  return __longlong_as_double((long long)(u >> 63 ? u ^ 0x8000000000000000ull : ~u));
}

// One CTA per problem: bitonic sort (strides below 32 stay within a warp: no
// block barrier), then suffix sums from the smallest weight on, by block scan.
// Bound by the latency of these stages; with the sums and the counts in loops
// of one thread, and FP64 compares, it took 0.31 ms at n = 1024 and 0.73 ms at
// 2048 (two steep problems); now 0.04 and 0.05.
__global__ void __launch_bounds__(SEL_T) k_select(const SelProb* __restrict__ probs, int chi_max,
                                                  double cutoff, double band, double resolved,
                                                  double floor2) {
  extern __shared__ unsigned char smraw[];
  unsigned long long* key = reinterpret_cast<unsigned long long*>(smraw);
  int* idx = reinterpret_cast<int*>(key + SEL_MAX);
  __shared__ double wsum_s[32], W_s;
  __shared__ int r_s, nz_s, lo_s, hi_s;
  const SelProb P = probs[blockIdx.x];
  const int n = P.n, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int np2 = 1;
  while (np2 < n) np2 <<= 1;
  for (int i = tid; i < np2; i += SEL_T) {
    key[i] = sel_enc(i < n ? P.rho[i] : -1.0);
    idx[i] = i;
  }
  if (tid == 0) { r_s = 1; nz_s = lo_s = hi_s = 0; }
  __syncthreads();
  for (int k = 2; k <= np2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < np2; i += SEL_T) {
        const int l = i ^ j;
        if (l > i) {
          // "before" = larger key, ties by smaller index
          const unsigned long long a = key[i], b = key[l];
          const int ia = idx[i], ib = idx[l];
          if ((a > b || (a == b && ia < ib)) == ((i & k) != 0)) {
            key[i] = b; key[l] = a;
            idx[i] = ib; idx[l] = ia;
          }
        }
      }
      if (max(j, j > 1 ? j >> 1 : k) >= 32) __syncthreads(); else __syncwarp();
    }
  }
  __syncthreads();
  // thread -> E neighbouring positions
  const int E = (np2 + SEL_T - 1) / SEL_T, i0 = tid * E;
  double v[SEL_MAX / SEL_T], raw[SEL_MAX / SEL_T], sum = 0;
#pragma unroll
  for (int e = SEL_MAX / SEL_T - 1; e >= 0; e--) {
    raw[e] = e < E && i0 + e < n ? sel_dec(key[i0 + e]) : 0.0;
    v[e] = raw[e] > 0 ? raw[e] : 0.0;
    sum += v[e];
  }
  double suf = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double x = __shfl_down_sync(0xffffffffu, suf, o);
    if (lane + o < 32) suf += x;
  }
  if (lane == 0) wsum_s[w] = suf;
  __syncthreads();
  if (w == 0) {                                  // weights behind each warp's positions
    double x = wsum_s[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_down_sync(0xffffffffu, x, o);
      if (lane + o < 32) x += y;
    }
    if (lane == 0) W_s = x;
    const double behind = __shfl_down_sync(0xffffffffu, x, 1);
    __syncwarp();
    wsum_s[lane] = lane < 31 ? behind : 0.0;
  }
  __syncthreads();
  const double inside = W_s;                     // weight inside the n directions
  double W = inside, outside = 0;                // weight outside the n directions (sketched split)
  if (P.W_ext && *P.W_ext > W) { outside = *P.W_ext - W; W = *P.W_ext; }
  const double top = sel_dec(key[0]);
  {
    double tail = __shfl_down_sync(0xffffffffu, suf, 1);
    tail = (lane < 31 ? tail : 0.0) + wsum_s[w] + outside;
    int r = 1, nz = 0;
#pragma unroll
    for (int e = SEL_MAX / SEL_T - 1; e >= 0; e--) {
      if (e >= E || i0 + e >= n) continue;
      tail += v[e];
      if (i0 + e >= 1 && r == 1 && tail > cutoff * W) r = i0 + e + 1;
      nz += raw[e] > floor2 * top ? 1 : 0;
    }
    r = __reduce_max_sync(0xffffffffu, r);
    nz = __reduce_add_sync(0xffffffffu, nz);
    if (lane == 0) {
      if (r > 1) atomicMax(&r_s, r);
      if (nz) atomicAdd(&nz_s, nz);
    }
  }
  __syncthreads();
  int r = cutoff > 0 ? r_s : n;
  if (nz_s < r) r = nz_s;
  if (P.rank_cap > 0 && r > P.rank_cap) r = P.rank_cap;   // rank(M) <= its row count
  if (r < 1) r = 1;
  const int uncapped = r;
  if (r > chi_max) r = chi_max;
  // the kept weight; directions whose weight is within band * W of the smallest kept one may still cross the cut:
  // [lo, hi) in the sorted order; kept directions below resolved * W are not resolved by the first pass either
  const double cut = sel_dec(key[r - 1]), d = band * W, above = fmax(cut + d, resolved * W), upto = cut - d;
  double kept = 0;
  int lo = 0, hi = 0;
#pragma unroll
  for (int e = SEL_MAX / SEL_T - 1; e >= 0; e--) {
    if (e >= E || i0 + e >= n) continue;
    if (i0 + e < r) kept += v[e];
    lo += raw[e] > above ? 1 : 0;
    hi += raw[e] >= upto ? 1 : 0;
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double x = __shfl_down_sync(0xffffffffu, kept, o);
    if (lane + o < 32) kept += x;
  }
  lo = __reduce_add_sync(0xffffffffu, lo);
  hi = __reduce_add_sync(0xffffffffu, hi);
  if (lane == 0) {
    wsum_s[w] = kept;                            // read by its own warp only since the last barrier
    if (lo) atomicAdd(&lo_s, lo);
    if (hi) atomicAdd(&hi_s, hi);
  }
  __syncthreads();
  if (w == 0) {
    double x = wsum_s[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double y = __shfl_down_sync(0xffffffffu, x, o);
      if (lane + o < 32) x += y;
    }
    if (lane == 0) {
      W_s = x;
      P.res[0] = r;
      P.res[1] = W > 0 ? fmin(x / W, 1.0) : 1.0;
      P.res[2] = W;
      P.res[3] = x;
      P.res[4] = uncapped;
      P.res[5] = inside;
      P.res[6] = lo_s;
      P.res[7] = hi_s;
    }
  }
  __syncthreads();
  kept = W_s;
  for (int i = tid; i < n; i += SEL_T) P.perm[i] = idx[i];
  for (int i = tid; i < r; i += SEL_T) P.lam_out[i] = kept > 0 ? sqrt(fmax(sel_dec(key[i]), 0.0) / kept) : 0.0;
}

cudaError_t launch_select(const SelProb* d_probs, int n_probs, int chi_max, double cutoff, double band,
                          double resolved, double floor2, cudaStream_t s) {
  if (n_probs <= 0) return cudaSuccess;
  const size_t sm = SEL_MAX * (sizeof(unsigned long long) + sizeof(int));
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_select, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    attr = true;
  }
  k_select<<<n_probs, SEL_T, sm, s>>>(d_probs, chi_max, cutoff, band, resolved, floor2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Write-back gathers: new right site B = (V_r)^dagger and the unweighted
// remainder Rbar_r = (Mbar V)[:, kept] / sqrt(kept weight).
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_gather(const GatherProb* __restrict__ probs) {
  using CT = typename C2<R>::T;
  const GatherProb P = probs[blockIdx.y];
  const long long tot = (long long)P.rows * P.r;
  const CT* src = (const CT*)P.src;
  CT* dst = (CT*)P.dst;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    if (P.mode == 0) {
      const int mu = (int)(e / P.rows), c = (int)(e % P.rows);
      const int j = P.perm[mu];
      const CT v = cconj(src[(long long)c * P.ld + j]);
      dst[e] = P.cs ? cscale(v, P.cs[j]) : v;
    } else {
      const long long row = e / P.r;
      const int mu = (int)(e % P.r);
      const int j = P.perm[mu];
      dst[e] = cscale(src[row * P.ld + j], P.cs ? P.scale * P.cs[j] : P.scale);
    }
  }
}

template <typename R>
cudaError_t launch_gather(const GatherProb* d_probs, int n_probs, long long max_elems,
                          cudaStream_t s) {
  if (n_probs <= 0 || max_elems <= 0) return cudaSuccess;
  long long gx = (max_elems + 255) / 256;
  if (gx > 65535) gx = 65535;
  k_gather<R><<<dim3((unsigned)gx, n_probs), 256, 0, s>>>(d_probs);
  return cudaGetLastError();
}
template cudaError_t launch_gather<float>(const GatherProb*, int, long long, cudaStream_t);
template cudaError_t launch_gather<double>(const GatherProb*, int, long long, cudaStream_t);

// The cluster unitary on small clusters (D = 2^k <= 16): a streaming
// transform of every (a, b) column, U in shared memory, coalesced along b.
// (As a GEMM its M = D rows would leave a 128-row tensor-core tile empty.)
template <typename R>
__global__ void __launch_bounds__(256) k_apply_u(const ApplyUProb* __restrict__ probs) {
  using CT = typename C2<R>::T;
  const ApplyUProb P = probs[blockIdx.y];
  __shared__ CT Us[16 * 16];
  const int D = P.D;
  for (int i = threadIdx.x; i < D * D; i += blockDim.x) Us[i] = ((const CT*)P.U)[i];
  __syncthreads();
  const CT* src = (const CT*)P.src;
  CT* dst = (CT*)P.dst;
  const long long cols = (long long)P.chiL * P.chiR;
  for (long long col = blockIdx.x * (long long)blockDim.x + threadIdx.x; col < cols;
       col += (long long)gridDim.x * blockDim.x) {
    const long long a = col / P.chiR, b = col % P.chiR;
    const long long base = a * D * (long long)P.chiR + b;
    CT v[16];
#pragma unroll
    for (int s = 0; s < 16; s++) v[s] = s < D ? src[base + (long long)s * P.chiR] : cmk<CT>(0, 0);
    for (int t = 0; t < D; t++) {
      CT acc = cmk<CT>(0, 0);
#pragma unroll
      for (int s = 0; s < 16; s++)
        if (s < D) cfma(acc, Us[t * D + s], v[s]);
      dst[base + (long long)t * P.chiR] = acc;
    }
  }
}

template <typename R>
cudaError_t launch_apply_u(const ApplyUProb* d_probs, int n_probs, long long max_cols, cudaStream_t s) {
  if (n_probs <= 0 || max_cols <= 0) return cudaSuccess;
  long long gx = (max_cols + 255) / 256;
  if (gx > 4096) gx = 4096;
  k_apply_u<R><<<dim3((unsigned)gx, n_probs), 256, 0, s>>>(d_probs);
  return cudaGetLastError();
}
template cudaError_t launch_apply_u<float>(const ApplyUProb*, int, long long, cudaStream_t);
template cudaError_t launch_apply_u<double>(const ApplyUProb*, int, long long, cudaStream_t);

template <typename R>
__global__ void k_permute(const PermProb* __restrict__ probs) {
  using CT = typename C2<R>::T;
  const PermProb P = probs[blockIdx.y];
  const CT* src = (const CT*)P.src;
  CT* dst = (CT*)P.dst;
  const long long tot = (long long)P.rows * (P.mode == 0 ? P.cols : P.rows);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    if (P.mode == 0) {
      const long long r = e / P.cols;
      const int c = (int)(e % P.cols);
      dst[r * P.ldd + c] = src[r * P.lds + P.perm[c]];
    } else {
      const int i = (int)(e / P.rows), j = (int)(e % P.rows);
      dst[(long long)i * P.ldd + j] = (i < P.cols && j < P.cols)
                                          ? src[(long long)P.perm[i] * P.lds + P.perm[j]]
                                          : cmk<CT>(0, 0);
    }
  }
}

template <typename R>
cudaError_t launch_permute(const PermProb* d_probs, int n_probs, long long max_elems, cudaStream_t s) {
  if (n_probs <= 0 || max_elems <= 0) return cudaSuccess;
  long long gx = (max_elems + 255) / 256;
  if (gx > 65535) gx = 65535;
  k_permute<R><<<dim3((unsigned)gx, n_probs), 256, 0, s>>>(d_probs);
  return cudaGetLastError();
}
template cudaError_t launch_permute<float>(const PermProb*, int, long long, cudaStream_t);
template cudaError_t launch_permute<double>(const PermProb*, int, long long, cudaStream_t);

// ---------------------------------------------------------------------------
// One-qubit gates on singleton sites, amplitudes, conversions.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_apply_1q(void* const* __restrict__ sites, const int* __restrict__ cls,
                           const int* __restrict__ crs, const double* __restrict__ us) {
  using CT = typename C2<R>::T;
  const int p = blockIdx.y;
  const int cl = cls[p], cr = crs[p];
  CT* S = (CT*)sites[p];
  const double* u = us + 8 * p;
  const CT u00 = cmk<CT>(u[0], u[1]), u01 = cmk<CT>(u[2], u[3]);
  const CT u10 = cmk<CT>(u[4], u[5]), u11 = cmk<CT>(u[6], u[7]);
  const long long tot = (long long)cl * cr;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
       e += (long long)gridDim.x * blockDim.x) {
    const long long a = e / cr, b = e % cr;
    const long long i0 = (a * 2) * cr + b, i1 = (a * 2 + 1) * cr + b;
    const CT x0 = S[i0], x1 = S[i1];
    CT y0 = cmul(u00, x0), y1 = cmul(u10, x0);
    cfma(y0, u01, x1);
    cfma(y1, u11, x1);
    S[i0] = y0;
    S[i1] = y1;
  }
}

template <typename R>
cudaError_t launch_apply_1q(void* const* d_sites, const int* d_cl, const int* d_cr,
                            const double* d_u, int n_sites, long long max_elems, cudaStream_t s) {
  if (n_sites <= 0) return cudaSuccess;
  long long gx = (max_elems + 255) / 256;
  if (gx > 65535) gx = 65535;
  if (gx < 1) gx = 1;
  k_apply_1q<R><<<dim3((unsigned)gx, n_sites), 256, 0, s>>>(d_sites, d_cl, d_cr, d_u);
  return cudaGetLastError();
}
template cudaError_t launch_apply_1q<float>(void* const*, const int*, const int*, const double*,
                                            int, long long, cudaStream_t);
template cudaError_t launch_apply_1q<double>(void* const*, const int*, const int*, const double*,
                                             int, long long, cudaStream_t);

// FP32 complex <-> complex128
__global__ void k_narrow_c128(const double2* __restrict__ src, float2* __restrict__ dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double2 v = src[i];
    dst[i] = make_float2((float)v.x, (float)v.y);
  }
}
__global__ void k_widen_c128(const float2* __restrict__ src, double2* __restrict__ dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float2 v = src[i];
    dst[i] = make_double2(v.x, v.y);
  }
}
cudaError_t launch_narrow_c128(const double* src, float* dst, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const long long g = (n + 255) / 256;
  k_narrow_c128<<<(unsigned)(g > 8192 ? 8192 : g), 256, 0, s>>>((const double2*)src, (float2*)dst, n);
  return cudaGetLastError();
}
cudaError_t launch_widen_c128(const float* src, double* dst, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const long long g = (n + 255) / 256;
  k_widen_c128<<<(unsigned)(g > 8192 ? 8192 : g), 256, 0, s>>>((const float2*)src, (double2*)dst, n);
  return cudaGetLastError();
}

// Several device buffers in one launch, 16 bytes a thread where both ends
// allow it.  A state of 48 tensors and 49 spectra: 97 copies of 4 us each.
__global__ void __launch_bounds__(256) k_copy_batch(const CopyProb* __restrict__ probs) {
  const CopyProb P = probs[blockIdx.y];
  const long long t0 = blockIdx.x * 256LL + threadIdx.x, step = gridDim.x * 256LL;
  if ((((uintptr_t)P.src | (uintptr_t)P.dst) & 15) == 0) {
    const uint4* a = (const uint4*)P.src;
    uint4* b = (uint4*)P.dst;
    for (long long i = t0; i < P.words / 2; i += step) b[i] = a[i];
    if ((P.words & 1) && t0 == 0) ((uint2*)P.dst)[P.words - 1] = ((const uint2*)P.src)[P.words - 1];
  } else {
    for (long long i = t0; i < P.words; i += step) ((uint2*)P.dst)[i] = ((const uint2*)P.src)[i];
  }
}
cudaError_t launch_copy_batch(const CopyProb* d_probs, int count, long long max_words, cudaStream_t s) {
  long long gx = (max_words / 2 + 1023) / 1024;
  if (gx > 1024) gx = 1024;
  if (gx < 1) gx = 1;
  for (int i = 0; i < count; i += 32768)
    k_copy_batch<<<dim3((unsigned)gx, (unsigned)(count - i < 32768 ? count - i : 32768)), 256, 0, s>>>(d_probs + i);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP32 FMA throughput probe (the CUDA-core roofline of the FP32 kernels):
// every thread runs 8 independent FMA chains; 2 flops per FMA.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_fma_peak(float* __restrict__ out, int iters, float x, float y) {
  float a[8];
#pragma unroll
  for (int i = 0; i < 8; i++) a[i] = x + 1e-7f * (float)threadIdx.x + (float)i;
  for (int it = 0; it < iters; it++) {
#pragma unroll
    for (int i = 0; i < 8; i++) a[i] = fmaf(a[i], y, x);
  }
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < 8; i++) sum += a[i];
  if (sum == 1234.5f) out[blockIdx.x * blockDim.x + threadIdx.x] = sum;   // keeps the chains live
}

cudaError_t launch_fma_peak(float* out, int blocks, int iters, cudaStream_t s) {
  k_fma_peak<<<blocks, 256, 0, s>>>(out, iters, 1e-3f, 0.999f);
  return cudaGetLastError();
}

}  // namespace ctebd
