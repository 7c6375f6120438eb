// Host program of test_gpu_numeric.py: evaluates the scalar routines of
// numeric.cuh and pair.cuh on numbers from standard input (FP64, binary) and
// writes the results as FP64 numbers (high and low part of each), or lets a
// bounded wait run out.
//   numeric_probe FUNCTION COUNT     sqrt32 rcp32 sqrt64 rcp64 pair_sqrt pair_rcp
//   numeric_probe wait 0             one poll of a slot that nothing fills
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "exchange.cuh"
#include "numeric.cuh"
#include "pair.cuh"

using namespace ctebd;

enum { SQRT32, RCP32, SQRT64, RCP64, PAIR_SQRT, PAIR_RCP };

// out: two numbers per input, high and low part of the result
__global__ void k_eval(int fn, const double* x, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  double h = 0, l = 0;
  if (fn == SQRT32) h = sqrt_nr((float)v);
  if (fn == RCP32) h = rcp_nr((float)v);
  if (fn == SQRT64) h = sqrt_nr(v);
  if (fn == RCP64) h = rcp_nr(v);
  if (fn == PAIR_SQRT || fn == PAIR_RCP) {
    const Pair p = Real<float>::of(v), r = fn == PAIR_SQRT ? Real<float>::root(p) : Real<float>::rcp(p);
    h = r.h; l = r.l;
  }
  out[2 * i] = h;
  out[2 * i + 1] = l;
}

__global__ void k_wait(const unsigned char* slot, int* err, int* ok) {
  const unsigned char* ad[1] = {slot};
  float2 v[1];
  *ok = poll(ad, 1u, v, err, kWaitSplit) ? 1 : 0;
}

static void check(cudaError_t e) {
  if (e != cudaSuccess) { std::fprintf(stderr, "%s\n", cudaGetErrorString(e)); std::exit(1); }
}

int main(int argc, char** argv) {
  if (argc < 3) return 2;
  if (!std::strcmp(argv[1], "wait")) {
    unsigned char* slot;
    int *w, h[2];
    check(cudaMalloc(&slot, 64));
    check(cudaMalloc(&w, sizeof(h)));
    check(cudaMemset(slot, 0, 64));
    check(cudaMemset(w, 0, sizeof(h)));
    k_wait<<<1, 1>>>(slot, w, w + 1);
    check(cudaDeviceSynchronize());
    check(cudaMemcpy(h, w, sizeof(h), cudaMemcpyDeviceToHost));
    std::printf("%d %d %s\n", h[0], h[1], wait_name(h[0]));
    return 0;
  }
  const char* names[] = {"sqrt32", "rcp32", "sqrt64", "rcp64", "pair_sqrt", "pair_rcp"};
  int fn = -1;
  for (int i = 0; i < 6; i++)
    if (!std::strcmp(argv[1], names[i])) fn = i;
  const int n = std::atoi(argv[2]);
  if (fn < 0 || n < 1) return 2;
  std::vector<double> x(n), y(2 * (size_t)n);
  if (std::fread(x.data(), sizeof(double), n, stdin) != (size_t)n) return 2;
  double *dx, *dy;
  check(cudaMalloc(&dx, sizeof(double) * n));
  check(cudaMalloc(&dy, sizeof(double) * 2 * n));
  check(cudaMemcpy(dx, x.data(), sizeof(double) * n, cudaMemcpyHostToDevice));
  k_eval<<<(n + 255) / 256, 256>>>(fn, dx, dy, n);
  check(cudaDeviceSynchronize());
  check(cudaMemcpy(y.data(), dy, sizeof(double) * y.size(), cudaMemcpyDeviceToHost));
  return std::fwrite(y.data(), sizeof(double), y.size(), stdout) == y.size() ? 0 : 1;
}
