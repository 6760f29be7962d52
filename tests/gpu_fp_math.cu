// Functions of csrc/fp_math.cuh on the device, against FP64 over ranges of FP32 bit
// patterns (built as a shared library by tests/test_gpu_fp_math.py).
#include <cstdint>

#include <cuda_runtime.h>

#include "fp_math.cuh"

namespace {

// kind 0: tanh_pair, 1: tanh_pair_grad
__device__ void tanh_of(int kind, float x0, float x1, float &y0, float &y1) {
  if (kind == 0)
    bsi::fpm::tanh_pair(x0, x1, y0, y1);
  else
    bsi::fpm::tanh_pair_grad(x0, x1, y0, y1);
}

__global__ void k_tanh(int kind, const float *x, float *y, int n) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  float y0, y1;
  tanh_of(kind, x[i], i + 1 < n ? x[i + 1] : 0.f, y0, y1);
  y[i] = y0;
  if (i + 1 < n) y[i + 1] = y1;
}

// largest relative error of tanh over the n arguments with bit patterns lo, lo + 1, ..,
// and the sum of the relative differences to the correctly rounded FP32 value
__global__ void k_tanh_err(int kind, uint32_t lo, uint32_t n, unsigned long long *mx, double *sum) {
  double m = 0.0, s = 0.0;
  for (uint32_t i = 2 * (blockIdx.x * blockDim.x + threadIdx.x); i < n; i += 2 * gridDim.x * blockDim.x) {
    const float x0 = __uint_as_float(lo + i), x1 = -__uint_as_float(lo + min(i + 1, n - 1));
    float y0, y1;
    tanh_of(kind, x0, x1, y0, y1);
    const double e0 = y0 / tanh((double)x0) - 1.0, e1 = y1 / tanh((double)x1) - 1.0;
    m = fmax(m, fmax(fabs(e0), fabs(e1)));
    const float r0 = (float)tanh((double)x0), r1 = (float)tanh((double)x1);
    s += ((double)y0 - r0) / r0 + (i + 1 < n ? ((double)y1 - r1) / r1 : 0.0);
  }
  atomicMax(mx, (unsigned long long)__double_as_longlong(m));
  atomicAdd(sum, s);
}

// u = (x - mu) / sd by pairs of columns, n rows of two
__global__ void k_norm(const float *x, const float *mu, const float *sd, float *u, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  bsi::fpm::DivPair t;
  bsi::fpm::div_column(mu[2 * i], sd[2 * i], t.nmu.x, t.c.x, t.r.x, t.ns.x);
  bsi::fpm::div_column(mu[2 * i + 1], sd[2 * i + 1], t.nmu.y, t.c.y, t.r.y, t.ns.y);
  bsi::fpm::normalise_pair(x[2 * i], x[2 * i + 1], t, u[2 * i], u[2 * i + 1]);
}

__global__ void k_rsqrt(const double *s, double *y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = bsi::fpm::rsqrt64(s[i]);
}

}  // namespace

extern "C" {

// y[n] = 1 / sqrt(s[n]), host pointers
int fpm_rsqrt(const double *s, double *y, int n) {
  double *d = nullptr;
  if (n < 1 || cudaMalloc(&d, 2 * (size_t)n * sizeof(double)) != cudaSuccess) return 1;
  cudaError_t e = cudaMemcpy(d, s, (size_t)n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_rsqrt<<<(n + 255) / 256, 256>>>(d, d + n, n);
    e = cudaMemcpy(y, d + n, (size_t)n * sizeof(double), cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  return e == cudaSuccess ? 0 : 1;
}


// in: x, mu, sd, 2 n values each; out: 2 n; host pointers
int fpm_normalise(const float *in, float *out, int n) {
  float *d = nullptr;
  if (n < 1 || cudaMalloc(&d, 8 * (size_t)n * sizeof(float)) != cudaSuccess) return 1;
  cudaError_t e = cudaMemcpy(d, in, 6 * (size_t)n * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_norm<<<(n + 255) / 256, 256>>>(d, d + 2 * n, d + 4 * n, d + 6 * n, n);
    e = cudaMemcpy(out, d + 6 * n, 2 * (size_t)n * sizeof(float), cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  return e == cudaSuccess ? 0 : 1;
}


// y[n] = tanh(x[n]), host pointers
int fpm_tanh(int kind, const float *x, float *y, int n) {
  float *d = nullptr;
  if (n < 1 || cudaMalloc(&d, 2 * (size_t)n * sizeof(float)) != cudaSuccess) return 1;
  cudaError_t e = cudaMemcpy(d, x, (size_t)n * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_tanh<<<((n + 1) / 2 + 255) / 256, 256>>>(kind, d, d + n, n);
    e = cudaMemcpy(y, d + n, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  return e == cudaSuccess ? 0 : 1;
}

// out: largest relative error, mean error
int fpm_tanh_err(int kind, uint32_t lo, uint32_t n, double *out) {
  double *d = nullptr;
  if (n < 1 || n > (1u << 30) || cudaMalloc(&d, 16) != cudaSuccess) return 1;
  double h[2] = {0.0, 0.0};
  cudaError_t e = cudaMemcpy(d, h, 16, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_tanh_err<<<152 * 8, 256>>>(kind, lo, n, reinterpret_cast<unsigned long long *>(d), d + 1);
    e = cudaMemcpy(h, d, 16, cudaMemcpyDeviceToHost);
  }
  cudaFree(d);
  out[0] = h[0];
  out[1] = h[1] / n;
  return e == cudaSuccess ? 0 : 1;
}

}  // extern "C"
