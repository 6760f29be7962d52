// Shared between the surrogate's FP32 SIMT kernels (mlp.cu) and its
// tensor-core kernels (mlp_tc.cu).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace bsi {

struct MlpDev {
  int d, w;
  float *p;       // master FP32 params, flat: W1 [w][d] | b1 | W2 [w][w] | b2 | w3 | b3
  float *g;       // gradient, same layout
  float *m, *v;   // Adam moments
  float *norm;    // mu_x [d] | sd_x [d] | mu_y | sd_y
};

__host__ __device__ inline unsigned long long mlp_mix(unsigned long long z) {  // SplitMix64
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
// Row of the data set that row r of a training step draws (with replacement).
__host__ __device__ inline int mlp_sample_row(unsigned long long seed, int step, int r, int n) {
  return (int)(mlp_mix(seed ^ mlp_mix(((unsigned long long)step << 32) | (unsigned)r)) %
               (unsigned long long)n);
}

// Tensor-core (mma.sync BF16, FP32 accumulation) forms.  Width 128, d <= 64.
// mlp_tc_infer: y of n rows.  mlp_tc_grad: the loss (added to *loss) and the
// partial gradients part[mlp_tc_parts(nrows)][] of the first nrows rows, or of
// nrows drawn ones; mlp_tc_reduce: their sum into M.g, or straight into an Adam
// step.  im: the network as the gradient kernel stages it (mlp_tc_image_bytes;
// zeroed once), made from M.p by mlp_tc_image and kept up by the Adam step.
bool mlp_tc_supported(int d, int w);
cudaError_t mlp_tc_infer(const MlpDev &M, const float *x, int n, float *y, cudaStream_t s);
size_t mlp_tc_image_bytes(int d);
cudaError_t mlp_tc_image(const MlpDev &M, unsigned char *im, cudaStream_t s);
int mlp_tc_parts(int nrows);
size_t mlp_tc_part_bytes(int d);  // of one partial gradient
cudaError_t mlp_tc_grad(const MlpDev &M, const float *x, const float *t, int n, int nrows, int sampled,
                        uint64_t seed, int step, const unsigned char *im, float *part, float *loss,
                        cudaStream_t s);
cudaError_t mlp_tc_reduce(const MlpDev &M, int nparts, const float *part, int adam, float lr, float b1,
                          float b2, float eps, int step, unsigned char *im, cudaStream_t s);

}  // namespace bsi
