// Error-bar surrogate on the tensor cores: the forward pass, the per-row
// backward and the weight gradients of the width-128 network as BF16
// mma.sync (m16n8k16, FP32 accumulation).  The FP32 SIMT kernels of mlp.cu
// compute the same quantities and serve as the checker.
//
// Precision.  The network's weights are BF16 values by definition (the FP32
// masters rounded when staged), so a weight operand is exact in BF16.  Every
// other operand x (activations, normalised inputs, back-propagated dz) is
// split x = hi + lo, hi = bf16(x), lo = bf16(x - hi): 16 significant bits.
// Forward and dz1 products take W hi + W lo (two MMAs); the weight gradients
// (both operands split) take hi hi + hi lo + lo hi (three MMAs; lo lo is
// below 2^-16 of the term).  Accumulation is FP32 throughout.
//
// Fragment layouts (PTX ISA, mma.m16n8k16 with .bf16 operands): g = lane / 4,
// t = lane % 4.  A (16 x 16, row major): a0 = (g, 2t..2t+1), a1 = (g + 8,
// 2t..), a2 = (g, 2t + 8..), a3 = (g + 8, 2t + 8..).  B (16 x 8, K x N):
// b0 = (k = 2t..2t+1, n = g), b1 = (k = 2t + 8.., n = g).  C (16 x 8):
// c0, c1 = (g, 2t..2t+1), c2, c3 = (g + 8, 2t..).  The lower half of each
// 32-bit register holds the element with the smaller index.  A C tile pair
// (n-tiles 2kk, 2kk + 1) is exactly the A fragment of k-step kk of the next
// layer, so activations stay in registers between the layers.
//
// Kernels:
//   inference     h1 = tanh(W1 xn + b1), h2 = tanh(W2 h1 + b2), yn = w3.h2 + b3
//   gradient      the same forward, dz2 = dyn w3 (1 - h2^2), dz1 = (W2^T dz2)(1 - h1^2),
//                 dW1 = dz1^T xn, dW2 = dz2^T h1, in one kernel: nothing of a row
//                 goes through global memory
#include <cuda_bf16.h>

#include <algorithm>

#include "bs_internal.h"
#include "fp_math.cuh"
#include "mlp_internal.h"

namespace bsi {

namespace {

using fpm::DivPair;
using fpm::normalise_pair;
using fpm::scale_pair;
using fpm::tanh_pair;
using fpm::tanh_pair_grad;

constexpr int W = 128;           // hidden width of the tensor-core kernels
constexpr int kWarps = 8, kThreads = 32 * kWarps, kRowsPerCta = 16 * kWarps;
constexpr int LD2 = W + 8;       // bf16 pitch of the staged W2 (conflict-free fragments)

__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b) {
  return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}
// hi / lo BF16 parts of two consecutive elements, packed
__device__ __forceinline__ void split2(float x0, float x1, uint32_t &hi, uint32_t &lo) {
  const __nv_bfloat16 h0 = __float2bfloat16_rn(x0), h1 = __float2bfloat16_rn(x1);
  const __nv_bfloat16 l0 = __float2bfloat16_rn(x0 - __bfloat162float(h0));
  const __nv_bfloat16 l1 = __float2bfloat16_rn(x1 - __bfloat162float(h1));
  hi = pack2(h0, h1);
  lo = pack2(l0, l1);
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// W1 [W][d] as BF16 rows of pitch K1 + 8 (zero beyond d), W2 [W][W] of pitch
// LD2, biases and w3 in FP32 (w3 BF16-rounded, as the network defines it).
template <int K1>
__device__ void stage_net(const MlpDev &M, __nv_bfloat16 *W1s, __nv_bfloat16 *W2s, float *b1,
                          float *b2, float *w3) {
  constexpr int LD1 = K1 + 8;
  const int d = M.d;
  const float *p = M.p;
  for (int q = threadIdx.x; q < W * K1; q += blockDim.x) {
    const int j = q / K1, k = q - j * K1;
    W1s[j * LD1 + k] = __float2bfloat16_rn(k < d ? p[j * d + k] : 0.f);
  }
  p += W * d;
  for (int q = threadIdx.x; q < W; q += blockDim.x) b1[q] = p[q];
  p += W;
  for (int q = threadIdx.x; q < W * W; q += blockDim.x) {
    const int j = q / W, k = q - j * W;
    W2s[j * LD2 + k] = __float2bfloat16_rn(p[q]);
  }
  p += W * W;
  for (int q = threadIdx.x; q < W; q += blockDim.x) b2[q] = p[q];
  p += W;
  for (int q = threadIdx.x; q < W; q += blockDim.x) w3[q] = __bfloat162float(__float2bfloat16_rn(p[q]));
}

// The normalisation of columns 2q and 2q + 1 in table entry q; columns beyond d pass zeros.
template <int K1>
__device__ void stage_norm(const MlpDev &M, DivPair *tab) {
  for (int q = threadIdx.x; q < K1 / 2; q += blockDim.x) {
    const int k = 2 * q, d = M.d;
    DivPair t;
    fpm::div_column(k < d ? M.norm[k] : 0.f, k < d ? M.norm[d + k] : 1.f, t.nmu.x, t.c.x, t.r.x, t.ns.x);
    fpm::div_column(k + 1 < d ? M.norm[k + 1] : 0.f, k + 1 < d ? M.norm[d + k + 1] : 1.f, t.nmu.y, t.c.y,
                    t.r.y, t.ns.y);
    tab[q] = t;
  }
}

// ------------------------------------------------------------- inference
//
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// Programmatic dependent launch.  A training step is two kernels of 4 and 16 us: the
// next one's blocks start while the last blocks of this one run (pdl_launch, once all
// have started), and wait (pdl_wait: complete and visible) before they touch what it
// writes.  The gradient kernel has its first rows staged by then.  24 steps with one
// large gradient and the statistics: 1.00 ms, 0.88 with it.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
cudaError_t launch_pdl(void (*k)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// B fragments of n-tiles j, j + 1 (rows 8j .. 8j + 15 of a weight matrix stored
// [n][k]) at k-step kk: the address this lane gives to ldsm4; r[0], r[1] are tile
// j's two registers, r[2], r[3] tile j + 1's.
__device__ __forceinline__ uint32_t b_addr(uint32_t base, int ld, int j, int kk, int lane) {
  return base + 2u * (uint32_t)((8 * j + (lane & 7) + ((lane >> 4) << 3)) * ld + 16 * kk + (lane & 8));
}

// y of n rows (no activations stored): the CTAs are persistent over tiles of 128
// rows, so the weights are staged once per CTA.  A tile's rows are contiguous and
// come in by 16-byte asynchronous copies while the previous tile computes (they
// are needed for its first layer only).
//
// Bound by instruction issue and the exponentials of 256 tanh a row, not by the
// tensor pipe or HBM: the kernel it replaced issued 5970 warp instructions per 16
// rows (weights staged for every 128 rows, one 32-bit shared load per B register,
// a division per input, the library tanh on two divergent branches) and kept the
// issue slots 47% busy.  1540 x 60^2 rows: 1.86 ms, 3.71 ms before.
template <int K1>
__global__ void __launch_bounds__(kThreads, 2) k_mlp_tc_infer(MlpDev M, const float *__restrict__ x,
                                                              int n, float *__restrict__ y) {
  constexpr int LD1 = K1 + 8, KS1 = K1 / 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __nv_bfloat16 *W1s = reinterpret_cast<__nv_bfloat16 *>(smem_raw);
  __nv_bfloat16 *W2s = W1s + W * LD1;
  float *b1 = reinterpret_cast<float *>(W2s + W * LD2), *b2 = b1 + W, *w3 = b2 + W;
  DivPair *norm = reinterpret_cast<DivPair *>(w3 + W);  // [K1 / 2]
  float *xs = reinterpret_cast<float *>(norm + K1 / 2);  // [128][d], 16-byte aligned
  const int d = M.d, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const bool wide = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const int ntile = (n + kRowsPerCta - 1) / kRowsPerCta;
  auto load = [&](int tile) {
    const long long e0 = (long long)tile * kRowsPerCta * d;
    const int ne = (int)min((long long)kRowsPerCta * d, (long long)n * d - e0);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(xs);
    const int n4 = wide ? ne / 4 : 0;
    for (int q = threadIdx.x; q < n4; q += kThreads)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * q), "l"(x + e0 + 4 * q)
                   : "memory");
    for (int q = 4 * n4 + threadIdx.x; q < ne; q += kThreads)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * q), "l"(x + e0 + q)
                   : "memory");
    for (int q = ne + threadIdx.x; q < kRowsPerCta * d; q += kThreads) xs[q] = 0.f;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (blockIdx.x < ntile) load(blockIdx.x);
  stage_net<K1>(M, W1s, W2s, b1, b2, w3);
  stage_norm<K1>(M, norm);
  const float b3 = M.p[(long long)W * d + W + W * W + W + W];
  const float my = M.norm[2 * d], sy = M.norm[2 * d + 1];
  const uint32_t a1 = (uint32_t)__cvta_generic_to_shared(W1s), a2 = (uint32_t)__cvta_generic_to_shared(W2s);
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const float *x0 = xs + (16 * warp + g) * d, *x1 = x0 + 8 * d;
    // layer 1: A = xn (hi, lo), B = W1^T, accumulators start at the bias
    uint32_t ah[KS1][4], al[KS1][4];
#pragma unroll
    for (int kk = 0; kk < KS1; ++kk) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {  // a0: (g, 2t), a1: (g+8, 2t), a2: (g, 2t+8), a3: (g+8, 2t+8)
        const int col = 16 * kk + 2 * t + ((q >> 1) << 3);
        const float *xr = (q & 1) ? x1 : x0;
        float u0, u1;
        normalise_pair(col < d ? xr[col] : 0.f, col + 1 < d ? xr[col + 1] : 0.f, norm[col / 2], u0, u1);
        split2(u0, u1, ah[kk][q], al[kk][q]);
      }
    }
    __syncthreads();
    if (tile + (int)gridDim.x < ntile) load(tile + gridDim.x);
    uint32_t h1h[8][4], h1l[8][4];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      float c[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 b = *reinterpret_cast<const float2 *>(b1 + 8 * (8 * half + j) + 2 * t);
        c[j][0] = c[j][2] = b.x;
        c[j][1] = c[j][3] = b.y;
      }
#pragma unroll
      for (int kk = 0; kk < KS1; ++kk) {
        uint32_t r[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) ldsm4(r[j], b_addr(a1, LD1, 8 * half + 2 * j, kk, lane));
#pragma unroll
        for (int j = 0; j < 8; ++j) mma16816(c[j], ah[kk], r[j / 2][2 * (j & 1)], r[j / 2][2 * (j & 1) + 1]);
#pragma unroll
        for (int j = 0; j < 8; ++j) mma16816(c[j], al[kk], r[j / 2][2 * (j & 1)], r[j / 2][2 * (j & 1) + 1]);
      }
      // h1 = tanh(z1): n-tile 2kk -> a0, a1 of k-step kk; 2kk + 1 -> a2, a3
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int kk = (8 * half + j) >> 1, hs = (j & 1) * 2;
        float p0, p1, q0, q1;
        tanh_pair(c[j][0], c[j][1], p0, p1);
        tanh_pair(c[j][2], c[j][3], q0, q1);
        split2(p0, p1, h1h[kk][hs], h1l[kk][hs]);
        split2(q0, q1, h1h[kk][hs + 1], h1l[kk][hs + 1]);
      }
    }
    float y0 = 0.f, y1 = 0.f;
#pragma unroll 1
    for (int qt = 0; qt < 4; ++qt) {  // layer 2, four n-tiles at a time
      float c[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 b = *reinterpret_cast<const float2 *>(b2 + 8 * (4 * qt + j) + 2 * t);
        c[j][0] = c[j][2] = b.x;
        c[j][1] = c[j][3] = b.y;
      }
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        uint32_t r[2][4];
#pragma unroll
        for (int j = 0; j < 2; ++j) ldsm4(r[j], b_addr(a2, LD2, 4 * qt + 2 * j, kk, lane));
#pragma unroll
        for (int j = 0; j < 4; ++j) mma16816(c[j], h1h[kk], r[j / 2][2 * (j & 1)], r[j / 2][2 * (j & 1) + 1]);
#pragma unroll
        for (int j = 0; j < 4; ++j) mma16816(c[j], h1l[kk], r[j / 2][2 * (j & 1)], r[j / 2][2 * (j & 1) + 1]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 w = *reinterpret_cast<const float2 *>(w3 + 8 * (4 * qt + j) + 2 * t);
        float p0, p1, q0, q1;
        tanh_pair(c[j][0], c[j][1], p0, p1);
        tanh_pair(c[j][2], c[j][3], q0, q1);
        y0 = fmaf(w.x, p0, fmaf(w.y, p1, y0));
        y1 = fmaf(w.x, q0, fmaf(w.y, q1, y1));
      }
    }
    // the four threads of a group hold the row's partial dot products
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    const int r0 = tile * kRowsPerCta + 16 * warp + g;
    if (t == 0 && r0 < n) y[r0] = my + sy * (y0 + b3);
    if (t == 0 && r0 + 8 < n) y[r0 + 8] = my + sy * (y1 + b3);
  }
}

// ------------------------------------------------------------- gradient
//
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr));
}

constexpr int kGradRows = 64, kGradThreads = 512;

// Floats from one partial gradient to the next (the parameters, padded to 16 bytes).
__host__ __device__ constexpr int part_stride(int d) {
  return (W * d + W + W * W + W + W + 1 + 3) / 4 * 4;
}
// The network as the gradient kernel stages it: W1 [W][K1 + 8] and W2 [W][LD2] in BF16,
// then b1, b2, w3 (BF16-rounded), in one block of 16-byte pieces.
constexpr int image_bytes(int k1) { return W * (k1 + 8) * 2 + W * LD2 * 2 + 3 * W * 4; }
// Parameter q's value into the image (b3 is read from the parameters).
__device__ __forceinline__ void image_put(unsigned char *im, int d, int k1, int q, float v) {
  __nv_bfloat16 *W1 = reinterpret_cast<__nv_bfloat16 *>(im), *W2 = W1 + W * (k1 + 8);
  float *vec = reinterpret_cast<float *>(W2 + W * LD2);
  if (q < W * d) {
    const int j = q / d;
    W1[j * (k1 + 8) + q - j * d] = __float2bfloat16_rn(v);
    return;
  }
  q -= W * d;
  if (q < W) {
    vec[q] = v;
    return;
  }
  q -= W;
  if (q < W * W) {
    W2[(q / W) * LD2 + q % W] = __float2bfloat16_rn(v);
    return;
  }
  q -= W * W;
  if (q < W)
    vec[W + q] = v;
  else if (q < 2 * W)
    vec[W + q] = __bfloat162float(__float2bfloat16_rn(v));
}
__global__ void k_mlp_tc_image(MlpDev M, int k1, int np, unsigned char *__restrict__ im) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < np) image_put(im, M.d, k1, q, M.p[q]);
}

// Shared memory of the gradient kernel (BF16 tiles row major, FP32 vectors).
template <int K1>
struct GradLay {
  static constexpr int LD1 = K1 + 8;
  static constexpr int W1s = 0, W2s = W1s + W * LD1 * 2, net = W2s + W * LD2 * 2;
  static constexpr int X = net + 3 * W * 4;             // hi, lo [64][LD1]
  static constexpr int H1 = X + 2 * kGradRows * LD1 * 2;  // hi, lo [64][LD2]
  static constexpr int Z2 = H1 + 2 * kGradRows * LD2 * 2, Z1 = Z2 + 2 * kGradRows * LD2 * 2;
  static constexpr int vec = Z1 + 2 * kGradRows * LD2 * 2;
  // gb1, gb2, gw3 [4][W], norm [K1 / 2], yn parts [4][64], tn, ok [64], row [64], gb3
  static constexpr int bytes = vec + (12 * W + 4 * K1 + 4 * kGradRows + 3 * kGradRows + 4) * 4;
};

// Loss and gradient of nrows rows (drawn as k_mlp_sample draws them when seeded:
// row r of step `step` is mix(seed, step, r) mod n) as one partial gradient per CTA,
// part[CTA][np], summed by k_mlp_tc_reduce; loss += mean of squared residuals.
//
// A tile of 64 rows takes the 16 warps through five MMA passes (forward 1 and 2,
// dz1, dW2, dW1) with its activations in shared memory: warp w has rows 16 (w % 4)
// and outputs 32 (w / 4) of the per-row passes, and keeps a 16 x 64 block of dW2
// and a 16 x K1/2 block of dW1 in registers over all its tiles.  Transposed operands
// (W2^T, dz^T, h1, xn by rows) come out of the row-major tiles with
// ldmatrix.trans.
//
// The three kernels it replaced wrote 559 floats a row to global memory and read
// them back, ran a batch of 8192 rows on 64 of the 152 SMs, staged the weights in
// each, transposed through strided 16-bit stores and added every CTA's 22 thousand
// weights with atomics.  24 steps of 8192 rows and one gradient of 122880 (d = 45): 2.43 ms in
// those kernels, 0.65 here (with k_mlp_tc_reduce).
template <int K1>
__global__ void __launch_bounds__(kGradThreads, 1)
    k_mlp_tc_grad(MlpDev M, const float *__restrict__ x, const float *__restrict__ tgt, int n,
                  int nrows, int sampled, unsigned long long seed, int step,
                  const unsigned char *im, float *__restrict__ part,
                  float *__restrict__ loss) {
  using Ly = GradLay<K1>;
  constexpr int LD1 = K1 + 8, KS1 = K1 / 16, NT1 = K1 / 16;  // dW1 n-tiles of a warp
  static_assert(part_stride(K1) * 4 <= Ly::vec - Ly::X, "the partial gradient over the tile's buffers");
  extern __shared__ __align__(16) unsigned char sm[];
  const float *b1 = reinterpret_cast<const float *>(sm + Ly::net), *b2 = b1 + W, *w3 = b2 + W;
  float *gb1 = reinterpret_cast<float *>(sm + Ly::vec), *gb2 = gb1 + 4 * W, *gw3 = gb2 + 4 * W;
  DivPair *norm = reinterpret_cast<DivPair *>(gw3 + 4 * W);
  float *ypart = reinterpret_cast<float *>(norm + K1 / 2), *tn = ypart + 4 * kGradRows, *okr = tn + kGradRows;
  int *rowid = reinterpret_cast<int *>(okr + kGradRows);
  float *gb3 = reinterpret_cast<float *>(rowid + kGradRows);
  const int d = M.d, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int rg = warp & 3, cq = warp >> 2;   // per-row passes: rows 16 rg.., outputs 32 cq..
  const int jb = warp & 7, kb = warp >> 3;   // weight gradients: rows 16 jb.., half kb of the inputs
  const uint32_t sb = (uint32_t)__cvta_generic_to_shared(sm);
  const uint32_t aW1 = sb + Ly::W1s, aW2 = sb + Ly::W2s;
  pdl_launch();
  for (int q = tid; q < 12 * W; q += kGradThreads) gb1[q] = 0.f;
  if (tid == 0) *gb3 = 0.f;
  stage_norm<K1>(M, norm);
  float b3 = 0.f;
  const float my = M.norm[2 * d], sy = M.norm[2 * d + 1];
  float l2 = 0.f, sdy = 0.f;  // sums of squared residuals and of dyn
  float gW2[8][4], gW1[NT1][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) gW2[j][0] = gW2[j][1] = gW2[j][2] = gW2[j][3] = 0.f;
#pragma unroll
  for (int j = 0; j < NT1; ++j) gW1[j][0] = gW1[j][1] = gW1[j][2] = gW1[j][3] = 0.f;

  // lane offsets (elements) of the 8x8 matrices of an ldmatrix.x4
  const int aro = lane & 15, aco = (lane >> 4) << 3;                       // A: rows, then k + 8
  const int tro = (lane & 7) + ((lane >> 4) << 3), tco = lane & 8;         // A^T from [k][m]
  const int bro = lane & 15, bco = (lane >> 4) << 3;                       // B from [k][n]: two n-tiles
  auto a_at = [&](uint32_t buf, int ld, int r0, int kk) {
    return buf + 2u * (uint32_t)((r0 + aro) * ld + 16 * kk + aco);
  };

  const int ntile = (nrows - 1) / kGradRows + 1;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    __syncthreads();  // the previous tile's readers are done
    if (tid < kGradRows) {
      const int r = tile * kGradRows + tid;
      int row = -1;
      if (r < nrows) row = sampled ? mlp_sample_row(seed, step, r, n) : r;
      rowid[tid] = row;
      okr[tid] = row >= 0 ? 1.f : 0.f;
      tn[tid] = row >= 0 ? (tgt[row] - my) / sy : 0.f;
    }
    __syncthreads();
    for (int q = tid; q < kGradRows * (K1 / 2); q += kGradThreads) {
      const int r = q / (K1 / 2), c = 2 * (q - r * (K1 / 2)), row = rowid[r];
      float v0 = 0.f, v1 = 0.f;
      if (row >= 0) {
        const float *xr = x + (long long)row * d;
        scale_pair(c < d ? xr[c] : 0.f, c + 1 < d ? xr[c + 1] : 0.f, norm[c / 2], v0, v1);
      }
      uint32_t hi, lo;
      split2(v0, v1, hi, lo);
      *reinterpret_cast<uint32_t *>(sm + Ly::X + 2 * (r * LD1 + c)) = hi;
      *reinterpret_cast<uint32_t *>(sm + Ly::X + 2 * (kGradRows * LD1 + r * LD1 + c)) = lo;
    }
    if (tile == (int)blockIdx.x) {  // the network, once the previous step has updated it
      pdl_wait();
      for (int q = tid; q < (Ly::net + 3 * W * 4) / 16; q += kGradThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sb + 16u * q), "l"(im + 16 * q)
                     : "memory");
      asm volatile("cp.async.wait_all;" ::: "memory");
      b3 = __ldcg(M.p + (long long)W * d + W + W * W + W + W);  // the step before writes it
    }
    __syncthreads();
    // ---- forward 1
    float h1[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 b = *reinterpret_cast<const float2 *>(b1 + 32 * cq + 8 * j + 2 * t);
      h1[j][0] = h1[j][2] = b.x;
      h1[j][1] = h1[j][3] = b.y;
    }
#pragma unroll
    for (int kk = 0; kk < KS1; ++kk) {
      uint32_t ah[4], al[4], r0[4], r1[4];
      ldsm4(ah, a_at(sb + Ly::X, LD1, 16 * rg, kk));
      ldsm4(al, a_at(sb + Ly::X + 2 * kGradRows * LD1, LD1, 16 * rg, kk));
      ldsm4(r0, b_addr(aW1, LD1, 4 * cq, kk, lane));
      ldsm4(r1, b_addr(aW1, LD1, 4 * cq + 2, kk, lane));
      mma16816(h1[0], ah, r0[0], r0[1]);
      mma16816(h1[1], ah, r0[2], r0[3]);
      mma16816(h1[2], ah, r1[0], r1[1]);
      mma16816(h1[3], ah, r1[2], r1[3]);
      mma16816(h1[0], al, r0[0], r0[1]);
      mma16816(h1[1], al, r0[2], r0[3]);
      mma16816(h1[2], al, r1[0], r1[1]);
      mma16816(h1[3], al, r1[2], r1[3]);
    }
    // a C tile's pair (row, columns 2t, 2t + 1) into a row-major hi / lo tile
    auto put = [&](int buf, int j, const float (&c)[4]) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t hi, lo;
        split2(c[2 * q], c[2 * q + 1], hi, lo);
        const int o = (16 * rg + g + 8 * q) * LD2 + 32 * cq + 8 * j + 2 * t;
        *reinterpret_cast<uint32_t *>(sm + buf + 2 * o) = hi;
        *reinterpret_cast<uint32_t *>(sm + buf + 2 * (kGradRows * LD2 + o)) = lo;
      }
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      tanh_pair_grad(h1[j][0], h1[j][1], h1[j][0], h1[j][1]);
      tanh_pair_grad(h1[j][2], h1[j][3], h1[j][2], h1[j][3]);
      put(Ly::H1, j, h1[j]);
    }
    __syncthreads();
    // ---- forward 2 and the output
    float c2[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 b = *reinterpret_cast<const float2 *>(b2 + 32 * cq + 8 * j + 2 * t);
      c2[j][0] = c2[j][2] = b.x;
      c2[j][1] = c2[j][3] = b.y;
    }
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      uint32_t ah[4], al[4], r0[4], r1[4];
      ldsm4(ah, a_at(sb + Ly::H1, LD2, 16 * rg, kk));
      ldsm4(al, a_at(sb + Ly::H1 + 2 * kGradRows * LD2, LD2, 16 * rg, kk));
      ldsm4(r0, b_addr(aW2, LD2, 4 * cq, kk, lane));
      ldsm4(r1, b_addr(aW2, LD2, 4 * cq + 2, kk, lane));
      mma16816(c2[0], ah, r0[0], r0[1]);
      mma16816(c2[1], ah, r0[2], r0[3]);
      mma16816(c2[2], ah, r1[0], r1[1]);
      mma16816(c2[3], ah, r1[2], r1[3]);
      mma16816(c2[0], al, r0[0], r0[1]);
      mma16816(c2[1], al, r0[2], r0[3]);
      mma16816(c2[2], al, r1[0], r1[1]);
      mma16816(c2[3], al, r1[2], r1[3]);
    }
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 w = *reinterpret_cast<const float2 *>(w3 + 32 * cq + 8 * j + 2 * t);
      tanh_pair_grad(c2[j][0], c2[j][1], c2[j][0], c2[j][1]);
      tanh_pair_grad(c2[j][2], c2[j][3], c2[j][2], c2[j][3]);
      y0 = fmaf(w.x, c2[j][0], fmaf(w.y, c2[j][1], y0));
      y1 = fmaf(w.x, c2[j][2], fmaf(w.y, c2[j][3], y1));
    }
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    if (t == 0) {
      ypart[cq * kGradRows + 16 * rg + g] = y0;
      ypart[cq * kGradRows + 16 * rg + g + 8] = y1;
    }
    __syncthreads();
    // ---- dz2 and the sums over rows that need no product
    float dyn[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int r = 16 * rg + g + 8 * q;
      const float yn = ypart[r] + ypart[kGradRows + r] + ypart[2 * kGradRows + r] +
                       ypart[3 * kGradRows + r] + b3;
      const float res = okr[r] != 0.f ? yn - tn[r] : 0.f;
      dyn[q] = 2.f * res / (float)nrows;
      if (cq == 0 && t == 0) {
        l2 += res * res;
        sdy += dyn[q];
      }
    }
    // sums over the warp's 16 rows of its 32 columns (v[2 j + q]: column 8 j + 2 t + q),
    // scattered over the row lanes: lane g ends with v[g], and adds it to the warp's
    // own slot (shared-memory atomics on one address per column cost more than the MMAs)
    auto colsum = [&](float *dst, float (&v)[8]) {
#pragma unroll
      for (int s = 4; s >= 1; s >>= 1) {
        const bool up = g & s;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (k < s) {
            const float keep = up ? v[k + s] : v[k], give = up ? v[k] : v[k + s];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * s);
          }
      }
      dst[rg * W + 32 * cq + 8 * (g >> 1) + 2 * t + (g & 1)] += v[0];
    };
    float s3[8], s2[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 w = *reinterpret_cast<const float2 *>(w3 + 32 * cq + 8 * j + 2 * t);
      s3[2 * j] = dyn[0] * c2[j][0] + dyn[1] * c2[j][2];
      s3[2 * j + 1] = dyn[0] * c2[j][1] + dyn[1] * c2[j][3];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float h0 = c2[j][2 * q], h1v = c2[j][2 * q + 1];
        c2[j][2 * q] = dyn[q] != 0.f ? dyn[q] * w.x * (1.f - h0 * h0) : 0.f;
        c2[j][2 * q + 1] = dyn[q] != 0.f ? dyn[q] * w.y * (1.f - h1v * h1v) : 0.f;
      }
      s2[2 * j] = c2[j][0] + c2[j][2];
      s2[2 * j + 1] = c2[j][1] + c2[j][3];
      put(Ly::Z2, j, c2[j]);
    }
    colsum(gw3, s3);
    colsum(gb2, s2);
    __syncthreads();
    // ---- dz1 = (dz2 W2)(1 - h1^2): B from W2 [j][k] by transposed loads
    float z1[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) z1[j][0] = z1[j][1] = z1[j][2] = z1[j][3] = 0.f;
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      uint32_t ah[4], al[4], r0[4], r1[4];
      ldsm4(ah, a_at(sb + Ly::Z2, LD2, 16 * rg, kk));
      ldsm4(al, a_at(sb + Ly::Z2 + 2 * kGradRows * LD2, LD2, 16 * rg, kk));
      const uint32_t o = aW2 + 2u * (uint32_t)((16 * kk + bro) * LD2 + 32 * cq + bco);
      ldsm4t(r0, o);
      ldsm4t(r1, o + 32);
      mma16816(z1[0], ah, r0[0], r0[1]);
      mma16816(z1[1], ah, r0[2], r0[3]);
      mma16816(z1[2], ah, r1[0], r1[1]);
      mma16816(z1[3], ah, r1[2], r1[3]);
      mma16816(z1[0], al, r0[0], r0[1]);
      mma16816(z1[1], al, r0[2], r0[3]);
      mma16816(z1[2], al, r1[0], r1[1]);
      mma16816(z1[3], al, r1[2], r1[3]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int q = 0; q < 4; ++q) z1[j][q] *= 1.f - h1[j][q] * h1[j][q];
      s2[2 * j] = z1[j][0] + z1[j][2];
      s2[2 * j + 1] = z1[j][1] + z1[j][3];
      put(Ly::Z1, j, z1[j]);
    }
    colsum(gb1, s2);
    __syncthreads();
    // ---- dW2 += dz2^T h1 and dW1 += dz1^T xn, K = the tile's rows.  A tile's products
    // start from zero and are added in FP32: the tensor core truncates its
    // accumulator, which over hundreds of rows is a bias
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      float c[4][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) c[j][0] = c[j][1] = c[j][2] = c[j][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < kGradRows / 16; ++kk) {
        uint32_t ah[4], al[4];
        uint32_t o = sb + Ly::Z2 + 2u * (uint32_t)((16 * kk + tro) * LD2 + 16 * jb + tco);
        ldsm4t(ah, o);
        ldsm4t(al, o + 2 * kGradRows * LD2);
        o = sb + Ly::H1 + 2u * (uint32_t)((16 * kk + bro) * LD2 + 64 * kb + 32 * half + bco);
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
          uint32_t bh[4], bl[4];
          ldsm4t(bh, o + 16 * j);
          ldsm4t(bl, o + 16 * j + 2 * kGradRows * LD2);
          mma16816(c[j], ah, bh[0], bh[1]);
          mma16816(c[j + 1], ah, bh[2], bh[3]);
          mma16816(c[j], ah, bl[0], bl[1]);
          mma16816(c[j + 1], ah, bl[2], bl[3]);
          mma16816(c[j], al, bh[0], bh[1]);
          mma16816(c[j + 1], al, bh[2], bh[3]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) gW2[4 * half + j][q] += c[j][q];
    }
    {
      float c[NT1][4];
#pragma unroll
      for (int j = 0; j < NT1; ++j) c[j][0] = c[j][1] = c[j][2] = c[j][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < kGradRows / 16; ++kk) {
        uint32_t ah[4], al[4];
        uint32_t o = sb + Ly::Z1 + 2u * (uint32_t)((16 * kk + tro) * LD2 + 16 * jb + tco);
        ldsm4t(ah, o);
        ldsm4t(al, o + 2 * kGradRows * LD2);
        o = sb + Ly::X + 2u * (uint32_t)((16 * kk + (lane & 15)) * LD1 + 8 * NT1 * kb);
#pragma unroll
        for (int j = 0; j < NT1; ++j) {
          uint32_t bh[2], bl[2];
          ldsm2t(bh, o + 16 * j);
          ldsm2t(bl, o + 16 * j + 2 * kGradRows * LD1);
          mma16816(c[j], ah, bh[0], bh[1]);
          mma16816(c[j], ah, bl[0], bl[1]);
          mma16816(c[j], al, bh[0], bh[1]);
        }
      }
#pragma unroll
      for (int j = 0; j < NT1; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) gW1[j][q] += c[j][q];
    }
  }
  // the CTA's partial gradient, in the order of the parameters, made in shared memory
  // (over the tile's buffers) and written by one bulk copy
  for (int o = 16; o > 0; o >>= 1) {
    l2 += __shfl_xor_sync(0xffffffffu, l2, o);
    sdy += __shfl_xor_sync(0xffffffffu, sdy, o);
  }
  if (cq == 0 && lane == 0) {
    if (loss) atomicAdd(loss, l2 / (float)nrows);
    atomicAdd(gb3, sdy);
  }
  __syncthreads();
  float *P = reinterpret_cast<float *>(sm + Ly::X), *P2 = P + W * d + W;  // P2: 16-byte aligned
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = 64 * kb + 8 * j + 2 * t;
#pragma unroll
    for (int q = 0; q < 2; ++q)
      *reinterpret_cast<float2 *>(P2 + (16 * jb + g + 8 * q) * W + k) =
          make_float2(gW2[j][2 * q], gW2[j][2 * q + 1]);
  }
#pragma unroll
  for (int j = 0; j < NT1; ++j) {
    const int k = 8 * (NT1 * kb + j) + 2 * t;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (k + (q & 1) < d) P[(16 * jb + g + 8 * (q >> 1)) * d + k + (q & 1)] = gW1[j][q];
  }
  if (tid < W) {
    auto sum4 = [&](const float *v) { return (v[tid] + v[W + tid]) + (v[2 * W + tid] + v[3 * W + tid]); };
    P[W * d + tid] = sum4(gb1);
    P2[W * W + tid] = sum4(gb2);
    P2[W * W + W + tid] = sum4(gw3);
  }
  if (tid < 4) P2[W * W + 2 * W + tid] = tid == 0 ? *gb3 : 0.f;  // and the padding
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (tid == 0) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                     part + (long long)blockIdx.x * part_stride(d)),
                 "r"(sb + Ly::X), "r"(part_stride(d) * 4)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // shared memory is read
  }
}

// g = sum of the partial gradients; with adam, the update of k_mlp_adam on top instead
// (M.g is not touched).  64 parameters per CTA, the partials in four interleaved groups.
//
// The blocks are resident while the gradient kernel still writes `part` (pdl_launch), so
// the partials change during this kernel's life: they are read after pdl_wait through L2
// (__ldcg), never through the read-only path that a __restrict__ pointer to constant
// data allows.
__global__ void __launch_bounds__(256) k_mlp_tc_reduce(MlpDev M, int np, int nparts,
                                                       const float *part, int adam,
                                                       float lr, float b1, float b2, float eps,
                                                       int step, int k1,
                                                       unsigned char *__restrict__ im) {
  __shared__ float sh[4][64];
  const int c = threadIdx.x & 63, grp = threadIdx.x >> 6, q = blockIdx.x * 64 + c;
  float s = 0.f;
  pdl_launch();
  pdl_wait();
  if (q < np) {
#pragma unroll 8
    for (int k = grp; k < nparts; k += 4) s += __ldcg(part + (long long)k * part_stride(M.d) + q);
  }
  sh[grp][c] = s;
  __syncthreads();
  if (grp || q >= np) return;
  const float g = (sh[0][c] + sh[1][c]) + (sh[2][c] + sh[3][c]);
  if (!adam) {
    M.g[q] = g;
    return;
  }
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  const float m = b1 * M.m[q] + (1.f - b1) * g;
  const float v = b2 * M.v[q] + (1.f - b2) * g * g;
  M.m[q] = m;
  M.v[q] = v;
  const float w = M.p[q] - lr * (m / c1) / (sqrtf(v / c2) + eps);
  M.p[q] = w;
  image_put(im, M.d, k1, q, w);  // for the next step
}

template <int K1>
cudaError_t infer_k(const MlpDev &M, const float *x, int n, float *y, cudaStream_t s) {
  cudaError_t e = smem_optin_once<k_mlp_tc_infer<K1>>();
  if (e != cudaSuccess) return e;
  const size_t sm = (size_t)W * (K1 + 8) * 2 + (size_t)W * LD2 * 2 + (3 * W + 4 * K1) * sizeof(float) +
                    (size_t)kRowsPerCta * M.d * sizeof(float);
  const int tiles = (n + kRowsPerCta - 1) / kRowsPerCta;
  k_mlp_tc_infer<K1><<<std::min(tiles, 2 * 152), kThreads, sm, s>>>(M, x, n, y);
  return cudaGetLastError();
}

template <int K1>
cudaError_t grad_k(const MlpDev &M, const float *x, const float *t, int n, int nrows, int sampled,
                   uint64_t seed, int step, const unsigned char *im, float *part, int nparts,
                   float *loss, cudaStream_t s) {
  cudaError_t e = smem_optin_once<k_mlp_tc_grad<K1>>();
  if (e != cudaSuccess) return e;
  return launch_pdl(k_mlp_tc_grad<K1>, nparts, kGradThreads, GradLay<K1>::bytes, s, M, x, t, n, nrows,
                    sampled, (unsigned long long)seed, step, im, part, loss);
}

}  // namespace

bool mlp_tc_supported(int d, int w) { return w == W && d >= 1 && d <= 64; }

cudaError_t mlp_tc_infer(const MlpDev &M, const float *x, int n, float *y, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  switch ((M.d + 15) / 16 * 16) {
    case 16: return infer_k<16>(M, x, n, y, s);
    case 32: return infer_k<32>(M, x, n, y, s);
    case 48: return infer_k<48>(M, x, n, y, s);
    default: return infer_k<64>(M, x, n, y, s);
  }
}

size_t mlp_tc_image_bytes(int d) { return image_bytes((d + 15) / 16 * 16); }

cudaError_t mlp_tc_image(const MlpDev &M, unsigned char *im, cudaStream_t s) {
  const int np = M.w * M.d + M.w + M.w * M.w + M.w + M.w + 1;
  k_mlp_tc_image<<<(np + 255) / 256, 256, 0, s>>>(M, (M.d + 15) / 16 * 16, np, im);
  return cudaGetLastError();
}

size_t mlp_tc_part_bytes(int d) { return (size_t)part_stride(d) * sizeof(float); }

int mlp_tc_parts(int nrows) { return std::min((nrows - 1) / kGradRows + 1, 152); }

cudaError_t mlp_tc_grad(const MlpDev &M, const float *x, const float *t, int n, int nrows, int sampled,
                        uint64_t seed, int step, const unsigned char *im, float *part, float *loss,
                        cudaStream_t s) {
  const int np = mlp_tc_parts(nrows);
  switch ((M.d + 15) / 16 * 16) {
    case 16: return grad_k<16>(M, x, t, n, nrows, sampled, seed, step, im, part, np, loss, s);
    case 32: return grad_k<32>(M, x, t, n, nrows, sampled, seed, step, im, part, np, loss, s);
    case 48: return grad_k<48>(M, x, t, n, nrows, sampled, seed, step, im, part, np, loss, s);
    default: return grad_k<64>(M, x, t, n, nrows, sampled, seed, step, im, part, np, loss, s);
  }
}

cudaError_t mlp_tc_reduce(const MlpDev &M, int nparts, const float *part, int adam, float lr, float b1,
                          float b2, float eps, int step, unsigned char *im, cudaStream_t s) {
  const int np = M.w * M.d + M.w + M.w * M.w + M.w + M.w + 1;
  return launch_pdl(k_mlp_tc_reduce, (np + 63) / 64, 256, 0, s, M, np, nparts, part, adam, lr, b1, b2,
                    eps, step, (M.d + 15) / 16 * 16, im);
}

}  // namespace bsi
