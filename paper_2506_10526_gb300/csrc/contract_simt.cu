// Triple contraction of Eq. (estimator_t), plain FP32 path (SIMT FMA):
//
//   S(i nu1, j nu2, l nu3) = sum_x F_{i,nu1}(x) F_{j,nu2}(x) F_{l,nu3}(x)
//
// cast as a GEMM: rows are channel pairs (nu1, nu2) of a ring pair (i, j)
// whose pair operand P(x) = F_{i,nu1}(x) F_{j,nu2}(x) is formed on the fly in
// registers; columns are fields (l, nu3) with l >= j and T(i, j, l) > 0;
// K runs over the M^2 image pixels.  One launch covers every image side and
// ring pair of a call: a block finds its work item (realisation, K segment, pair
// rectangle, column window) from its index in the tile list, whose entries are
// sorted by cost.
//
// CTA tile: 128 H rows = H rectangles of 16 (nu1) x 8 (nu2), 128 / H columns;
// 256 threads, 8 x 8 accumulators each.  H = 1, 2 or 4 is chosen per column list
// so that the least of the tile is padding: the lists of a few channels and image
// sides hold 16 to 100 columns, and all three forms do the same 16384 products
// per pixel.
//
// The FP32 FMA pipe bounds the kernel: per pixel a thread issues 64 products
// as 32 packed FMAs (fma.rn.f32x2: two rows, the same rounding as two FMAs) and
// 8 multiplications for the pair operand; packing leaves issue slots for the
// shared loads.  Rows of 32 pixels arrive by 16-byte asynchronous copies in the
// fields' own order (pixel fastest, pitch 36 floats: 8 columns of a load on 8
// different bank groups) in a four-stage ring, with one barrier per 32 pixels.
// The kernel it replaced transposed every 16-pixel chunk through scalar stores
// with 4-way bank conflicts, kept the pair operand in shared memory and stopped at
// three barriers per chunk.  32 channels, 256^2 grid, 20 rings, ten image sides:
// 28.4 ms, 121.4 before (1.45e12 FLOP: 51 and 12 TFLOP/s of the 76.6 measured; the
// rest is padding of the tiles); 27 channels, 90^2 grid, 7 rings, two
// realisations: 4.0 ms, 9.3 before.
//
// Partial sums are FP32, folded into a second FP32 set (in shared memory) every
// 1024 pixels: two-level summation bounds the rounding growth over long K.  The
// K range can be split across CTAs; tile results meet in FP64 global atomics:
//   FULL  out[b][trip][nu1][nu2][nu3] += S / (A M^2 T(trip))
//   DELTA dsum[b][trip][nu1-nu3][nu2-nu3] += S, after a shared-memory
//         pre-reduction of each 16 x 8 rectangle keyed by (segment of equal trip,
//         nu1-nu2, nu2-nu3).
#include <algorithm>

#include "bs_internal.h"

namespace bsi {

namespace {

constexpr int TR1 = 16, TR2 = 8, KC = 32, NST = 4;
constexpr int PITCH = KC + 4;    // floats per staged row
constexpr int KOUTER = 1024 / KC;  // stages between folds into the outer accumulators
constexpr int RED_CAP = 6144;    // floats of one rectangle's DELTA pre-reduction buffer
constexpr int MAX_SEG = 64;
constexpr int kSimtThreads = 256;
constexpr int kStageFloats = (TR1 + TR2 + 128) * PITCH;  // the widest form, H = 1
constexpr int kOuterFloats = 64 * kSimtThreads;
constexpr size_t kSimtSmem = (size_t)(NST * kStageFloats + kOuterFloats) * sizeof(float);
static_assert(4 * RED_CAP <= NST * kStageFloats + kOuterFloats, "reduction buffers alias the ring");

__device__ __forceinline__ uint64_t pk(float a, float b) {
  return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}
__device__ __forceinline__ float lo_f(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_f(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

struct ColInfo {
  int field[128], trip[128], nu3[128], seg[128];
  int seg_trip[MAX_SEG], seg_base[MAX_SEG], seg_e[MAX_SEG], seg_hi[MAX_SEG];
  int nseg, total;
};

template <int H, bool FULL, bool DELTA>
__device__ __forceinline__ void simt_tile(const ContractArgs &a, const SimtTile &pt, long long local,
                                          float *sm, ColInfo &ci) {
  constexpr int NCOL = 128 / H, TX = NCOL / 8, NR = TR1 + TR2 * H + NCOL;
  constexpr int STAGE = NR * PITCH, NCP = (NR * (KC / 4) + kSimtThreads - 1) / kSimtThreads;
  // column of staged row r: a thread's columns are runs of four (c & 3 = its step), so
  // the reduction below adds an entry's terms by c & 3 within a row of the pair
  // rectangle, whatever H; staged so that a load's 8 rows are adjacent
  auto col_of = [](int r) { return 4 * (r % TX) + (r / TX & 3) + 4 * TX * (r / TX >> 2); };
  const int tid = threadIdx.x;
  const int n_r1 = (a.nu1_hi - a.nu1_lo + TR1 - 1) / TR1;
  const int n_r2 = (a.nu2_hi - a.nu2_lo + TR2 * H - 1) / (TR2 * H);
  const int rt = (int)(local % (n_r1 * n_r2)), z = (int)(local / (n_r1 * n_r2));
  const int nu1_0 = a.nu1_lo + (rt / n_r2) * TR1, nu2_0 = a.nu2_lo + (rt % n_r2) * TR2 * H;
  const SimtLevel &lv = a.lev[pt.level];
  const int kseg = z % pt.nk, b = z / pt.nk;
  const int k0 = kseg * pt.kseg_len, k1 = min(lv.M2, k0 + pt.kseg_len);
  const float *Fb = lv.F + (long long)b * lv.bstride;

  __syncthreads();  // the previous item's readers are done with ci and sm
  for (int c = tid; c < NCOL; c += kSimtThreads) {
    const int cc = pt.col0 + c;
    ColEntry e{-1, -1, 0, 0};
    if (cc < pt.ncol) e = a.cols[pt.col_off + cc];
    ci.field[c] = e.field;
    ci.trip[c] = e.trip;
    ci.nu3[c] = e.nu3;
  }
  __syncthreads();
  if (DELTA && tid < 32) {
    // segments of consecutive columns with the same ring triple (nu3 ascends within one)
    int ns = 0;
    for (int c0 = 0; c0 < NCOL; c0 += 32) {
      const int c = c0 + tid;
      const bool live = ci.field[c] >= 0;
      const bool start = live && (c == 0 || ci.trip[c] != ci.trip[c - 1]);
      const unsigned m = __ballot_sync(0xffffffffu, start);
      const int sg = ns + __popc(m & (0xffffffffu >> (31 - tid))) - 1;
      ci.seg[c] = sg;
      if (start && sg < MAX_SEG) {
        ci.seg_trip[sg] = ci.trip[c];
        ci.seg_base[sg] = ci.nu3[c];  // its lowest nu3, until the bases are summed below
      }
      const bool last = live && (c == NCOL - 1 || ci.field[c + 1] < 0 || ci.trip[c + 1] != ci.trip[c]);
      if (last && sg < MAX_SEG) ci.seg_hi[sg] = ci.nu3[c];
      ns += __popc(m);
    }
    __syncwarp();
    if (tid == 0) {
      int base = 0;
      for (int sg = 0; sg < min(ns, MAX_SEG); ++sg) {
        const int e = (TR2 - 1) + (ci.seg_hi[sg] - ci.seg_base[sg]) + 1;
        ci.seg_base[sg] = base;
        ci.seg_e[sg] = e;
        base += (TR1 + TR2 - 1) * e;
      }
      ci.nseg = min(ns, MAX_SEG);
      ci.total = ns > MAX_SEG ? RED_CAP + 1 : base;  // too many segments: direct atomics
    }
  }

  // this thread's 16-byte pieces of a stage: staged row r (F_i rows, F_j rows,
  // columns), pixels 4 (q & 7); rows without a field are filled with zeros
  const float *src[NCP];
  uint32_t dst[NCP];
  bool have[NCP];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sm);
#pragma unroll
  for (int m = 0; m < NCP; ++m) {
    const int q = tid + m * kSimtThreads, r = q >> 3;
    long long f = -1;
    if (r < TR1) {
      if (nu1_0 + r < a.nu1_hi) f = (long long)pt.ri * a.nc + nu1_0 + r;
    } else if (r < TR1 + TR2 * H) {
      const int nu2 = nu2_0 + r - TR1;
      if (nu2 < a.nu2_hi) f = (long long)pt.rj * a.nc + nu2;
    } else if (r < NR) {
      f = ci.field[col_of(r - TR1 - TR2 * H)];
    }
    have[m] = f >= 0;
    src[m] = Fb + (f >= 0 ? f * lv.M2 : 0) + 4 * (q & 7);
    dst[m] = sbase + 4u * (uint32_t)(r * PITCH + 4 * (q & 7));
  }
  auto load = [&](int st) {
    const int k = k0 + st * KC;
    if (k < k1) {
      const uint32_t o = 4u * (uint32_t)((st % NST) * STAGE);
#pragma unroll
      for (int m = 0; m < NCP; ++m) {
        if (NR * (KC / 4) % kSimtThreads && tid + m * kSimtThreads >= NR * (KC / 4)) continue;
        const bool in = have[m] && k + 4 * ((tid + m * kSimtThreads) & 7) < k1;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst[m] + o),
                     "l"(in ? src[m] + k : Fb), "r"(in ? 16 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const int tx = tid % TX, ty = tid / TX;
  const int half = ty >> 4, tyl = ty & 15;
  const int i0 = tyl >> 1, j0 = TR2 * half + 4 * (tyl & 1);  // rows (i0, j0 + y), (i0 + 8, j0 + y)
  uint64_t acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0;
  uint64_t *outer = reinterpret_cast<uint64_t *>(sm + NST * kStageFloats) + tid;
  bool folded = false;

  const int nst = (k1 - k0 + KC - 1) / KC;
#pragma unroll
  for (int s = 0; s < NST - 1; ++s) load(s);
  for (int st = 0; st < nst; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(NST - 2) : "memory");
    __syncthreads();
    load(st + NST - 1);
    const float *S = sm + (st % NST) * STAGE;
    const float *Si = S + i0 * PITCH, *Sj = S + (TR1 + j0) * PITCH,
                *Sc = S + (TR1 + TR2 * H + tx) * PITCH;
#pragma unroll 2
    for (int q = 0; q < KC / 4; ++q) {
      float fi[2][4], fj[4][4], fc[8][4];
#pragma unroll
      for (int y = 0; y < 2; ++y)
        *reinterpret_cast<float4 *>(fi[y]) =
            *reinterpret_cast<const float4 *>(Si + 8 * y * PITCH + 4 * q);
#pragma unroll
      for (int y = 0; y < 4; ++y)
        *reinterpret_cast<float4 *>(fj[y]) = *reinterpret_cast<const float4 *>(Sj + y * PITCH + 4 * q);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        *reinterpret_cast<float4 *>(fc[u]) =
            *reinterpret_cast<const float4 *>(Sc + TX * u * PITCH + 4 * q);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint64_t P[4];
#pragma unroll
        for (int y = 0; y < 4; ++y)
          P[y] = pk(fi[y >> 1][k] * fj[2 * (y & 1)][k], fi[y >> 1][k] * fj[2 * (y & 1) + 1][k]);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint64_t cc = pk(fc[u][k], fc[u][k]);
#pragma unroll
          for (int y = 0; y < 4; ++y) acc[y][u] = fma2(P[y], cc, acc[y][u]);
        }
      }
    }
    if ((st + 1) % KOUTER == 0) {
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          uint64_t *o = outer + (y * 8 + u) * kSimtThreads;
          *o = folded ? add2(*o, acc[y][u]) : acc[y][u];
          acc[y][u] = 0;
        }
      folded = true;
    }
  }
  if (folded) {
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int u = 0; u < 8; ++u) acc[y][u] = add2(outer[(y * 8 + u) * kSimtThreads], acc[y][u]);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();  // the ring and the outer sums are free

  const bool use_red = DELTA && ci.total <= RED_CAP;
  float *red = sm + half * RED_CAP;
  if (use_red) {
    for (int q = tid; q < H * ci.total; q += kSimtThreads)
      sm[(q / ci.total) * RED_CAP + q % ci.total] = 0.f;
    __syncthreads();
  }
#pragma unroll
  for (int y = 0; y < 8; ++y) {  // row (i0 + 8 (y >> 2), j0 + (y & 3))
    const int nu1 = nu1_0 + i0 + 8 * (y >> 2), nu2 = nu2_0 + j0 + (y & 3);
    if (nu1 >= a.nu1_hi || nu2 >= a.nu2_hi) continue;
#pragma unroll
    for (int step = 0; step < 8; ++step) {
      const int u = H == 1 ? step : (step >> 1) + 4 * (step & 1);
      const int c = col_of(tx + TX * u);
      if (ci.field[c] < 0) continue;
      const uint64_t v = acc[(y >> 2) * 2 + ((y & 3) >> 1)][u];
      const float s = (y & 1) ? hi_f(v) : lo_f(v);
      const int trip = ci.trip[c], nu3 = ci.nu3[c];
      if (FULL) {
        const long long o = (long long)b * a.full_bstride +
                            (((long long)trip * a.nc + nu1) * a.nc + nu2) * a.nc + nu3;
        atomicAdd(a.out_full + o, (double)s * a.tnorm[trip]);
      }
      if (DELTA) {
        if (use_red) {
          const int sg = ci.seg[c];
          const int d = (i0 + 8 * (y >> 2)) - (j0 - TR2 * half + (y & 3)) + (TR2 - 1);
          const int e = (j0 - TR2 * half + (y & 3)) + ci.seg_hi[sg] - nu3;
          atomicAdd(&red[ci.seg_base[sg] + d * ci.seg_e[sg] + e], s);
        } else {
          const int n2 = 2 * a.nc - 1;
          const long long o = (long long)b * a.dsum_bstride +
                              ((long long)trip * n2 + (nu1 - nu3 + a.nc - 1)) * n2 +
                              (nu2 - nu3 + a.nc - 1);
          atomicAdd(a.dsum + o, (double)s);
        }
      }
    }
  }
  if (use_red) {
    __syncthreads();
    const int n2 = 2 * a.nc - 1;
    for (int r = tid; r < H * ci.total; r += kSimtThreads) {
      const int hh = r / ci.total, q = r - hh * ci.total;
      const float v = sm[hh * RED_CAP + q];
      if (v == 0.f) continue;
      int sg = 0;
      while (sg + 1 < ci.nseg && ci.seg_base[sg + 1] <= q) ++sg;
      const int off = q - ci.seg_base[sg], E = ci.seg_e[sg];
      const int d = off / E;
      const int d2 = off - d * E + nu2_0 + TR2 * hh - ci.seg_hi[sg];
      const int d1 = d + nu1_0 - nu2_0 - TR2 * hh - (TR2 - 1) + d2;
      const long long o = (long long)b * a.dsum_bstride +
                          ((long long)ci.seg_trip[sg] * n2 + (d1 + a.nc - 1)) * n2 + (d2 + a.nc - 1);
      atomicAdd(a.dsum + o, (double)v);
    }
  }
}

template <bool FULL, bool DELTA>
__global__ void __launch_bounds__(kSimtThreads, 1)
    k_contract_simt(const __grid_constant__ ContractArgs a) {
  extern __shared__ __align__(16) float simt_sm[];
  __shared__ ColInfo ci;
  for (long long item = blockIdx.x; item < a.nitem; item += gridDim.x) {
    int lo = 0, hi = a.ntile - 1;  // the last entry with first <= item
    while (lo < hi) {
      const int m = (lo + hi + 1) >> 1;
      if (a.tiles[m].first <= item) lo = m; else hi = m - 1;
    }
    const SimtTile pt = a.tiles[lo];
    const long long local = item - pt.first;
    if (pt.h == 1)
      simt_tile<1, FULL, DELTA>(a, pt, local, simt_sm, ci);
    else if (pt.h == 2)
      simt_tile<2, FULL, DELTA>(a, pt, local, simt_sm, ci);
    else
      simt_tile<4, FULL, DELTA>(a, pt, local, simt_sm, ci);
  }
}

template <bool FULL, bool DELTA>
cudaError_t launch(const ContractArgs &a, cudaStream_t s) {
  cudaError_t e = smem_optin_once<k_contract_simt<FULL, DELTA>>();
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)std::min<long long>(a.nitem, 0x7fffffffLL);
  k_contract_simt<FULL, DELTA><<<grid, kSimtThreads, kSimtSmem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

// The form of a column list: the least number of tiles (each is 16384 products a
// pixel); the widest one on ties, whose reduction adds the fewest terms in FP32.
int simt_form(int n_nu1, int n_nu2, int ncol) {
  int best = 1;
  long long cost = 0;
  for (int h = 1; h <= 4; h *= 2) {
    const long long n = (long long)((n_nu1 + TR1 - 1) / TR1) * ((n_nu2 + TR2 * h - 1) / (TR2 * h)) *
                        ((ncol + 128 / h - 1) / (128 / h));
    if (h == 1 || n < cost) {
      cost = n;
      best = h;
    }
  }
  return best;
}

cudaError_t launch_contract_simt(const ContractArgs &a, cudaStream_t s) {
  if (a.nitem == 0) return cudaSuccess;
  const bool full = a.out_full != nullptr, delta = a.dsum != nullptr;
  if (full && delta) return launch<true, true>(a, s);
  if (full) return launch<true, false>(a, s);
  if (delta) return launch<false, true>(a, s);
  return cudaSuccess;
}

}  // namespace bsi
