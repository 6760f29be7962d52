// Triple contraction on the tensor cores for short column lists: the sums, the
// operand splits, the tile list and the order of every FP32 accumulation are those
// of contract_tc.cu; the roles of the two GEMM operands are exchanged.
//
//   rows (M = 2 x 128)   channel pairs: 16 nu1 x 16 nu2, two MMAs of 128 rows
//   columns (N <= 128)   fields (l, nu3) of the column list
//   K                    image pixels in stages of 32
//
// contract_tc.cu multiplies 256 fields x 512 pairs per tile and pays for all of
// them: with 16 channels a list holds 16 to 128 fields and a rectangle 256 pairs,
// and a tenth of its tensor work was used (271 us for the 64^2 x 16 channel grid,
// 27.5 ms for 256 such fields at once).  Here the tile is exact to 16 fields and 256
// pairs: 118 us, and 5.4 ms.
//
// The pair operand lives in tensor memory: a producer lane owns one row (pair) of
// each MMA and stores its hi and lo parts with tcgen05.st, so the operand costs no
// shared-memory bandwidth in either direction.  Per stage of 32 pixels the MMAs take 6
// cycles a field; the producers (8192 products and splits, about 1100 warp
// instructions at the 0.42 a cycle and scheduler that their chains allow) take 750 to
// 1000, which is what bounds it.  Four groups of four producer warps work on four
// stages at once, since a stage's latency (row loads, products, tensor-memory
// stores, MMAs, commit) is several times that.
//
// Work item: one 128-field half of a tile of the list (the fields one CTA of
// contract_tc.cu's pair would take) x its 32 x 16 pair rectangle x its K segment, as
// two sub-tiles: pair halves nu1_0 + 16.., then nu1_0...  Each (ring triple,
// nu1 - nu2, nu2 - nu3) entry of the item is summed in FP32 in that order, pairs
// ascending -- the order in which contract_tc.cu's lanes reach it, up to races between
// its warps -- and enters the FP64 collapse sums once.
//
// Roles (672 threads): warps 0-15 producers (group w / 4 makes every fourth stage;
// warp w has TMEM lanes 32 (w % 4)..) and epilogue; warps 16 and 20 TMA of the fields'
// hi and lo parts; warps 17 and 19 a thread each for the two MMAs, warp 17 also the
// TMEM allocation; warp 18 TMA of the producers' FP32 rows.  One thread issues an MMA
// or a copy every 40 to 100 cycles, which one thread for all of a kind made the
// stage's length for short lists.
//
// Tensor memory (512 columns): accumulators [0, 128) and [128, 256); stage s of the
// pair operand at 256 + 64 s: per MMA 16 columns hi, 16 lo (two pixels a column).
//
// Every wait is bounded as in contract_tc.cu.
#include <algorithm>
#include <unordered_map>

#include "bs_internal.h"
#include "tc_ptx.cuh"

namespace bsi {

namespace {

using namespace tc;

constexpr int KC = 32, MROWS = 128, P1 = 32, P2 = 16;
constexpr int NGRPW = 4;                 // producer groups of four warps
constexpr int NPROD = 4 * NGRPW, NTHREADS = 32 * (NPROD + 5), EPI = 32 * NPROD;
constexpr int BST = 5, RST = 8, AST = NGRPW;  // ring depths: fields, FP32 rows, pair operand
constexpr int GROUP = 8, NGRP = MROWS / GROUP;
constexpr int B_BYTES = MROWS * KC * 2;  // 8 KB: hi or lo
constexpr int RAW_BYTES = 32 * KC * 4;   // 4 KB: 16 rows of F_i, 16 of F_j
constexpr int TPITCH = 257;              // floats per field of the epilogue's tile
constexpr int TFLOATS = 16 * TPITCH;
constexpr int RED_CAP = 12544;           // floats of the reduction buffer
constexpr int TMEM_A = 256, TMEM_COLS = 512;
constexpr int NBAR = 2 * BST + 2 * RST + 2 * AST + 5;

constexpr int OFF_B = 0;
constexpr int OFF_RAW = OFF_B + BST * 2 * B_BYTES;
constexpr int OFF_T = OFF_RAW + RST * RAW_BYTES;
constexpr int OFF_RED = OFF_T + 2 * TFLOATS * 4;
constexpr int OFF_COL = OFF_RED + RED_CAP * 4;
constexpr int OFF_GRP = OFF_COL + MROWS * 16;
constexpr int OFF_SEG = OFF_GRP + NGRP * 16;
constexpr int OFF_SSC = OFF_SEG + NGRP * 16;
constexpr int OFF_BAR = OFF_SSC + NGRP * 8;
constexpr int OFF_BOX = (OFF_BAR + NBAR * 8 + 15) / 16 * 16;
constexpr int OFF_MISC = OFF_BOX + 2 * 16 * 16;
constexpr int SMEM_BYTES = OFF_MISC + 32 + 1024;
static_assert(OFF_RAW % 1024 == 0 && OFF_COL % 16 == 0 && OFF_BAR % 8 == 0,
              "alignment of the swizzled, int4 and barrier areas");
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory of one CTA");

__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc,
                                       uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
__device__ __forceinline__ void st8(uint32_t taddr, const uint32_t *r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
// Two products and their split, with packed FP32 operations (the same roundings as
// split2 / split2_f16 of contract_tc.cu).
__device__ __forceinline__ uint64_t pk(float a, float b) {
  return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}
template <bool F16>
__device__ __forceinline__ void pair_split(uint64_t fi, uint64_t fj, uint32_t &hi, uint32_t &lo) {
  uint64_t v, r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(fi), "l"(fj));
  const float v0 = __uint_as_float((uint32_t)v), v1 = __uint_as_float((uint32_t)(v >> 32));
  if constexpr (F16) {
    const __half2 h = __floats2half2_rn(v0, v1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    const float2 hf = __half22float2(h);
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(v), "l"(pk(-hf.x, -hf.y)));
    const __half2 l = __floats2half2_rn(__uint_as_float((uint32_t)r), __uint_as_float((uint32_t)(r >> 32)));
    lo = *reinterpret_cast<const uint32_t *>(&l);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    const uint64_t hf = (uint64_t)(hi << 16) | ((uint64_t)(hi & 0xffff0000u) << 32);
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(hf), "l"(pk(-1.f, -1.f)), "l"(v));
    const __nv_bfloat162 l =
        __floats2bfloat162_rn(__uint_as_float((uint32_t)r), __uint_as_float((uint32_t)(r >> 32)));
    lo = *reinterpret_cast<const uint32_t *>(&l);
  }
}
__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
      " [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// What every role derives from an item: the tile, its fields and sub-tiles.
struct Item {
  TcTile t;
  int cbase, nrow, pa_hi, pb_hi, dmax, k0, k1;
  __device__ __forceinline__ bool load(const TcArgs &a, int item) {
    t = a.tiles[item % a.ntiles];
    const TcGroup &G = a.groups[t.group];
    cbase = t.col0 + MROWS * (item / a.ntiles);
    nrow = min(MROWS, t.ncol - cbase);
    if (nrow <= 0) return false;
    pa_hi = min(P1, G.nu1_hi - t.nu1_0);
    pb_hi = min(P2, G.nu2_hi - t.nu2_0);
    dmax = t.diag ? t.nu2_0 - t.nu1_0 : P1;
    k0 = t.kseg * G.kseg_len;
    k1 = min(G.Kpad, k0 + G.kseg_len);
    return true;
  }
  // a pair half with pairs in the block and on the kept side of the diagonal
  __device__ __forceinline__ bool half(int h) const {
    return 16 * h < pa_hi && 16 * h - (pb_hi - 1) <= dmax;
  }
  // fields, rounded to the MMA's granularity
  __device__ __forceinline__ int width() const { return (nrow + 15) & ~15; }
};

template <bool F16>
__global__ void __launch_bounds__(NTHREADS, 1) k_contract_tcs(const __grid_constant__ TcArgs a) {
  extern __shared__ unsigned char smem_dyn[];
  unsigned char *sm = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const uint32_t sB = smem_u32(sm + OFF_B), sRaw = smem_u32(sm + OFF_RAW);
  const uint32_t sBar = smem_u32(sm + OFF_BAR);
  auto b_full = [&](int s) { return sBar + 8 * s; };
  auto b_empty = [&](int s) { return sBar + 8 * (BST + s); };
  auto raw_full = [&](int s) { return sBar + 8 * (2 * BST + s); };
  auto raw_empty = [&](int s) { return sBar + 8 * (2 * BST + RST + s); };
  auto a_full = [&](int s) { return sBar + 8 * (2 * BST + 2 * RST + s); };
  auto a_empty = [&](int s) { return sBar + 8 * (2 * BST + 2 * RST + AST + s); };
  const uint32_t acc_full = sBar + 8 * (2 * BST + 2 * RST + 2 * AST), acc_empty = acc_full + 8,
                 stall_bar = acc_full + 16;
  auto done = [&](uint32_t q) { return acc_full + 24 + 8 * q; };  // an MMA thread's last commit
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sm + OFF_MISC);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(sm + OFF_MISC + 4);
  int *total_s = reinterpret_cast<int *>(sm + OFF_MISC + 8);
  int *nseg_s = reinterpret_cast<int *>(sm + OFF_MISC + 12);

  if (threadIdx.x == 0) {
    for (int s = 0; s < BST; ++s) {
      mbar_init(b_full(s), 2);
      mbar_init(b_empty(s), 2);
    }
    for (int s = 0; s < RST; ++s) {
      mbar_init(raw_full(s), 1);
      mbar_init(raw_empty(s), 4);
    }
    for (int s = 0; s < AST; ++s) {
      mbar_init(a_full(s), 4);
      mbar_init(a_empty(s), 2);
    }
    mbar_init(acc_full, 2);
    mbar_init(acc_empty, NPROD);
    mbar_init(stall_bar, 1);
    mbar_init(done(0), 1);
    mbar_init(done(1), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == NPROD + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const long long limit = a.wait_limit_ns;
  const int nitem = 2 * a.ntiles;
  const CUtensorMap *maps = reinterpret_cast<const CUtensorMap *>(a.maps);
  auto fail = [&]() {
    *abort_flag = 1;
    atomicExch(a.err, 1);
  };

  if (warp == NPROD + 2) {
    // ------------------------------------------------------------ TMA of the FP32 rows
    if (elect_one()) {
      uint32_t s = 0, ph = 1, armed = 0;
      bool ok = true;
      Item w;
      for (int item = blockIdx.x; item < nitem && ok; item += gridDim.x) {
        if (!w.load(a, item)) continue;
        const TcTile &t = w.t;
        const TcGroup &G = a.groups[t.group];
        const CUtensorMap *mr = maps + kTcMaps * t.group + 11;
        const int rowj = t.b * G.nf + t.rj * G.nc + t.nu2_0;
        for (int h = 1; h >= 0; --h) {
          if (!w.half(h)) continue;
          const int rowi = t.b * G.nf + t.ri * G.nc + t.nu1_0 + 16 * h;
          for (int kc = w.k0; kc < w.k1 && ok; kc += KC) {
            if (!mbar_wait(raw_empty(s), ph, limit, abort_flag)) {
              fail();
              ok = false;
              break;
            }
            const uint32_t d = sRaw + s * RAW_BYTES, bar = raw_full(s);
            mbar_expect_tx(bar, RAW_BYTES);
            tma_load_2d(d, mr, kc, rowi, bar);
            tma_load_2d(d + RAW_BYTES / 2, mr, kc, rowj, bar);
            ++armed;
            if (++s == RST) {
              s = 0;
              ph ^= 1;
            }
          }
        }
      }
      // copies in flight land before the CTA can exit
      volatile int never = 0;
      for (uint32_t n = armed > RST ? armed - RST : 0; n < armed; ++n)
        if (!mbar_wait(raw_full(n % RST), (n / RST) & 1, limit, &never)) atomicExch(a.err, 1);
    }
  } else if (warp == NPROD || warp == NPROD + 4) {
    // ------------------------------------------------------------ TMA of the fields (hi or lo)
    const int part = warp == NPROD ? 0 : 1;
    int4 *list = reinterpret_cast<int4 *>(sm + OFF_BOX) + 16 * part;
    uint32_t s = 0, ph = 1, armed = 0;
    bool ok = true;
    Item w;
    for (int item = blockIdx.x; item < nitem; item += gridDim.x) {
      if (!w.load(a, item)) continue;
      const TcTile &t = w.t;
      const TcGroup &G = a.groups[t.group];
      const int ng = w.width() / GROUP;
      // field rows of the 8-row groups; past the list: out of range, which TMA fills
      // with zeros
      const int e = w.cbase + (lane & 15) * GROUP;
      int f = -1;
      if (lane < ng && e < t.ncol) f = G.cols[t.col_off + e].field;
      const int nbox = box_list(maps + kTcMaps * t.group + part, f >= 0 ? t.b * G.nf + f : G.batch * G.nf,
                                lane < ng, list, lane);
      if (elect_one()) {
        const uint32_t bytes = ng * GROUP * KC * 2;
        const Boxes boxes(list, nbox);
        const int halves = (w.half(0) ? 1 : 0) + (w.half(1) ? 1 : 0);
        for (int h = 0; h < halves && ok; ++h)
          for (int kc = w.k0; kc < w.k1; kc += KC) {
            if (!mbar_wait(b_empty(s), ph, limit, abort_flag)) {
              fail();
              ok = false;
              break;
            }
            const uint32_t d = sB + s * 2 * B_BYTES + part * B_BYTES, bar = b_full(s);
            mbar_expect_tx(bar, bytes);
            boxes.load(d, kc, bar);
            ++armed;
            if (++s == BST) {
              s = 0;
              ph ^= 1;
            }
          }
      }
      __syncwarp();
    }
    // copies in flight land before the CTA can exit
    if (elect_one()) {
      volatile int never = 0;
      for (uint32_t n = armed > BST ? armed - BST : 0; n < armed; ++n)
        if (!mbar_wait(b_full(n % BST), (n / BST) & 1, limit, &never)) atomicExch(a.err, 1);
    }
  } else if (warp == NPROD + 1 || warp == NPROD + 3) {
    // ------------------------------------------------------------ MMA threads
    if (elect_one()) {
      const uint32_t mq = warp == NPROD + 1 ? 0 : 1, acc = tmem + mq * MROWS;
      const uint64_t desc0 = sw64_desc(sB);  // descriptors differ in the address field (16-byte units)
      uint32_t sa = 0, pha = 0, sb = 0, phb = 0, tc = 0;
      bool ok = true, issued = false;
      if (a.stall_test) {  // failure-injection test: a barrier nothing arrives at
        if (!mbar_wait(stall_bar, 0, limit, abort_flag)) {
          fail();
          ok = false;
        }
      }
      Item w;
      for (int item = blockIdx.x; item < nitem && ok; item += gridDim.x) {
        if (!w.load(a, item)) continue;
        const uint32_t n = (uint32_t)w.width();
        // instruction descriptor, kind::f16: D f32, A and B bf16 (1) or f16 (0), M = 128
        const uint32_t idesc = (1u << 4) | ((F16 ? 0u : 1u) << 7) | ((F16 ? 0u : 1u) << 10) |
                               ((n >> 3) << 17) | ((128u >> 4) << 24);
        const int halves = (w.half(0) ? 1 : 0) + (w.half(1) ? 1 : 0);
        for (int h = 0; h < halves && ok; ++h, ++tc) {
          if (!mbar_wait(acc_empty, (tc & 1) ^ 1, limit, abort_flag)) {
            fail();
            ok = false;
            break;
          }
          uint32_t more = 0;  // 0: the sub-tile's first MMA overwrites the accumulator
          for (int kc = w.k0; kc < w.k1; kc += KC) {
            if (!mbar_wait(b_full(sb), phb, limit, abort_flag) ||
                !mbar_wait(a_full(sa), pha, limit, abort_flag)) {
              fail();
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t dh = desc0 + (uint64_t)(sb * (2 * B_BYTES >> 4)), dl = dh + (B_BYTES >> 4);
            const uint32_t ah = tmem + TMEM_A + sa * 64 + mq * 32, al = ah + 16;
            mma_ts(acc, ah, dh, idesc, more);
            more = 1;
            mma_ts(acc, al, dh, idesc, 1u);
            mma_ts(acc, ah, dl, idesc, 1u);
            mma_ts(acc, ah + 8, dh + 2, idesc, 1u);  // pixels 16..31: 32 bytes on
            mma_ts(acc, al + 8, dh + 2, idesc, 1u);
            mma_ts(acc, ah + 8, dl + 2, idesc, 1u);
            commit(a_empty(sa));
            commit(b_empty(sb));
            issued = true;
            if (++sa == AST) {
              sa = 0;
              pha ^= 1;
            }
            if (++sb == BST) {
              sb = 0;
              phb ^= 1;
            }
          }
          if (ok) commit(acc_full);
        }
      }
      if (issued) {  // every MMA issued has finished before TMEM is freed
        volatile int never = 0;
        commit(done(mq));
        if (!mbar_wait(done(mq), 0, limit, &never)) atomicExch(a.err, 1);
      }
    }
  } else {
    // ------------------------------------------------------------ producers + epilogue
    const int pw = warp, ptid = threadIdx.x;
    const int quad = pw & 3, grpw = pw >> 2;  // TMEM lanes; producer group
    const unsigned char *rawb = sm + OFF_RAW;
    float *T = reinterpret_cast<float *>(sm + OFF_T);
    float *red = reinterpret_cast<float *>(sm + OFF_RED);
    ColEntry *colbuf = reinterpret_cast<ColEntry *>(sm + OFF_COL);
    int4 *grp = reinterpret_cast<int4 *>(sm + OFF_GRP);  // (segment, first nu3, fields, -)
    int4 *seginfo = reinterpret_cast<int4 *>(sm + OFF_SEG);  // (base, E | swapped << 16, trip, hi)
    double *segscale = reinterpret_cast<double *>(sm + OFF_SSC);  // 2^-(k_i+k_j+k_l)
    const uint32_t tlane = tmem + ((uint32_t)(32 * quad) << 16);
    const int pb_l = lane & 15, pa_l = 2 * quad + (lane >> 4);  // rows pa_l and 8 + pa_l of F_i
    // 16-byte chunk c of a swizzled row is at (its chunk 0) ^ 16 c
    const uint32_t oj = sw128_off(16 + pb_l, 0), oi0 = sw128_off(pa_l, 0), oi1 = sw128_off(8 + pa_l, 0);
    uint32_t it = 0, tc = 0;
    Item w;
    for (int item = blockIdx.x; item < nitem; item += gridDim.x) {
      if (!w.load(a, item)) continue;
      const TcTile &t = w.t;
      const TcGroup &G = a.groups[t.group];
      const int b = t.b;
      float sc_i = 1.f, sc_p = 1.f;  // split FP16: 2^(k_i + k_j), as in contract_tc.cu
      if constexpr (F16) {
        const int ki = G.kexp[b * G.nslot + t.ri], kj = G.kexp[b * G.nslot + t.rj];
        const int kij = ki + kj;
        if (kij >= -120 && kij <= 120) {
          sc_i = exp2i_f32(kij);
        } else {
          sc_i = exp2i_f32(ki);
          sc_p = exp2i_f32(kj);
        }
      }
      // the item's fields, in groups of 8 of one ring triple (runs of a list are
      // padded to 8); consecutive groups of one ring triple form a segment
      if (ptid < MROWS) {
        ColEntry ce{-2, 0, 0, 0};
        if (ptid < w.nrow) ce = G.cols[t.col_off + w.cbase + ptid];
        colbuf[ptid] = ce;
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
      const int npa = w.pa_hi > 16 ? 32 : 16;  // nu1 rows of the reduction's key range
      if (pw == 0) {
        const int g = lane & 15;
        const ColEntry c0 = colbuf[8 * g];
        int nv = 0;
        if (c0.field >= 0)
          for (int q = 0; q < 8; ++q) nv += colbuf[8 * g + q].field >= 0 ? 1 : 0;
        const int key = c0.field >= 0 ? 2 * c0.trip + c0.swapped : -1 - g;
        const int prev = __shfl_up_sync(0xffffffffu, key, 1);
        const bool live = lane < 16 && c0.field >= 0, start = live && (g == 0 || prev != key);
        const unsigned m = __ballot_sync(0xffffffffu, start);
        const int sg = __popc(m & (0xffffffffu >> (31 - lane))) - 1;
        const int next = __shfl_down_sync(0xffffffffu, key, 1);
        const bool last = live && (g == 15 || next != key);
        const unsigned ml = __ballot_sync(0xffffffffu, last);
        // per segment (lane sg): lo, hi
        const int nseg = __popc(m);
        const int gs = __fns(m, 0, min(lane, 15) + 1) & 31, ge = __fns(ml, 0, min(lane, 15) + 1) & 31;
        const int lo = __shfl_sync(0xffffffffu, c0.nu3, gs);
        const int hi = __shfl_sync(0xffffffffu, c0.nu3 + nv - 1, ge);
        const int E = lane < nseg ? (P2 - 1) + (hi - lo) + 1 : 0;
        int inc = (npa + P2 - 1) * E;
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += v;
        }
        const int trip = __shfl_sync(0xffffffffu, c0.trip, gs);
        const int sw = __shfl_sync(0xffffffffu, c0.swapped, gs);
        const int field = __shfl_sync(0xffffffffu, c0.field, gs);
        if (lane < nseg) {
          seginfo[lane] = make_int4(inc - (npa + P2 - 1) * E, E | (sw ? 1 << 16 : 0), trip, hi);
          double usc = 1.0;  // undoes the split-FP16 operand scales of this ring triple
          if constexpr (F16)
            usc = exp2i_f64(-(G.kexp[b * G.nslot + t.ri] + G.kexp[b * G.nslot + t.rj] +
                              G.kexp[b * G.nslot + field / G.nc]));
          segscale[lane] = usc;
        }
        if (lane < 16) grp[g] = make_int4(live ? sg : -1, c0.nu3, nv, 0);
        if (lane == 31) {
          *total_s = min(inc, RED_CAP);  // tcs_wins: never above RED_CAP
          *nseg_s = nseg;
        }
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
      for (int q = ptid; q < *total_s; q += EPI) red[q] = 0.f;

      for (int h = 1; h >= 0; --h) {
        if (!w.half(h)) continue;
        const uint32_t it0 = it, nst = (uint32_t)(w.k1 - w.k0) / KC;
        it += nst;
        // this group's stages of the sub-tile: it % AST == grpw
        for (uint32_t st = it0 + ((grpw - it0) & (AST - 1)); st < it; st += AST) {
          const int sr = st % RST;
          bool ok = !*abort_flag;
          if (ok && !mbar_wait(raw_full(sr), (st / RST) & 1, limit, abort_flag)) {
            fail();
            ok = false;
          }
          if (ok && !mbar_wait(a_empty(grpw), ((st / AST) & 1) ^ 1, limit, abort_flag)) {
            fail();
            ok = false;
          }
          ok = __all_sync(0xffffffffu, ok);
          if (ok) {
            tc_fence_after();
            const unsigned char *rb = rawb + sr * RAW_BYTES;
            const uint32_t o = tlane + TMEM_A + grpw * 64;
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {  // 16 pixels at a time
              uint64_t fj[8], fi[2][8];
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const uint32_t x = 16u * (4 * kh + c);
                *reinterpret_cast<ulonglong2 *>(fj + 2 * c) = *reinterpret_cast<const ulonglong2 *>(rb + (oj ^ x));
                *reinterpret_cast<ulonglong2 *>(fi[0] + 2 * c) = *reinterpret_cast<const ulonglong2 *>(rb + (oi0 ^ x));
                *reinterpret_cast<ulonglong2 *>(fi[1] + 2 * c) = *reinterpret_cast<const ulonglong2 *>(rb + (oi1 ^ x));
              }
              if constexpr (F16) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(fi[0][k]) : "l"(fi[0][k]), "l"(pk(sc_i, sc_i)));
                  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(fi[1][k]) : "l"(fi[1][k]), "l"(pk(sc_i, sc_i)));
                }
                if (sc_p != 1.f) {  // tile-uniform: only for extreme field scales
#pragma unroll
                  for (int k = 0; k < 8; ++k)
                    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(fj[k]) : "l"(fj[k]), "l"(pk(sc_p, sc_p)));
                }
              }
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                uint32_t H[8], L[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) pair_split<F16>(fi[q][k], fj[k], H[k], L[k]);
                st8(o + q * 32 + kh * 8, H);
                st8(o + q * 32 + 16 + kh * 8, L);
              }
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
          }
          __syncwarp();
          if (lane == 0 && ok) {
            mbar_arrive(raw_empty(sr));
            mbar_arrive(a_full(grpw));
          }
        }

        // ---------------------------------------------------- sub-tile sums
        bool ok = !*abort_flag;
        if (ok && !mbar_wait(acc_full, tc & 1, limit, abort_flag)) {
          fail();
          ok = false;
        }
        ++tc;
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
        const int n = w.width(), pan = min(16, w.pa_hi - 16 * h);
        // 32 fields at a time through shared memory (two buffers of 16): groups 0 and 1
        // bring the first 16 of the two MMAs, groups 2 and 3 the other 16
        for (int c0 = 0; c0 < n; c0 += 32) {
          const int mine = c0 + 16 * (grpw >> 1);
          uint32_t v[16];
          const bool have = ok && mine < n;
          if (have) ld16(tlane + (grpw & 1) * MROWS + mine, v);
          asm volatile("bar.sync 1, 512;" ::: "memory");  // the previous fields are summed
          if (have) {
            float *Tw = T + (grpw >> 1) * TFLOATS + (grpw & 1) * 128 + 32 * quad + lane;
#pragma unroll
            for (int c = 0; c < 16; ++c) Tw[c * TPITCH] = __uint_as_float(v[c]);
          }
          if (c0 + 32 >= n) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && ok) mbar_arrive(acc_empty);
          }
          asm volatile("bar.sync 1, 512;" ::: "memory");
          // a warp owns the entries of its nu1 - nu2, a lane those of its e2 mod 32: no two
          // threads ever add to one entry
          const int ng = min(4, (n - c0) / GROUP);
          for (int g = 0; g < ng; ++g) {
            const int4 gi = grp[c0 / GROUP + g];
            if (gi.x < 0) continue;
            const int4 si = seginfo[gi.x];
            const int E = si.y & 0xffff, sw = si.y >> 16, nv = gi.z;
            // field f of the group meets pair (pa, pb) at e2 = hi - nu3 + pb = (hi - x0) - C
            // (ordinary) or nu1 - lo + 15 - pb = (x0 - lo) + 15 + C (swapped), C = f - pb
            const int base = sw ? gi.y - (si.w - (E - P2)) : si.w - gi.y - 7;
            const int e2 = base + ((lane - base) & 31);
            if (e2 - base > 22 || e2 < 0 || e2 >= E) continue;
            const int C = sw ? e2 - base - 15 : 7 - (e2 - base);
            const float *Tg = T + (g >> 1) * TFLOATS + (g & 1) * GROUP * TPITCH - 17 * C;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const int dd = pw + 16 * k - 15;  // pa - pb within the half
              if (dd > 15 || 16 * h + dd > w.dmax) continue;
              // fields with 0 <= pb < pb_hi and 0 <= pa = pb + dd < pan
              const int f0 = max(0, max(C, C - dd));
              const unsigned cnt = (unsigned)max(0, min(nv, min(C + w.pb_hi, C - dd + pan)) - f0);
              float *r = red + si.x + (dd + 15 + 16 * h) * E + e2;
              const float *Tk = Tg + 16 * dd;
              float s = *r;
#pragma unroll
              for (int f = 0; f < GROUP; ++f)
                if ((unsigned)(f - f0) < cnt) s += Tk[f * (TPITCH + 17)];
              *r = s;
            }
          }
        }
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
      if (!*abort_flag) {
        // flush in the order of the (d1, d2) plane (coalesced FP64 atomics), as contract_tc.cu
        const int n2 = 2 * G.nc - 1, ns = *nseg_s;
        for (int sg = 0; sg < ns; ++sg) {
          const int4 si = seginfo[sg];
          const int E = si.y & 0xffff;
          const double sc = F16 ? segscale[sg] : 1.0;
          double *plane = G.dsum + (long long)b * G.dsum_bstride + (long long)si.z * n2 * n2;
          const float *rs = red + si.x;
          if (si.y >> 16) {
            const int lo = si.w - (E - P2);
            const int c1 = lo - (P2 - 1) - t.nu2_0 + G.nc - 1;
            const int c2 = t.nu1_0 - t.nu2_0 - (P2 - 1) + G.nc - 1;
            for (int e2 = pw; e2 < E; e2 += NPROD) {
              const long long row = (long long)(e2 + c1) * n2;
              for (int dd = lane; dd < npa + P2 - 1; dd += 32) {
                const float v = rs[dd * E + e2];
                if (v == 0.f) continue;
                if (BS_CHK(e2 + c1, n2, 37) && BS_CHK(dd + c2, n2, 38))
                  atomicAdd(plane + row + (dd + c2), F16 ? (double)v * sc : (double)v);
              }
            }
            continue;
          }
          const int d1base = t.nu1_0 - (P2 - 1) - si.w + G.nc - 1;
          const int d2base = t.nu2_0 - si.w + G.nc - 1;
          const int nrow = (npa + P2 - 1) + E - 1;
          for (int r = pw; r < nrow; r += NPROD) {
            const int e2lo = max(0, r - (npa + P2 - 2)), e2hi = min(E - 1, r);
            const long long row = (long long)(r + d1base) * n2;
            for (int e2 = e2lo + lane; e2 <= e2hi; e2 += 32) {
              const float v = rs[(r - e2) * E + e2];
              if (v == 0.f) continue;
              if (BS_CHK(r + d1base, n2, 39) && BS_CHK(e2 + d2base, n2, 40))
                atomicAdd(plane + row + (e2 + d2base), F16 ? (double)v * sc : (double)v);
            }
          }
        }
      }
      asm volatile("bar.sync 1, 512;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();  // every MMA has completed (the MMA thread waited for them)
  tc_fence_after();
  if (warp == NPROD + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
}

template <bool F16>
cudaError_t launch_tcs(const TcArgs &a, int nsm, cudaStream_t s) {
  cudaError_t e = smem_optin_once<k_contract_tcs<F16>>();
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<long long>(2LL * a.ntiles, nsm);
  k_contract_tcs<F16><<<grid, NTHREADS, SMEM_BYTES, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_contract_tcs(const TcArgs &a, int nsm, cudaStream_t s) {
  return a.f16 ? launch_tcs<true>(a, nsm, s) : launch_tcs<false>(a, nsm, s);
}

namespace {

// What the rule takes from one half (128 fields) of a tile's column window.
struct WindowHalf {
  int nrow;         // fields, padding of the runs included; <= 0: none
  long long spans;  // sum over its segments (one ring triple) of P2 + highest - lowest nu3
  bool split;       // a segment crosses 32 rows: several warps of contract_tc.cu add to an entry
};

WindowHalf scan_half(const ColEntry *cols, int nrow) {
  WindowHalf w{nrow, 0, false};
  for (int g = 0; g < nrow;) {
    const ColEntry &first = cols[g];
    int hi = first.nu3, e = g, last = g;
    for (; e < nrow; ++e) {
      const ColEntry &ce = cols[e];
      if (ce.field >= 0 && (ce.trip != first.trip || ce.swapped != first.swapped)) break;
      if (ce.field >= 0) {
        hi = ce.nu3;
        last = e;
      }
    }
    w.split = w.split || g / 32 != last / 32;
    w.spans += P2 + hi - first.nu3;
    g = e;
  }
  return w;
}

}  // namespace

// The sum of SM cycles either kernel takes for the tiles, by their stages, as
// measured: contract_tc.cu 1700 a stage of a CTA pair plus 12000 a tile; this one the
// larger of 8.5 a field and 800 (split FP16, whose conversions are dearer: 1050) a
// stage and sub-tile, plus its sums.  So lists up to 128 fields of a tile come here
// (raw sampling, 64 channels: 3.4 against 4.0 ms; 16 channels: 118 against 271 us alone,
// 5.4 against 27.5 ms for 256 realisations), fuller tiles stay (256-channel cube: 607
// against 464 ms where the tiles are full).  `fixed_order`: only where
// every entry is summed by one warp of contract_tc.cu, so that both kernels give the
// same bits (one pair half, the ring triples' fields within 32 rows); elsewhere
// contract_tc.cu's order depends on the race of its warps.
bool tcs_wins(const TcTile *tiles, size_t ntiles, const TcGroup *groups, const ColEntry *cols,
              bool fixed_order) {
  double cost_s = 0, cost_l = 0;
  // A column window belongs to every pair rectangle, K segment and realisation of its
  // list, and is scanned once (tile by tile, 20 thousand tiles with full windows took
  // the host 4.3 ms before the launch, 0.2 now).
  struct Window {
    WindowHalf half[2];
  };
  std::unordered_map<long long, Window> seen;
  long long key = -1;
  const Window *win = nullptr;
  for (size_t q = 0; q < ntiles; ++q) {
    const TcTile &t = tiles[q];
    const TcGroup &G = groups[t.group];
    if (!G.dsum || G.out_full) return false;  // this kernel writes the collapse sums only
    const int pa_hi = std::min(P1, G.nu1_hi - t.nu1_0), pb_hi = std::min(P2, G.nu2_hi - t.nu2_0);
    if (fixed_order && pa_hi > 16) return false;
    const int dmax = t.diag ? t.nu2_0 - t.nu1_0 : P1, npa = pa_hi > 16 ? 32 : 16;
    const int nst = std::max(0, std::min(G.Kpad, (t.kseg + 1) * G.kseg_len) - t.kseg * G.kseg_len) / KC;
    int halves = 0;
    for (int h = 0; h < 2; ++h) halves += 16 * h < pa_hi && 16 * h - (pb_hi - 1) <= dmax;
    cost_l += 2.0 * (1700.0 * nst + 12000.0);  // a pair of SMs per tile
    // the first column's index names the window: lists do not overlap
    if (const long long k = (long long)t.col_off + t.col0; !win || k != key) {
      key = k;
      const auto at = seen.try_emplace(k);
      Window &w = at.first->second;
      if (at.second)
        for (int r = 0; r < 2; ++r)
          w.half[r] = scan_half(cols + k + MROWS * r, std::min(MROWS, t.ncol - t.col0 - MROWS * r));
      win = &w;
    }
    for (const WindowHalf &w : win->half) {
      if (w.nrow <= 0) continue;
      if (fixed_order && w.split) return false;
      if ((npa + P2 - 1) * w.spans > RED_CAP) return false;  // floats of the reduction buffer
      const int n = (w.nrow + 15) & ~15;
      cost_s += halves * (nst * std::max(8.5 * n, G.kexp ? 1050.0 : 800.0) + 2500.0 + 60.0 * n) + 4000.0;
    }
  }
  return ntiles > 0 && cost_s < cost_l;
}

}  // namespace bsi
