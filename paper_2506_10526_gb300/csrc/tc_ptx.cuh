// tcgen05, TMA and mbarrier instruction forms and the operand splits shared by
// the two tensor-core contraction kernels (contract_tc.cu, contract_tcs.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "bs_internal.h"

namespace bsi {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_count() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// Shared-memory address of the same variable in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrive on an mbarrier of any CTA of the cluster (address from map_rank).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
template <bool CLUSTER>
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  if (CLUSTER)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
  return ok != 0;
}
// Bounded wait; false on timeout or when the CTA is aborting.  CLUSTER: the
// phase was completed by arrivals from the other CTA of the pair.
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long limit_ns,
                                          volatile int *abort_flag) {
  if (mbar_try<CLUSTER>(bar, parity)) return true;
  const uint64_t t0 = gtime();
  while (true) {
    if (mbar_try<CLUSTER>(bar, parity)) return true;
    if (*abort_flag) return false;
    if ((long long)(gtime() - t0) > limit_ns) return false;
  }
}
// One lane of the (converged) warp, always the same.  The MMA and TMA instructions
// take their operands from uniform registers: inside `if (elect_one())` the compiler
// moves them there directly, inside `if (lane == 0)` it wraps every instruction in a
// loop over the lanes that might be active.  Measured per tcgen05.mma issued back to
// back: 140 to 230 cycles against 58 (and then the MMA's own 64 at N = 128, 128 at
// N = 256).  A single thread's instruction costs it 4 to 5 cycles, so what it computes
// per stage counts as well.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
// The copies of a list of 16 groups of 8 field rows: lane g < 16 has group g's first
// row (`live`: a group of the list).  Runs of consecutive rows become one box of 16,
// 32, 64 or 128 rows.  Fills list[0..n) with (row, byte offset of the group in a
// 64-byte-row operand, address of the map) and returns n; mg: the level's hi maps, or
// one on, its lo maps.  Called by a whole warp.
__device__ __forceinline__ int box_list(const CUtensorMap *mg, int row, bool live, int4 *list,
                                        int lane) {
  int box = lane < 16 && live ? 1 : 0;  // rows / 8; 0: covered by an earlier box
#pragma unroll
  for (int n = 2; n <= 16; n *= 2) {
    const int pbox = __shfl_down_sync(0xffffffffu, box, n / 2);
    const int prow = __shfl_down_sync(0xffffffffu, row, n / 2);
    const int join = (lane & (n - 1)) == 0 && box == n / 2 && pbox == n / 2 && prow == row + 4 * n;
    const int joined = __shfl_up_sync(0xffffffffu, join, n / 2);
    if (join) box = n;
    if ((lane & (n - 1)) == n / 2 && joined) box = 0;
  }
  const unsigned m = __ballot_sync(0xffffffffu, box > 0);
  if (box > 0) {
    const uint64_t mp =
        (uint64_t)(mg + (box == 1 ? 0 : box == 2 ? 7 : box == 4 ? 2 : box == 8 ? 9 : 4));
    list[__popc(m & ((1u << lane) - 1))] =
        make_int4(row, lane * 8 * 64, (int)(uint32_t)mp, (int)(uint32_t)(mp >> 32));
  }
  __syncwarp();
  return __popc(m);
}
__device__ __forceinline__ const CUtensorMap *box_map(const int4 &x) {
  return reinterpret_cast<const CUtensorMap *>((uint64_t)(uint32_t)x.z | ((uint64_t)(uint32_t)x.w << 32));
}
// The first four boxes of a list in registers (a read of the list on every stage lies
// on the issuing thread's path), the others from shared memory.
struct Boxes {
  int4 b[4];
  int n;
  const int4 *list;
  __device__ __forceinline__ Boxes(const int4 *l, int nbox) : n(nbox), list(l) {
#pragma unroll
    for (int q = 0; q < 4; ++q) b[q] = q < nbox ? l[q] : make_int4(0, 0, 0, 0);
  }
  // the copies of one stage (pixels kc..) to dst
  __device__ __forceinline__ void load(uint32_t dst, int kc, uint32_t bar) const {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < n) tma_load_2d(dst + b[q].y, box_map(b[q]), kc, b[q].x, bar);
    for (int q = 4; q < n; ++q) {
      const int4 x = list[q];
      tma_load_2d(dst + x.y, box_map(x), kc, x.x, bar);
    }
  }
};
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Arrive (once) on the mbarrier at this shared offset in both CTAs of the pair
// when every MMA issued so far has completed.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  const uint16_t mask = 3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// Shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512 B apart.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}
// Shared-memory float reduction (no return value) at a shared-space address.
__device__ __forceinline__ void red_add_shared(uint32_t addr, float v) {
  asm volatile("red.shared.add.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// Byte offset of 16-byte chunk c (0..3) of row r in a 64B-swizzled K-major tile.
__device__ __forceinline__ uint32_t sw64_off(int r, int c) {
  return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4));
}
// Byte offset of 16-byte chunk c (0..7) of row r in a 128B-swizzled tile of
// 128-byte rows (TMA SWIZZLE_128B on a 1024-byte aligned buffer).
__device__ __forceinline__ uint32_t sw128_off(int r, int c) {
  return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4));
}
// BF16 hi/lo split of two FP32 values, packed (element 0 in the low half).
__device__ __forceinline__ void split2(float v0, float v1, uint32_t &hi, uint32_t &lo) {
  __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
  hi = *reinterpret_cast<uint32_t *>(&h);
  const float h0 = __uint_as_float(hi << 16), h1 = __uint_as_float(hi & 0xffff0000u);
  __nv_bfloat162 l = __floats2bfloat162_rn(v0 - h0, v1 - h1);
  lo = *reinterpret_cast<uint32_t *>(&l);
}
// FP16 hi/lo split of two FP32 values, packed (element 0 in the low half).
__device__ __forceinline__ void split2_f16(float v0, float v1, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(v0, v1);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  const float2 hf = __half22float2(h);
  const __half2 l = __floats2half2_rn(v0 - hf.x, v1 - hf.y);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}
// 2^k as FP32 (|k| <= 126) and as FP64 (|k| <= 1022), built from the exponent field.
__device__ __forceinline__ float exp2i_f32(int k) { return __uint_as_float((uint32_t)(k + 127) << 23); }
__device__ __forceinline__ double exp2i_f64(int k) {
  return __longlong_as_double((long long)(k + 1023) << 52);
}

}  // namespace tc
}  // namespace bsi
