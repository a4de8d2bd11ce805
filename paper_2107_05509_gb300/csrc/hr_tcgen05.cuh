// Device building blocks of the tensor-core kernels (hr_gemm.cu, hr_conv.cu): bounded
// mbarrier waits, TMA loads, tcgen05 descriptors, products and accumulator reads.
#pragma once

#include <algorithm>

#include <cuda.h>
#include <cuda_bf16.h>

#include "hr_internal.h"

namespace hr {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for the phase of `parity` to complete; false when it ran out.  The bound is
// on the SM's clock: reading the global timer between two tries held up the wake-up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long clocks) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 16; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > clocks) return false;
  }
}

// the same for arrivals from the other CTA of a cluster
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, long long clocks) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > clocks) return false;
  }
}

// When a wait has run out, its role stops, the others' waits run out likewise, and no
// block may end, nor its tensor memory be freed, before the copies and the products that
// are under way are done:
//   the copies: fill n of a ring of S slots is in slot n % S and completes phase n / S of
//   its barrier.  Of `issued` fills the last S can be under way; each is waited for in its
//   own phase (a slot is filled again only when the fill before it has been used, so no
//   older phase is open), all of them for `kWaitClocks` at most: a fill that another
//   role shares in and never made completes no phase, and its copy has landed by then.
//   the products: a last commit, by the thread that issued them, on a barrier of its own.
template <int S>
__device__ __forceinline__ void drain_fills(uint64_t* full, int issued) {
  const long long t0 = clock64();
  for (int n = issued > S ? issued - S : 0; n < issued; ++n)
    while (!mbar_try_wait(smem_u32(&full[n % S]), (n / S) & 1))
      if (clock64() - t0 > kWaitClocks) return;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// this thread's warp in the block, in a form the compiler knows to be the same for the
// whole warp, and the choice of one of its threads.  The warps that issue TMA loads and
// products run their loops as a whole, with uniform registers, and only the instruction
// itself is one thread's: in a loop of one thread (lane == 0) every descriptor went
// through per-thread registers, and issuing took longer than the products.
__device__ __forceinline__ int warp_id() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
  return ok != 0;
}

// tcgen05 shared-memory matrix descriptors, 128-byte swizzle, in halves: the low word
// holds the start address (and the leading byte offset), so that a step along the operand
// is one 32-bit addition of (bytes >> 4).
//   K-major: rows of 128 bytes (64 bf16 along K), 8-row groups 1024 bytes apart
//   MN-major: rows of 128 bytes hold 64 values along M (or N) of one k, 8 k's 1024 bytes
//   apart, the next 64 along M `block` bytes on
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);   // stride, version, swizzle
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFF) | (1u << 16); }
__device__ __forceinline__ uint32_t desc_mn_lo(uint32_t saddr, uint32_t block) {
  return ((saddr >> 4) & 0x3FFF) | (((block >> 4) & 0x3FFF) << 16);
}

// instruction descriptor of kind::f16: bf16 x bf16 -> f32, M x N, operands K-major or
// (mn) both MN-major
__host__ __device__ constexpr uint32_t mma_idesc(int M, int N, bool mn = false) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (1u << 15) | (1u << 16) : 0u) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %5};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}\n" ::"r"(tmem),
      "r"(a_lo), "r"(b_lo), "r"(idesc), "r"((uint32_t)accumulate), "r"(kDescHi)
      : "memory");
}
// the products of one 64-wide K step of K-major tiles (one thread)
__device__ __forceinline__ void mma_step(uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, bool accumulate) {
#pragma unroll
  for (int k = 0; k < 4; ++k) mma_bf16(tmem, a_lo + 2 * k, b_lo + 2 * k, idesc, accumulate || k > 0);
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// ---- pairs of CTAs (a cluster of two): the product of one 256-row tile on both SMs ----
// the address of `saddr` in the shared memory of the cluster's CTA `rank`
__device__ __forceinline__ uint32_t cluster_addr(uint32_t saddr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void store_cluster(uint32_t cluster_addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// load into this CTA's shared memory, counted on a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(cluster_bar)
      : "memory");
}
__device__ __forceinline__ void mma_step_pair(uint32_t tmem, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, bool accumulate) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %5};\n"
        " tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n}\n" ::"r"(tmem),
        "r"(a_lo + 2 * k), "r"(b_lo + 2 * k), "r"(idesc), "r"((uint32_t)(accumulate || k > 0)), "r"(kDescHi)
        : "memory");
}
// the products issued so far arrive on this barrier in both CTAs
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}
// by one whole warp of each CTA
template <int kCols>
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_slot) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_slot), "r"(kCols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
template <int kCols>
__device__ __forceinline__ void tmem_free_pair(uint32_t tmem) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

// tensor-memory allocation and release by one whole warp; kCols a power of two >= 32
template <int kCols>
__device__ __forceinline__ void tmem_alloc(uint32_t smem_slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_slot), "r"(kCols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int kCols>
__device__ __forceinline__ void tmem_free(uint32_t tmem) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 2-D bf16 tensor map over rows x cols (cols contiguous, row pitch ld elements) with
// boxes of 64 columns x box_rows, 128-byte swizzle; values outside are zero (hr_gemm.cu)
bool tma_map(CUtensorMap* map, const void* ptr, long long rows, int cols, int ld, int box_rows);

}  // namespace hr
