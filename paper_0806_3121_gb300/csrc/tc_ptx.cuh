// Inline-PTX helpers for the Blackwell (sm_103a) tensor-core path: mbarriers
// with bounded waits, TMA tiled loads and stores, TMEM allocation, tcgen05.mma
// issue, commit and TMEM loads.  Device code only.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace abft {
namespace tc {

// A wait that has not completed after this long gives up (the kernel then
// records a timeout instead of hanging).  One phase of any barrier here spans
// at most one tile's K loop, which takes well under a millisecond.
constexpr uint64_t kWaitLimitNs = 4000000000ull;

// The limit in force (a kernel may shorten it for its timeout test).
__device__ __forceinline__ uint64_t& wait_limit_ns() {
  static __shared__ uint64_t lim;
  return lim;
}

// True in one lane of a converged warp.  The roles that issue tcgen05 and TMA
// instructions run in this lane: under `lane == 0` the compiler cannot tell that
// one thread is active, so it builds the uniform-register operands of every such
// instruction in a loop over the lanes.  Measured per k-step of four M = 128 MMAs
// with a commit and a wait: 552 clocks at any N under `lane == 0`; here, with the
// four MMAs in one asm block (mma4), 236 / 256 / 512 at N = 64 / 128 / 256, the
// tensor pipe's own rate.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for the phase of parity `parity` of barrier `bar` to complete.  Gives
// up (returns false) when *abort is set by another role or after
// kWaitLimitNs, in which case it sets *abort itself.
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
    if (globaltimer() - t0 > wait_limit_ns()) {
      *abort = 1;
      return false;
    }
  }
}

// Holds a worker (CTA pair) of a persistent kernel back until the others have come as far:
// one thread of each calls this `calls` times per tile, the n-th time in its `round`-th
// tile with call = n.  It only orders reads, so that workers find each other's panels in
// L2: a worker whose fellows are not running (another stream's kernel holds their SMs)
// gets false after limit_ns, stops waiting and only counts itself in.
__device__ __forceinline__ bool keep_step(uint32_t* arrivals, uint32_t workers, int64_t total,
                                          uint32_t round, uint32_t call, uint32_t calls,
                                          uint64_t limit_ns) {
  const int64_t in_round = min((int64_t)workers, total - (int64_t)round * workers);
  const uint32_t target = round * workers * calls + call * (uint32_t)in_round;
  if ((int32_t)(atomicAdd(arrivals, 1u) + 1 - target) >= 0) return true;
  const uint64_t t0 = globaltimer();
  while ((int32_t)(*(volatile uint32_t*)arrivals - target) < 0)
    if (globaltimer() - t0 > limit_ns) return false;
  return true;
}

// 2-D tiled TMA load of the box at element coordinates (x inner, y outer)
// into shared memory, completing on barrier `bar` (transaction bytes).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int32_t x, int32_t y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

// 3-D tiled TMA load (x inner, then y, then z) into shared memory.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int32_t x, int32_t y, int32_t z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}

// 2-D tiled TMA store of a box from shared memory to global memory (tracked
// by the bulk async-group of the issuing thread).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int32_t x,
                                             int32_t y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Every committed bulk store of this thread has finished reading its source.
__device__ __forceinline__ void bulk_wait_read0() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// Every committed bulk store of this thread has completed.
__device__ __forceinline__ void bulk_wait0() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
// Generic-proxy writes to shared memory become visible to the async proxy
// (TMA) -- each writing thread, before the store is issued.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// ---- TMEM
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Arrive once on `bar` when every tcgen05.mma issued so far by this thread
// has completed.
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   bar)
               : "memory");
}

// The four K steps of one stage, D[tmem] (+)= A[smem] * B[smem] with fp32
// accumulation: kind::f16 (16-bit inputs, K = 16 each) or kind::f8f6f4 (8-bit
// floating-point inputs, K = 32 each), on one CTA or a CTA pair.  The descriptors
// advance by SA / SB 16-byte units per step; accumulate = 0: the first step
// overwrites D.
#define ABFT_MMA4(NAME, GROUP, KIND)                                                           \
  template <int SA, int SB>                                                                    \
  __device__ __forceinline__ void NAME(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,     \
                                       uint32_t accumulate) {                                  \
    asm volatile(                                                                              \
        "{\n\t.reg .pred p, q;\n\t.reg .b64 x, y;\n\t"                                         \
        "setp.ne.b32 p, %4, 0;\n\t"                                                            \
        "setp.eq.u32 q, 0, 0;\n\t"                                                             \
        "tcgen05.mma." GROUP "." KIND " [%0], %1, %2, %3, p;\n\t"                              \
        "add.s64 x, %1, %5;\n\tadd.s64 y, %2, %6;\n\t"                                         \
        "tcgen05.mma." GROUP "." KIND " [%0], x, y, %3, q;\n\t"                                \
        "add.s64 x, %1, %7;\n\tadd.s64 y, %2, %8;\n\t"                                         \
        "tcgen05.mma." GROUP "." KIND " [%0], x, y, %3, q;\n\t"                                \
        "add.s64 x, %1, %9;\n\tadd.s64 y, %2, %10;\n\t"                                        \
        "tcgen05.mma." GROUP "." KIND " [%0], x, y, %3, q;\n\t}\n" ::"r"(d),                  \
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "n"(SA), "n"(SB), "n"(2 * SA),            \
        "n"(2 * SB), "n"(3 * SA), "n"(3 * SB)                                                  \
        : "memory");                                                                           \
  }
ABFT_MMA4(mma4_f16_cta, "cta_group::1", "kind::f16")
ABFT_MMA4(mma4_f16_pair, "cta_group::2", "kind::f16")
ABFT_MMA4(mma4_f8_cta, "cta_group::1", "kind::f8f6f4")
ABFT_MMA4(mma4_f8_pair, "cta_group::2", "kind::f8f6f4")
#undef ABFT_MMA4

// Shared-memory matrix descriptor (tcgen05): start address, leading and
// stride byte offsets, descriptor version 1, 128-byte swizzle.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;  // descriptor version (sm_100 family)
  d |= static_cast<uint64_t>(2) << 61;  // SWIZZLE_128B
  return d;
}

// Instruction descriptor for kind::f16: bf16 x bf16 -> f32, M x N, A K-major,
// B K-major (b_mn_major = 0) or MN-major (1).
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, int b_mn_major) {
  return (1u << 4)                                 // D format f32
         | (1u << 7)                               // A format bf16
         | (1u << 10)                              // B format bf16
         | (static_cast<uint32_t>(b_mn_major) << 16)  // B major-ness
         | (static_cast<uint32_t>(N >> 3) << 17)   // N / 8
         | (static_cast<uint32_t>(M >> 4) << 24);  // M / 16
}

// Instruction descriptor for kind::f16 with MN-major A (the A operand's M
// index contiguous, as B's N index in an N-major B) and K-major B: bf16 x bf16
// -> f32, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_mn_a(int M, int N) {
  return (1u << 4)                                 // D format f32
         | (1u << 7)                               // A format bf16
         | (1u << 10)                              // B format bf16
         | (1u << 15)                              // A MN-major
         | (static_cast<uint32_t>(N >> 3) << 17)   // N / 8
         | (static_cast<uint32_t>(M >> 4) << 24);  // M / 16
}

// Instruction descriptor for kind::f8f6f4: e4m3 x e4m3 -> f32 (format code 0
// for both operands), M x N, A K-major, B K-major (0) or MN-major (1).
__host__ __device__ constexpr uint32_t idesc_e4m3(int M, int N, int b_mn_major) {
  return (1u << 4)                                 // D format f32
         | (0u << 7)                               // A format e4m3
         | (0u << 10)                              // B format e4m3
         | (static_cast<uint32_t>(b_mn_major) << 16)  // B major-ness
         | (static_cast<uint32_t>(N >> 3) << 17)   // N / 8
         | (static_cast<uint32_t>(M >> 4) << 24);  // M / 16
}

// ---- CTA pairs (cta_group::2): two CTAs of a cluster run one M = 256 MMA.
// Each CTA holds 128 rows of A and half of B's columns in its own shared
// memory and 128 rows of the accumulator in its own TMEM; one thread of the
// even CTA issues the MMAs.  A kernel uses either the single-CTA or the pair
// forms of the tcgen05 instructions, never both.
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t num_clusters() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// Address, in the cluster's shared window, of the variable at shared address
// `addr` of this CTA in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Every thread of both CTAs: writes before it are visible to the whole
// cluster after it.
__device__ __forceinline__ void cluster_sync() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrive on a barrier given by its cluster address (this CTA's or the peer's).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cbar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cbar)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// wait(), ordered after the other CTA's writes before its arrivals.
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (true) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if (*abort) return false;
    if (globaltimer() - t0 > wait_limit_ns()) {
      *abort = 1;
      return false;
    }
  }
}
// TMA loads into this CTA's shared memory whose bytes complete on a barrier
// of either CTA of the pair (cbar: its cluster address).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map,
                                                 uint32_t cbar, int32_t x, int32_t y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(cbar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map,
                                                 uint32_t cbar, int32_t x, int32_t y, int32_t z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(cbar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// One warp of each CTA of the pair, together: the same TMEM columns in both.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
// Arrive once on the barrier at shared address `bar` of every CTA in
// `cta_mask` when the pair MMAs issued so far by this thread have completed.
__device__ __forceinline__ void commit_pair(uint32_t bar, uint16_t cta_mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar),
      "h"(cta_mask)
      : "memory");
}

// The single-CTA or the pair form, chosen at compile time.
template <bool kPair, int SA, int SB>
__device__ __forceinline__ void mma4_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t i,
                                         uint32_t acc) {
  if constexpr (kPair) mma4_f16_pair<SA, SB>(d, a, b, i, acc);
  else mma4_f16_cta<SA, SB>(d, a, b, i, acc);
}
template <bool kPair, int SA, int SB>
__device__ __forceinline__ void mma4_f8(uint32_t d, uint64_t a, uint64_t b, uint32_t i,
                                        uint32_t acc) {
  if constexpr (kPair) mma4_f8_pair<SA, SB>(d, a, b, i, acc);
  else mma4_f8_cta<SA, SB>(d, a, b, i, acc);
}
// Stage / accumulator signal: the pair's commit reaches both CTAs' barriers.
template <bool kPair>
__device__ __forceinline__ void commit_x(uint32_t bar) {
  if constexpr (kPair) commit_pair(bar, 3); else commit(bar);
}

// 32 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace tc
}  // namespace abft
