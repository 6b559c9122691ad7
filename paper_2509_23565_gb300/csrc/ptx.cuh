// Inline-PTX helpers for sm_103a: mbarrier, TMA (cp.async.bulk.tensor),
// tcgen05 (TMEM alloc, MMA, commit, ld) and the UMMA shared-memory /
// instruction descriptors.  Every wait is bounded: after `limit` cycles it
// returns false so the caller can record an error and leave.
#pragma once
#include <cstdint>
#include <cuda.h>

namespace emul {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- dependent launches
// A kernel launched with launch_dependent() (launch.h) may start while the one
// before it in the stream still runs.  grid_wait: until that one has completed
// and its writes are visible; before any access to memory that others write or
// read.  grid_launch: lets the next one start (it waits in the same way); a kernel
// with TMEM calls it once the block's allocation stands, as a block of the next
// kernel could otherwise take the columns and wait for this one to complete.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait on the phase with the given parity.  Returns false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (clock64() - t0 > limit) return false;
  }
}
// Relaxed arrive on this CTA's barrier (the TMEM-slot release: see mbar_arrive_cluster).
__device__ __forceinline__ void mbar_arrive_relaxed(uint64_t* bar) {
  asm volatile("mbarrier.arrive.relaxed.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// Generic writes to this CTA's shared memory, ordered before reads by the async proxy (MMA, TMA).
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------- TMA
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// ---------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulate (kind::f16): both
// K = 16 MMAs of a staged K chunk of 32 (64-byte rows: the second one reads 32
// bytes, two descriptor units, further), issued by one elected lane of a
// converged warp.  The whole warp runs the issuing loop, so every operand is
// warp-uniform and stays in the uniform datapath; one thread alone recomputing
// descriptors issues an MMA only every ~84 cycles, short of the 64 a 128 x 128
// x 16 MMA takes.  Descriptors come as their low word (the start address, the
// only part that changes) and high word.
template <bool PAIR>
__device__ __forceinline__ void mma_bf16_k32_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t hi,
                                                   uint32_t idesc, uint32_t accumulate) {
  if constexpr (PAIR)
    asm volatile(
        "{\n.reg .pred e, p;\n.reg .b32 a1, b1;\n.reg .b64 da, db, dc, dd;\nelect.sync _|e, 0xffffffff;\n"
        "setp.ne.b32 p, %5, 0;\nadd.u32 a1, %1, 2;\nadd.u32 b1, %2, 2;\n"
        "mov.b64 da, {%1, %3};\nmov.b64 db, {%2, %3};\nmov.b64 dc, {a1, %3};\nmov.b64 dd, {b1, %3};\n"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, p;\n"
        "@e tcgen05.mma.cta_group::2.kind::f16 [%0], dc, dd, %4, 1;\n}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate));
  else
    asm volatile(
        "{\n.reg .pred e, p;\n.reg .b32 a1, b1;\n.reg .b64 da, db, dc, dd;\nelect.sync _|e, 0xffffffff;\n"
        "setp.ne.b32 p, %5, 0;\nadd.u32 a1, %1, 2;\nadd.u32 b1, %2, 2;\n"
        "mov.b64 da, {%1, %3};\nmov.b64 db, {%2, %3};\nmov.b64 dc, {a1, %3};\nmov.b64 dd, {b1, %3};\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], dc, dd, %4, 1;\n}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate));
}
// Arrive on `bar` once every tcgen05 operation issued so far by the elected lane of a
// converged warp has completed.
__device__ __forceinline__ void mma_commit_elect(uint64_t* bar) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar))
      : "memory");
}
// TMA 3D load issued by one elected lane of a converged warp.
__device__ __forceinline__ void tma_load_3d_elect(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                                  int c2) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
      "[%2];\n}\n" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx_elect(uint64_t* bar, uint32_t bytes) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(smem_u32(bar)), "r"(bytes)
      : "memory");
}
// Bounded wait by every lane of a warp; true only if every lane saw the phase
// complete (a warp-uniform answer).
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, long long limit) {
  const bool ok = mbar_wait(bar, parity, limit);
  return __all_sync(0xFFFFFFFFu, ok);
}

// ---------------------------------------------------------------- CTA pairs
// A cluster of two CTAs sharing one product tile (cta_group::2): rank 0 issues
// the MMAs for both, reading the operand tiles each CTA staged in its own
// shared memory at the same offsets; each CTA's TMEM holds its 128 rows.
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Shared::cluster address of `p` (this CTA's shared memory) in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa_rank(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
  return r;
}
// The shared::cluster address `addr` of this CTA (smem_u32) in CTA `rank`.
__device__ __forceinline__ uint32_t mapa_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Plain accesses to a CTA's shared memory in the cluster (ordered by cluster_sync).
__device__ __forceinline__ double ld_cluster_f64(uint32_t addr_cl) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr_cl) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_f64(uint32_t addr_cl, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr_cl), "d"(v) : "memory");
}
// Store 8 bytes into a CTA of the cluster and count them on a barrier there.
__device__ __forceinline__ void st_async_b64(uint32_t addr_cl, uint64_t v, uint32_t bar_cl) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr_cl), "l"(v),
               "r"(bar_cl)
               : "memory");
}
// Bounded wait with acquire at cluster scope by one thread (for st_async data).
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, long long limit) {
  auto try_once = [&]() {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
  };
  if (try_once()) return true;
  const long long t0 = clock64();
  while (!try_once())
    if (clock64() - t0 > limit) return false;
  return true;
}
// Every thread of both CTAs (no timeout exists for it: callers reach it on every path).
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
// Commit of the pair's MMAs arriving on `bar` at the same offset in both CTAs.
__device__ __forceinline__ void mma_commit_pair_both_elect(uint64_t* bar) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n"
      ::"r"(smem_u32(bar)), "h"((uint16_t)3)
      : "memory");
}
// TMA 3D load into this CTA's shared memory whose completion is counted on
// the barrier at shared::cluster address `bar_cl` (rank 0's barrier).
__device__ __forceinline__ void tma_load_3d_pair_elect(void* dst, const CUtensorMap* map, uint32_t bar_cl, int c0,
                                                       int c1, int c2) {
  asm volatile(
      "{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
      "@e cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], "
      "[%1, {%3, %4, %5}], [%2];\n}\n" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cl), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
// Arrive on the barrier at shared::cluster address `bar_cl`, relaxed: it
// orders nothing but itself.  The TMEM-slot release needs no more: the slot's
// tcgen05.ld have completed (tcgen05.wait::ld) before it, and the global
// updates of C the thread issued are not what the barrier protects (a release
// at cluster scope would wait for every one of them to be performed).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cl) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cl) : "memory");
}
// Bounded wait with acquire at cluster scope (arrivals from the other CTA), by
// every lane of a warp; warp-uniform answer.
__device__ __forceinline__ bool mbar_wait_cluster_warp(uint64_t* bar, uint32_t parity, long long limit) {
  auto try_once = [&]() {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
  };
  bool ok = try_once();
  if (!ok) {
    const long long t0 = clock64();
    while (!(ok = try_once()))
      if (clock64() - t0 > limit) break;
  }
  return __all_sync(0xFFFFFFFFu, ok);
}

// 32 lanes x 16 consecutive 32-bit columns: thread i of the warp gets lane (base+i).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// UMMA shared-memory descriptor, K-major operand with the given swizzle.
//   swizzle: 2 = 128 B rows (atom 8 rows x 128 B), 4 = 64 B rows (atom 8 x 64 B),
//            6 = 32 B rows (atom 8 x 32 B)
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t row_bytes, uint32_t swizzle_code) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr >> 4) & 0x3FFF);
  d |= static_cast<uint64_t>(1) << 16;                                   // LBO (unused, K-major swizzled)
  d |= static_cast<uint64_t>(((8 * row_bytes) >> 4) & 0x3FFF) << 32;    // SBO: one 8-row atom
  d |= static_cast<uint64_t>(1) << 46;                                   // descriptor version
  d |= static_cast<uint64_t>(swizzle_code) << 61;
  return d;
}
// Instruction descriptor: bf16 x bf16 -> f32, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

}  // namespace emul
