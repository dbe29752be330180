// Fifth-generation tensor-core building blocks (sm_103a): TMEM allocation, tcgen05.mma
// (A in TMEM, B in shared memory), its commit, TMEM loads and stores, tiled TMA loads, clusters.
//
// B tiles are K-major with the 128-byte swizzle: a tile row (one N index)
// is 64 16-bit K entries = 128 bytes, 16-byte chunk c of row r sits at
// 128 r + 16 (c ^ (r & 7)), and tiles start on 1024-byte boundaries.  One
// tcgen05.mma covers 16 of the 64 K entries (32 bytes along the row).
#pragma once

#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "kd_bulk.cuh"

namespace kd {

// shared-memory matrix descriptor of a tile row block: start address, 1024 bytes
// between groups of eight rows, 128-byte swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}

// instruction descriptor of kind::f16: fp32 accumulators, both operands bf16 or both
// fp16, K-major, M = 128, N columns
__host__ __device__ constexpr uint32_t tc_idesc(bool bf16, int n) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((uint32_t)(n / 8) << 17) |
         ((128u / 16u) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t cols) {  // one whole warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t addr, uint32_t cols) {  // the allocating warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}

// true in one lane (always the same) of a converged warp.  Code that issues tcgen05 and
// TMA instructions is branched on this and not on a lane number: only then does the
// compiler know that one thread runs it, and issues them without a loop over the lanes.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

// D (TMEM) = A B (+ D), one K = 16 step; issued by one thread.  A is in TMEM: lane = row, each 32-bit column two consecutive K entries
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}

// eight 32-bit columns of this warp's 32 TMEM lanes; complete after tmem_wait_st
__device__ __forceinline__ void tmem_st8(uint32_t addr, uint4 lo, uint4 hi) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(lo.x),
               "r"(lo.y), "r"(lo.z), "r"(lo.w), "r"(hi.x), "r"(hi.y), "r"(hi.z), "r"(hi.w)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// arrives on bar once every tcgen05.mma this thread issued before has completed
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// Waits, bounded, until every tcgen05.mma that this thread issued has completed; `bar` (one
// arrival) serves this alone.  Before shared memory or TMEM is used for anything else or given
// back: after an expired wait nobody has waited for the sums.
__device__ __forceinline__ void tc_drain(uint64_t* bar, int* fail) {
  tc_commit(bar);
  if (!mbar_wait_bounded(bar, 0)) *(volatile int*)fail = 1;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// eight consecutive fp32 columns of this warp's 32 TMEM lanes (lane l of the warp gets
// lane l's values); the values are valid after tmem_wait_ld
__device__ __forceinline__ void tmem_ld8(float* v, uint32_t addr) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(addr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld4(float* v, uint32_t addr) {  // four columns
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// tiled TMA load of the map's box at element coordinates (c0, c1); c0 is a multiple of
// 64 16-bit elements, so every copy starts on a 16-byte boundary
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}

// Bounded wait for the phase of `bar` with this parity: false, with *fail set, once a wait of
// this CTA has taken kWaitTries tries (every later one then gives up at once).  A try parks the
// thread for 7,762 cycles where nothing arrives (measured), so the limit is a second.  The loop is a try, a
// counter and two branches: with a clock and a flag read in it, polling took a fifth of the
// instructions of the whole kernel.  Lanes of a warp may get different answers, and lanes that
// gave up would leave the others in a later elect.sync, without limit: a warp that elects a lane
// after its waits votes on them first.
#ifndef KD_MBAR_WAIT  // a build of the tests: test_wait, which does not park the thread
#define KD_MBAR_WAIT "mbarrier.try_wait"
#endif
#ifndef KD_WAIT_TRIES
#define KD_WAIT_TRIES (1u << 18)
#endif
constexpr uint32_t kWaitTries = KD_WAIT_TRIES;
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity, int* fail) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t" KD_MBAR_WAIT
      ".parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  if (done) return true;
  if (*(volatile int*)fail) return false;
  uint32_t left = kWaitTries;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "TRY_%=:\n\t"
      KD_MBAR_WAIT ".parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra DONE_%=;\n\t"
      "add.u32 %0, %0, -1;\n\t"
      "setp.ne.u32 q, %0, 0;\n\t"
      "@q bra TRY_%=;\n\t"
      "DONE_%=:\n\t}"
      : "+r"(left)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  if (left != 0) return true;
  *(volatile int*)fail = 1;
  return false;
}

// Programmatic dependent launch: the next launch of the stream, if it asks for it, may start
// once every CTA of this one has come here; it then waits for this one's end and its writes.
__device__ __forceinline__ void grid_dependents_start() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// fp32 word of CTA `rank`'s shared memory at the address that `local` has in this CTA
__device__ __forceinline__ float ld_dsmem(uint32_t local, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

}  // namespace kd
