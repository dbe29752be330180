// Arithmetic of the tensor-core kernels that a host compiler takes too (checked there by
// tests/test_tc_host.py).
#pragma once

#ifdef __CUDACC__
#define KD_TC_HD __host__ __device__
#else
#define KD_TC_HD
#endif

namespace kd {

// Parity of the barrier phase that the last copy into slot s completes, after `issued` copies
// round-robin over a ring of `slots` (one phase of a slot's barrier per copy); -1: none went
// there.  Waiting for this one parity waits for that copy.  A loop that stops at either parity
// waits for nothing: one of the two always reads as complete.
KD_TC_HD constexpr int ring_last_parity(int issued, int slots, int s) {
  return s < issued ? ((issued - 1 - s) / slots) & 1 : -1;
}

// Dynamic shared memory that a CTA with `cols` columns of TMEM (256 or 512 of the SM's 512) asks
// for at least.  CTAs whose shared memory fits on an SM together then have their columns there
// too, whichever of the kernels and streams they come from: three of 256, or 256 beside 512, do
// not fit (228 KB per SM, 1 KB of it reserved per CTA).  Otherwise tcgen05.alloc would wait for a
// resident CTA to end, and two clusters that hold columns on one SM and want them on another
// would wait for each other at their cluster barriers.
constexpr int kSmemPerSM = 228 * 1024;
KD_TC_HD constexpr int tc_smem_floor(int cols) { return kSmemPerSM / 768 * cols; }

}  // namespace kd
