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

}  // namespace kd
