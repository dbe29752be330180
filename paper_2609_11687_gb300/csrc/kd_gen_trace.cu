// Run-time-length decompose kernel with the sign trace, any n.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_trace() { return gen_decompose_kernel<true, false, 0, 64>; }
}  // namespace kd
