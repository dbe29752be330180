// Run-time-length decompose kernel, 20 < n / 256 <= 32.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_32() { return gen_decompose_kernel<false, true, 20, 32>; }
}  // namespace kd
