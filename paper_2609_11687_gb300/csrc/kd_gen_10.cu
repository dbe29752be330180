// Run-time-length decompose kernel, 4 < n / 256 <= 10.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_10() { return gen_decompose_kernel<false, true, 4, 10>; }
}  // namespace kd
