// Run-time-length decompose kernel, 44 < n / 256 <= 55.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_55() { return gen_decompose_kernel<false, true, 44, 55>; }
}  // namespace kd
