// Run-time-length decompose kernel, 0 < n / 256 <= 4.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_4() { return gen_decompose_kernel<false, true, 0, 4>; }
}  // namespace kd
