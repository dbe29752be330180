// Run-time-length decompose kernel, 10 < n / 256 <= 20.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_20() { return gen_decompose_kernel<false, true, 10, 20>; }
}  // namespace kd
