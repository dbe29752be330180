// Run-time-length decompose kernel, 32 < n / 256 <= 44.
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_44() { return gen_decompose_kernel<false, true, 32, 44>; }
}  // namespace kd
