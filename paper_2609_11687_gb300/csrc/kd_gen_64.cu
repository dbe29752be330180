// Run-time-length decompose kernel, u in the workspace (44 < n / 256 <= 64).
#include "kd_generic.cuh"

namespace kd {
GenDec gen_dec_64() { return gen_decompose_kernel<false, false, 44, 64>; }
}  // namespace kd
