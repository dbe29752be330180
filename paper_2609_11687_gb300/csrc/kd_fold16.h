// The two kernels of the 16-bit 2-bit product (kd_fold16.cu: up to 8 batch rows,
// kd_fold16_tc.cu: more).
#pragma once

#include <cuda_runtime.h>

#include "kashin.h"

namespace kd {

// kd_matmul_2bit_f16_batch (bf: _bf16_batch) on validated descriptors, batch >= 1 and at
// least one matrix with m > 0
kd_status fold16_tc_run(const kd_fold_mat_f16* mats, int count, int64_t batch, cudaStream_t s, bool bf);

}  // namespace kd
