// The tcgen05 kernel of the 16-bit 2-bit product (kd_fold16.cu has the other one and the choice).
#pragma once

#include <cuda_runtime.h>

#include "kashin.h"

namespace kd {

// kd_matmul_2bit_f16_batch (bf: _bf16_batch) on validated descriptors, batch >= 1
kd_status fold16_tc_run(const kd_fold_mat_f16* mats, int count, int64_t batch, cudaStream_t s, bool bf);

}  // namespace kd
