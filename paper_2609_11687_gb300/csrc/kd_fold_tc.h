// The tensor-core form of the fp32 2-bit product (kd_fold_tc.cu).
#pragma once

#include <cuda_runtime.h>

#include "kashin.h"

namespace kd {

// kd_matmul_2bit_batch on validated descriptors, batch >= 1
kd_status fold_tc_run(const kd_fold_mat* mats, int count, int64_t batch, cudaStream_t s);

}  // namespace kd
