// Launch helpers shared by the per-N translation units.
#pragma once

#include "kd_kernels.cuh"
#include "kd_ops.h"

namespace kd {

// Opt the kernel in to its dynamic shared memory (> 48 KB for large N).  Done on
// every launch: the attribute is per function and per device, and the call
// costs about a microsecond next to millisecond-scale kernels.
template <class K>
inline cudaError_t prepare(K kernel, size_t smem) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <class K>
inline int occupancy(K kernel, int threads, size_t smem) {
  if (prepare(kernel, smem) != cudaSuccess) return 0;
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem) != cudaSuccess) return 0;
  return nb;
}

// The plan of the kernels without u (P and the re-materialisation): the length's own, or one
// with the same tables that keeps nothing for u (kd_plans.cuh).
template <class PL>
struct LightPlan {
  using type = PL;
};

template <class PL>
struct Ops {
  using LP = typename LightPlan<PL>::type;
  static_assert(LP::N == PL::N && LP::THREADS == PL::THREADS && LP::Q == PL::Q && LP::TWN == PL::TWN &&
                    LP::TW2 == PL::TW2 && Xform<LP>::CWN == Xform<PL>::CWN && LP::BATCH == PL::BATCH,
                "one set of tables serves both");
  static cudaError_t decompose(const DecParams& p, const BatchParams* bp, int grid, cudaStream_t s) {
    auto k = p.trace ? decompose_kernel<PL, true> : decompose_kernel<PL, false>;
    cudaError_t e = prepare(k, PL::SMEM);
    if (e != cudaSuccess) return e;
    if (bp) {
      k<<<grid, PL::THREADS, PL::SMEM, s>>>(p, *bp);
    } else {
      BatchParams none{};
      k<<<grid, PL::THREADS, PL::SMEM, s>>>(p, none);
    }
    return cudaGetLastError();
  }
  static cudaError_t reconstruct(const RecParams& p, const RecBatch* rb, int grid, cudaStream_t s) {
    auto k = reconstruct_kernel<LP>;
    cudaError_t e = prepare(k, LP::SMEM);
    if (e != cudaSuccess) return e;
    if (rb) {
      k<<<grid, LP::THREADS, LP::SMEM, s>>>(p, *rb);
    } else {
      RecBatch none{};
      k<<<grid, LP::THREADS, LP::SMEM, s>>>(p, none);
    }
    return cudaGetLastError();
  }
  static cudaError_t apply(const ApplyParams& p, const ApplyBatch* ab, int grid, cudaStream_t s) {
    auto k = apply_p_kernel<LP>;
    cudaError_t e = prepare(k, LP::SMEM);
    if (e != cudaSuccess) return e;
    if (ab) {
      k<<<grid, LP::THREADS, LP::SMEM, s>>>(p, *ab);
    } else {
      ApplyBatch none{};
      k<<<grid, LP::THREADS, LP::SMEM, s>>>(p, none);
    }
    return cudaGetLastError();
  }
  static cudaError_t setup(float2* twt, uint32_t* eps, uint32_t* status, const SeedList& sl, int64_t, cudaStream_t s) {
    const int blocks = setup_table_blocks<PL>() + sl.count * sl.words * 32 / kSetupThreads;
    setup_kernel<PL><<<blocks, kSetupThreads, 0, s>>>(twt, eps, status, sl);
    return cudaGetLastError();
  }
  static int ctas_per_sm(int which, int64_t) {
    if (which == 0) return occupancy(decompose_kernel<PL, false>, PL::THREADS, PL::SMEM);
    if (which == 1) return occupancy(apply_p_kernel<LP>, LP::THREADS, LP::SMEM);
    return occupancy(reconstruct_kernel<LP>, LP::THREADS, LP::SMEM);
  }
  static const PlanOps* ops() {
    static const PlanOps o{PL::N, PL::THREADS, PL::Q, PL::SMEM, PL::UMODE == UGMEM, PL::BATCH, PL::TWN + Xform<PL>::CWN,
                           &Ops::ctas_per_sm, &Ops::decompose, &Ops::apply, &Ops::reconstruct, &Ops::setup};
    return &o;
  }
};

}  // namespace kd
