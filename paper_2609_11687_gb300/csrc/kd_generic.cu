// Host side of the run-time-length path (kd_generic.cuh): plans, tables, dispatch, and its
// kernels for P and the dense re-materialisation.
#include <map>
#include <mutex>

#include "kd_generic.cuh"

namespace kd {

bool gen_plan(int64_t n, GenPlan* g) {
  if (n < 1 || n > kGenMaxN) return false;
  static const int radices[] = {16, 8, 4, 2, 9, 3, 5, 7, 11, 13, 43};
  int rem = (int)n, np = 0;
  for (int r : radices) {
    while (rem % r == 0) {
      if (np == kGenMaxPasses) return false;
      g->R[np++] = r;
      rem /= r;
    }
  }
  if (rem != 1) return false;
  g->n = (int)n;
  g->np = np;
  g->fused = np >= 1 && g->R[np - 1] <= 16;
  int b = (int)n, off = 0;
  for (int i = 0; i < np; ++i) {
    g->B[i] = b;
    g->S[i] = b / g->R[i];
    g->tw[i] = off;
    if (i < np - 1) off += b;
    b = g->S[i];
  }
  g->bufn = 1;
  for (int i = np - 1; i >= 0; --i) {
    g->P[i] = i == np - 1 ? 1 : g->bufn | 1;
    g->bufn = g->P[i] * g->R[i];
  }
  g->woff = off;
  int u32 = 2 * (g->woff + (int)n / 2 + 1);
  for (int i = 0; i < np - g->fused; ++i) {
    g->base[i] = u32;
    u32 += (int)n / g->R[i];
  }
  g->addroff = 2 * u32;
  g->freqoff = g->addroff + (int)n;
  const int u16 = g->freqoff + (g->fused ? (int)n / g->R[np - 1] : (int)n);
  g->twn = (u16 + 3) / 4;
  return true;
}

namespace {

// y_j = P x_j (fp32, vector-major rows of length n)
__global__ void __launch_bounds__(kGenThreads, 2) gen_apply_kernel(ApplyParams p, const __grid_constant__ GenPlan g) {
  constexpr int T = kGenThreads;
  const int n = g.n;
  const int lt = threadIdx.x;
  gen_stage_plan(g, lt);
  float2* buf = gen_buf();
  void* mask = buf + gen_bufn(g) + kGenRedFloats / 2;
  gen_stage_masks(g, mask, p.eps, lt);  // read after gen_apply's barriers
  const uint16_t* addr = reinterpret_cast<const uint16_t*>(p.twt) + g.addroff;
  for (int64_t pr = blockIdx.x; pr < p.npairs; pr += gridDim.x) {
    const int64_t colA = 2 * pr;
    const bool hasB = (colA + 1) < p.m;
    for (int s = lt; s < n; s += T) {
      const int nat = gen_nat(s, n);
      buf[__ldg(&addr[s])] = make_float2(__ldg(&p.x[colA * n + nat]), hasB ? __ldg(&p.x[(colA + 1) * n + nat]) : 0.f);
    }
    gen_apply(p.twt, p.eps, mask, lt);  // its first barrier orders every load before any store (x, y may alias)
    for (int s = lt; s < n; s += T) {
      const int nat = gen_nat(s, n);
      const float2 v = buf[__ldg(&addr[s])];
      p.y[colA * n + nat] = v.x;
      if (hasB) p.y[(colA + 1) * n + nat] = v.y;
    }
    __syncthreads();
  }
}

// W_hat_j = cu_j[code_u] + P(cv_j[code_v])  (App. C)
__global__ void __launch_bounds__(kGenThreads, 2) gen_reconstruct_kernel(RecParams p, const __grid_constant__ GenPlan g) {
  constexpr int T = kGenThreads;
  const int n = g.n;
  const int WPV = (n + 15) / 16;
  const int lt = threadIdx.x;
  gen_stage_plan(g, lt);
  float2* buf = gen_buf();
  void* mask = buf + gen_bufn(g) + kGenRedFloats / 2;
  gen_stage_masks(g, mask, p.eps, lt);  // read after gen_apply's barriers
  const uint16_t* addr = reinterpret_cast<const uint16_t*>(p.twt) + g.addroff;
  auto pick = [](const float4& c, uint32_t q) -> float {
    const float lo = (q & 1u) ? c.y : c.x;
    const float hi = (q & 1u) ? c.w : c.z;
    return (q & 2u) ? hi : lo;
  };
  for (int64_t pr = blockIdx.x; pr < p.npairs; pr += gridDim.x) {
    const int64_t colA = 2 * pr;
    const bool hasB = (colA + 1) < p.m;
    const int64_t colB = hasB ? colA + 1 : colA;
    const float4 cuA = __ldg(reinterpret_cast<const float4*>(p.centres_u) + colA);
    const float4 cuB = __ldg(reinterpret_cast<const float4*>(p.centres_u) + colB);
    const float4 cvA = __ldg(reinterpret_cast<const float4*>(p.centres_v) + colA);
    const float4 cvB = __ldg(reinterpret_cast<const float4*>(p.centres_v) + colB);
    auto code = [&](const uint32_t* planes, int64_t col, int nat) -> uint32_t {
      return (__ldg(&planes[col * WPV + (nat >> 4)]) >> (2 * (nat & 15))) & 3u;
    };
    for (int s = lt; s < n; s += T) {
      const int nat = gen_nat(s, n);
      buf[__ldg(&addr[s])] = make_float2(pick(cvA, code(p.codes_v, colA, nat)), pick(cvB, code(p.codes_v, colB, nat)));
    }
    gen_apply(p.twt, p.eps, mask, lt);
    for (int nat = lt; nat < n; nat += T) {
      const float2 v = buf[__ldg(&addr[gen_slot(nat, n)])];
      const float a = __fadd_rn(pick(cuA, code(p.codes_u, colA, nat)), v.x);
      store_elem(p.out, p.dtype, elem_index(p.layout, colA, nat, p.ld), a);
      if (hasB) {
        const float b = __fadd_rn(pick(cuB, code(p.codes_u, colB, nat)), v.y);
        store_elem(p.out, p.dtype, elem_index(p.layout, colB, nat, p.ld), b);
      }
    }
    __syncthreads();
  }
}

// Tables of one call: pass twiddles, exp(i pi k/n), group bases, addresses by position and by
// frequency, sign bits (setup_signs) and the cleared status word.  One entry per thread, the
// kinds one after another, each from a block of its own.
__host__ __device__ inline int gen_setup_blocks(const GenPlan& g, int (&first)[6]) {
  int bases = 0;
  for (int i = 0; i < g.np - g.fused; ++i) bases += g.n / g.R[i];
  const int freqs = g.fused ? g.n / g.R[g.np - 1] : g.n;
  const int len[5] = {g.woff, g.n / 2 + 1, bases, g.n, freqs};
  first[0] = 0;
  for (int i = 0; i < 5; ++i) first[i + 1] = first[i] + (len[i] + kSetupThreads - 1) / kSetupThreads;
  return first[5];
}

__global__ void gen_setup_kernel(float2* tab, uint32_t* eps, uint32_t* status, const __grid_constant__ SeedList sl,
                                 const __grid_constant__ GenPlan g) {
  int first[6];
  gen_setup_blocks(g, first);
  const int blk = blockIdx.x;
  const int n = g.n;
  if (blk == 0 && threadIdx.x == 0) *status = 0u;
  auto address = [&](int s) {  // of slot s
    int at = 0;
    for (int i = 0; i < g.np; ++i) {
      const int d = s / g.S[i];
      s -= d * g.S[i];
      at += d * g.P[i];
    }
    return at;
  };
  uint16_t* at16 = reinterpret_cast<uint16_t*>(tab);
  if (blk < first[1]) {
    const int e = blk * kSetupThreads + threadIdx.x;
    if (e >= g.woff) return;
    int i = 0;
    while (i + 1 < g.np - 1 && e >= g.tw[i + 1]) ++i;
    const int r = e - g.tw[i];
    const int j = r / g.S[i], sp = r - j * g.S[i];
    tab[e] = root_w((long long)sp * j, g.B[i]);
  } else if (blk < first[2]) {
    const int k = (blk - first[1]) * kSetupThreads + threadIdx.x;
    if (2 * k <= n) tab[g.woff + k] = expi_pi(k, n);
  } else if (blk < first[3]) {
    int k = (blk - first[2]) * kSetupThreads + threadIdx.x;
    int i = 0;
    while (i < g.np - g.fused && k >= n / g.R[i]) k -= n / g.R[i++];
    if (i == g.np - g.fused) return;
    const int bk = k / g.S[i], sp = k - bk * g.S[i];
    reinterpret_cast<uint32_t*>(tab)[g.base[i] + k] = (uint32_t)address(bk * g.B[i] + sp) | (uint32_t)sp << 16;
  } else if (blk < first[4]) {
    const int s = (blk - first[3]) * kSetupThreads + threadIdx.x;
    if (s < n) at16[g.addroff + s] = (uint16_t)address(s);
  } else if (blk < first[5]) {
    const int k = (blk - first[4]) * kSetupThreads + threadIdx.x;
    if (k >= (g.fused ? n / g.R[g.np - 1] : n)) return;
    int x = k, s = 0;
    for (int i = 0; i < g.np - g.fused; ++i) {
      const int q = x / g.R[i];
      s += (x - q * g.R[i]) * g.S[i];
      x = q;
    }
    at16[g.freqoff + k] = (uint16_t)address(s);
  } else {
    setup_signs(eps, sl, first[5]);
  }
}

// ---------------------------------------------------------------------------
// Host side: PlanOps for one run-time length
// ---------------------------------------------------------------------------
// the decompose kernel for n: positions per thread rounded up; u in the workspace where it
// does not fit beside the exchange buffer, and with the trace
struct GenChoice {
  GenDec kernel;
  bool u_smem;
};
GenChoice gen_choose(const GenPlan& g, bool trace) {
  const int e = (g.n + kGenThreads - 1) / kGenThreads;
  if (trace) return {gen_dec_trace(), false};
  if (!gen_u_smem(g)) return {gen_dec_64(), false};
  if (e <= 4) return {gen_dec_4(), true};
  if (e <= 10) return {gen_dec_10(), true};
  if (e <= 20) return {gen_dec_20(), true};
  if (e <= 32) return {gen_dec_32(), true};
  if (e <= 44) return {gen_dec_44(), true};
  if (e <= 55) return {gen_dec_55(), true};
  return {gen_dec_64(), false};
}

template <class K>
int gen_occupancy(K kernel, size_t smem) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 0;
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kGenThreads, smem) != cudaSuccess) return 0;
  return nb;
}

int gen_ctas(int which, int64_t n) {
  GenPlan g;
  if (!gen_plan(n, &g)) return 0;
  if (which == 0) {
    const GenChoice c = gen_choose(g, false);
    return gen_occupancy(c.kernel, gen_smem(g, c.u_smem));
  }
  if (which == 1) return gen_occupancy(gen_apply_kernel, gen_smem(g, false));
  return gen_occupancy(gen_reconstruct_kernel, gen_smem(g, false));
}

cudaError_t gen_decompose(const DecParams& p, const BatchParams* bp, int grid, cudaStream_t s) {
  GenPlan g;
  if (bp || !gen_plan(p.n, &g)) return cudaErrorInvalidValue;
  const GenChoice c = gen_choose(g, p.trace != nullptr);
  const size_t smem = gen_smem(g, c.u_smem);
  cudaError_t e = cudaFuncSetAttribute(c.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  c.kernel<<<grid, kGenThreads, smem, s>>>(p, g);
  return cudaGetLastError();
}

cudaError_t gen_apply_launch(const ApplyParams& p, const ApplyBatch*, int grid, cudaStream_t s) {
  GenPlan g;
  if (!gen_plan(p.n, &g)) return cudaErrorInvalidValue;
  const size_t smem = gen_smem(g, false);
  cudaError_t e = cudaFuncSetAttribute(gen_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  gen_apply_kernel<<<grid, kGenThreads, smem, s>>>(p, g);
  return cudaGetLastError();
}

cudaError_t gen_reconstruct(const RecParams& p, const RecBatch* rb, int grid, cudaStream_t s) {
  GenPlan g;
  if (rb || !gen_plan(p.n, &g)) return cudaErrorInvalidValue;
  const size_t smem = gen_smem(g, false);
  cudaError_t e = cudaFuncSetAttribute(gen_reconstruct_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  gen_reconstruct_kernel<<<grid, kGenThreads, smem, s>>>(p, g);
  return cudaGetLastError();
}

cudaError_t gen_setup(float2* tab, uint32_t* eps, uint32_t* status, const SeedList& sl, int64_t n, cudaStream_t s) {
  GenPlan g;
  if (!gen_plan(n, &g)) return cudaErrorInvalidValue;
  int first[6];
  const int blocks = gen_setup_blocks(g, first) + sl.count * sl.words * 32 / kSetupThreads;
  gen_setup_kernel<<<blocks, kSetupThreads, 0, s>>>(tab, eps, status, sl, g);
  return cudaGetLastError();
}

}  // namespace

bool generic_length(int64_t n) {
  GenPlan g;
  return gen_plan(n, &g);
}

const PlanOps* generic_plan_ops(int64_t n) {
  GenPlan g;
  if (!gen_plan(n, &g)) return nullptr;
  static std::mutex mu;
  static std::map<int64_t, PlanOps> cache;  // node addresses stay valid
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(n);
  if (it != cache.end()) return &it->second;
  const PlanOps o{(int)n, kGenThreads, 1, gen_smem(g, true), true, false, g.twn,
                  &gen_ctas, &gen_decompose, &gen_apply_launch, &gen_reconstruct, &gen_setup};
  return &cache.emplace(n, o).first->second;
}

}  // namespace kd
