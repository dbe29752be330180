// Run-time-length path: the vector lengths without a compiled plan.
//
// Any n with 1 <= n <= 16384 whose prime factors all lie in {2, 3, 5, 7, 11, 13, 43}
// runs here with the same method and outputs as the per-length plans (Algorithm 1,
// the closed-form centres of Sec. 2.1, the optional k-means refinement, the 2-bit
// codes of App. C; P, and the dense re-materialisation).  What changes is the
// transform's shape, which is chosen when the call is made:
//  - every radix pass of the complex FFT is a shared-memory pass over the pair (two vectors
//    packed as one complex vector, Makhoul order), with the radices 16, 8, 4, 2, 9, 3, 5, 7,
//    11, 13, 43 chosen from the factorisation of n;
//  - one CTA of 256 threads per vector pair holds the pair in registers through each two
//    greedy steps (positions t + 256 j) and in shared memory through P; u lives beside the
//    exchange buffer where both fit in shared memory, else in a per-CTA workspace slot.
//
// Slot layout.  A slot s has one digit per pass (d_i < R_i, stride S_i); it is kept at
// sum d_i P_i with padded strides P_i, all odd (P of the last pass is 1).  The elements of a
// group of any pass are then an arithmetic progression, so a pass adds one stride per element
// where the spare slots of the compiled plans' padding would cost a run-time length a dozen
// integer instructions, and any 16 consecutive values of one digit fall in distinct banks.
// Group bases, the positions' addresses and the frequency groups' come from tables of the
// call's set-up kernel.
//
// Last pass.  Where the last radix is at most 16 a thread takes the two last-pass groups of
// frequencies K + (n/R) j and n - (K + (n/R) j), transforms both, applies the middle
// operator M to the frequency pairs in registers and runs their inverse transforms: no pass
// of its own for M and one exchange less in each direction.
//
// Bound by latency (issue 38 %, the first stall is table loads that miss L1), by the
// instructions around the arithmetic, and from n = 1025 to 8192 by spills: two CTAs per SM leave
// 128 registers a thread, of which E = 10, 20 and 32 spill 96, 840 and 996 bytes (E = 4 and 44
// none).  Measured at 16 blocks, before (run-time padding, a pass
// for M, the greedy steps in shared memory, 288 instructions per element and P, half the
// shared-memory wavefronts conflicts) and now:
//   n = 640 x 8000 2.75 -> 1.91 ms, 2560 x 6000 4.92 -> 3.29, 5120 x 5120 (columns, 3
//   refinements) 8.04 -> 5.92, 10000 x 2000 9.59 -> 6.24, 12288 x 2000 9.68 -> 6.35,
//   13824 x 2000 12.73 -> 9.94.
// Every result keeps its bits: the same operations on the same values in the same order.
//
// Makhoul's reordering and the middle operator hold for odd n as well (the even
// positions take the first ceil(n/2) slots); the code words of a vector are
// ceil(n/16), the last one padded with zero codes.
#pragma once

#include "kd_kernels.cuh"
#include "kd_ops.h"

namespace kd {

constexpr int kGenMaxPasses = 16;
constexpr int kGenThreads = 256;
constexpr int64_t kGenMaxN = 16384;
constexpr int kGenRedFloats = 160;  // >= 16 (warps + 1) (k-means sums) and 4 warps (l1 sums)

// Team shape for the shared reduction helpers: the whole CTA is one team.
struct GenTeam {
  static constexpr int T = kGenThreads;
  static constexpr int NW = kGenThreads / 32;
};

// Radix passes of one length: pass i splits sub-transforms of length B[i] into
// R[i] interleaved ones of length S[i] = B[i] / R[i] (decimation in frequency).
struct GenPlan {
  int n, np;
  int fused;  // the last pass carries M (np >= 1 and its radix <= 16)
  int R[kGenMaxPasses], S[kGenMaxPasses], B[kGenMaxPasses];
  int P[kGenMaxPasses];     // address stride of pass i's digit
  int tw[kGenMaxPasses];    // float2 offset of pass i's twiddles [j][s] = W_{B[i]}^{s j} (not the last pass)
  int base[kGenMaxPasses];  // uint32 offset of pass i's groups: address of the first element | s << 16
  int bufn;                 // float2 slots of the exchange buffer
  int woff;                 // float2 offset of exp(i pi k / n), k = 0 .. n/2
  int addroff;              // uint16 offset of the positions' addresses, s < n
  int freqoff;              // uint16 offset of addresses by frequency: of the last-pass group of k, k < n / R (fused),
                            // or of frequency k itself, k < n
  int twn;                  // float2 units of the whole table
};

bool gen_plan(int64_t n, GenPlan* g);  // false: n has no plan

// Shared memory: [plan][exchange buffer, later the code bytes][reduction slots][sign masks of the
// last pass][u, if it fits].
constexpr int kGenPlanSlots = (sizeof(GenPlan) + 15) / 16 * 2;  // float2 slots
KD_HD inline int gen_bufn(const GenPlan& g) {
  const int codes = (4 * ((g.n + 15) / 16 * 16) + 7) / 8;  // float2 slots of four planes of code bytes
  return ((g.bufn > codes ? g.bufn : codes) + 1) / 2 * 2;
}
// float2 slots of the sign masks: one for each pair of last-pass groups, of twice as many bits
// as the last radix has values (16 up to radix 8: n = 13824 then fits with u)
KD_HD inline int gen_maskn(const GenPlan& g) {
  if (!g.fused) return 0;
  const int R = g.R[g.np - 1], bytes = (g.n / R / 2 + 1) * (R <= 8 ? 2 : 4);
  return (bytes + 15) / 16 * 2;
}
constexpr size_t kGenMaxSmem = 227 * 1024;
inline size_t gen_smem_base(const GenPlan& g) {
  return (size_t)(kGenPlanSlots + gen_bufn(g) + gen_maskn(g)) * sizeof(float2) + kGenRedFloats * sizeof(float);
}
inline bool gen_u_smem(const GenPlan& g) { return gen_smem_base(g) + (size_t)g.n * sizeof(float2) <= kGenMaxSmem; }
inline size_t gen_smem(const GenPlan& g, bool u) { return gen_smem_base(g) + (u && gen_u_smem(g) ? (size_t)g.n * sizeof(float2) : 0); }

// Natural index of Makhoul slot s, and its inverse (any n).
__device__ __forceinline__ int gen_nat(int s, int n) { return s < ((n + 1) >> 1) ? 2 * s : 2 * n - 1 - 2 * s; }
__device__ __forceinline__ int gen_slot(int nat, int n) { return (nat & 1) ? n - ((nat + 1) >> 1) : nat >> 1; }

extern __shared__ __align__(16) float2 gen_smem_mem[];
__device__ __forceinline__ const GenPlan& gen_shared_plan() { return *reinterpret_cast<const GenPlan*>(gen_smem_mem); }
__device__ __forceinline__ float2* gen_buf() { return gen_smem_mem + kGenPlanSlots; }

// the call's plan into shared memory (the passes read it there)
__device__ __forceinline__ void gen_stage_plan(const GenPlan& g, int lt) {
  const int* src = reinterpret_cast<const int*>(&g);
  for (int i = lt; i < (int)(sizeof(GenPlan) / 4); i += kGenThreads) reinterpret_cast<int*>(gen_smem_mem)[i] = src[i];
  __syncthreads();
}

// One shared-memory radix pass over all groups of the pair buffer.  Forward (DIR < 0):
// DFT then the twiddles of the next level; inverse: conjugate twiddles then IDFT.  A last
// pass has no twiddles.
template <int R, int DIR>
__device__ __forceinline__ void gen_pass_r(float2* buf, const float2* __restrict__ tw, const uint32_t* __restrict__ base,
                                           int G, uint32_t S, int P, bool last, int lt) {
  for (int g = lt; g < G; g += kGenThreads) {
    const uint32_t e = __ldg(&base[g]);
    float2* q = buf + (e & 0xFFFFu);
    const uint32_t sp = e >> 16;
    if constexpr (kd_is_big_prime<R>()) {
      // streaming form (Rader's for 43, direct otherwise): every load precedes the first store
      if constexpr (DIR < 0) {
        dft_prime_pass<R, -1>([&](auto jc) { return q[decltype(jc)::value * P]; },
                                [&](auto kc, float2 x) {
                                  constexpr int K = decltype(kc)::value;
                                  if (K > 0 && !last) x = cmul(x, __ldg(&tw[K * S + sp]));
                                  q[K * P] = x;
                                });
      } else {
        dft_prime_pass<R, +1>(
            [&](auto jc) {
              constexpr int J = decltype(jc)::value;
              float2 x = q[J * P];
              if (J > 0 && !last) x = cmulc(x, __ldg(&tw[J * S + sp]));
              return x;
            },
            [&](auto kc, float2 x) { q[decltype(kc)::value * P] = x; });
      }
    } else {
      float2 v[R];
#pragma unroll
      for (int j = 0; j < R; ++j) v[j] = q[j * P];
      if constexpr (DIR < 0) {
        Dft<R, -1>::run(v);
        if (!last) {
#pragma unroll
          for (int j = 1; j < R; ++j) v[j] = cmul(v[j], __ldg(&tw[j * S + sp]));
        }
      } else {
        if (!last) {
#pragma unroll
          for (int j = 1; j < R; ++j) v[j] = cmulc(v[j], __ldg(&tw[j * S + sp]));
        }
        Dft<R, +1>::run(v);
      }
#pragma unroll
      for (int j = 0; j < R; ++j) q[j * P] = v[j];
    }
  }
}

template <int DIR>
__device__ __forceinline__ void gen_pass(const GenPlan& g, int i, float2* buf, const float2* __restrict__ tab, int lt) {
  const bool last = (i == g.np - 1);
  const float2* tw = tab + g.tw[i];
  const uint32_t* base = reinterpret_cast<const uint32_t*>(tab) + g.base[i];
  const uint32_t S = (uint32_t)g.S[i];
  const int P = g.P[i], R = g.R[i], G = g.n / R;
  switch (R) {
    case 16: gen_pass_r<16, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 8: gen_pass_r<8, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 4: gen_pass_r<4, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 2: gen_pass_r<2, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 9: gen_pass_r<9, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 3: gen_pass_r<3, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 5: gen_pass_r<5, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 7: gen_pass_r<7, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 11: gen_pass_r<11, DIR>(buf, tw, base, G, S, P, last, lt); break;
    case 13: gen_pass_r<13, DIR>(buf, tw, base, G, S, P, last, lt); break;
    default: gen_pass_r<43, DIR>(buf, tw, base, G, S, P, last, lt); break;
  }
}

// M on the frequency pair (k, n - k), 0 < 2 k < n, 1/n folded in: if eps_k == eps_{n-k},
// Z'_k = eps_k Z_k / n and Z'_{n-k} = eps_k Z_{n-k} / n; otherwise (diff) Z'_k = eps_k w_k Z_{n-k} / n
// and Z'_{n-k} = eps_k conj(w_k) Z_k / n (w_k = exp(i pi k/n)).  neg: eps_k < 0.
__device__ __forceinline__ void gen_mpair(float2& a, float2& b, int k, bool neg, bool diff, float inv,
                                          const float2* __restrict__ wk) {
  const float f = neg ? -inv : inv;
  float2 za = a, zb = b;
  if (diff) {
    const float2 w = __ldg(&wk[k]);
    za = cmul(b, w);
    zb = cmulc(a, w);
  }
  a = make_float2(__fmul_rn(za.x, f), __fmul_rn(za.y, f));
  b = make_float2(__fmul_rn(zb.x, f), __fmul_rn(zb.y, f));
}

// M on a frequency that pairs with itself (0 and n/2): Z'_k = eps_k Z_k / n
__device__ __forceinline__ void gen_mself(float2& a, bool neg, float inv) {
  const float f = neg ? -inv : inv;
  a = make_float2(__fmul_rn(a.x, f), __fmul_rn(a.y, f));
}

// Frequencies of the last pass.  Group p holds the frequencies p + M j (M = n / R) in its R
// consecutive slots, its partner group M - p their mirrors in reverse; p = 0 (j against
// R - j) and p = M / 2 pair with themselves.  Item p < M / 2 takes both groups: pair q has
// the lower frequency k(q) = p + M q for q < (R + 1) / 2, then M - p + M (q - (R + 1) / 2).
// Its sign mask has eps_k < 0 at bit q and eps_k != eps_{n-k} in its upper half (q <= 8 pairs for
// the two groups that pair with themselves, q = 0 or R / 2 the frequency 0 or n/2).
__device__ __forceinline__ void gen_stage_masks(const GenPlan& g, void* mask, const uint32_t* __restrict__ eb, int lt) {
  if (!g.fused) return;
  const int n = g.n, R = g.R[g.np - 1], M = n / R, h = (R + 1) / 2, up = R <= 8 ? 8 : 16;
  for (int p = lt; 2 * p <= M; p += kGenThreads) {
    uint32_t m = 0;
    for (int q = 0; q < R; ++q) {
      const int k = q < h ? p + M * q : M - p + M * (q - h);
      if (2 * k > n) continue;
      const bool e = eps_neg(eb, k), d = k > 0 && e != eps_neg(eb, n - k);
      m |= (uint32_t)e << q | (uint32_t)d << (up + q);
    }
    if (p == 0 && R % 2 == 0) {  // frequency n/2, pair q = R / 2 of group 0
      m &= ~(1u << (R / 2) | 1u << (up + R / 2));
      m |= (uint32_t)eps_neg(eb, n / 2) << (R / 2);
    }
    if (R <= 8) static_cast<uint16_t*>(mask)[p] = (uint16_t)m;
    else static_cast<uint32_t*>(mask)[p] = m;
  }
}

// Last pass forward, M, last pass inverse.
template <int R>
__device__ __forceinline__ void gen_last_r(float2* buf, int n, const float2* __restrict__ wk,
                                           const uint16_t* __restrict__ freq, const void* mask, int lt) {
  using Word = typename std::conditional<(R <= 8), uint16_t, uint32_t>::type;
  constexpr int H = (R + 1) / 2, UP = R <= 8 ? 8 : 16;
  const int M = n / R;
  const float inv = __fdiv_rn(1.f, (float)n);
  for (int p = lt; 2 * p <= M; p += kGenThreads) {
    float2* q = buf + __ldg(&freq[p]);
    const uint32_t m = static_cast<const Word*>(mask)[p];
    auto pair = [&](float2& a, float2& b, int k, int bit) {
      gen_mpair(a, b, k, (m >> bit) & 1u, (m >> (UP + bit)) & 1u, inv, wk);
    };
    float2 v[R];
#pragma unroll
    for (int j = 0; j < R; ++j) v[j] = q[j];
    if (p > 0 && 2 * p < M) {
      float2* q2 = buf + __ldg(&freq[M - p]);
      float2 w[R];
#pragma unroll
      for (int j = 0; j < R; ++j) w[j] = q2[j];
      Dft<R, -1>::run(v);
      Dft<R, -1>::run(w);
#pragma unroll
      for (int j = 0; j < H; ++j) pair(v[j], w[R - 1 - j], p + M * j, j);
#pragma unroll
      for (int j = 0; j < R / 2; ++j) pair(w[j], v[R - 1 - j], M - p + M * j, H + j);
      Dft<R, +1>::run(w);
#pragma unroll
      for (int j = 0; j < R; ++j) q2[j] = w[j];
    } else {
      Dft<R, -1>::run(v);
      if (p == 0) {
        gen_mself(v[0], m & 1u, inv);
#pragma unroll
        for (int j = 1; j < H; ++j) pair(v[j], v[R - j], M * j, j);
        if constexpr (R % 2 == 0) gen_mself(v[R / 2], (m >> (R / 2)) & 1u, inv);
      } else {
#pragma unroll
        for (int j = 0; j < R / 2; ++j) pair(v[j], v[R - 1 - j], p + M * j, j);
        if constexpr (R % 2 == 1) gen_mself(v[R / 2], (m >> (R / 2)) & 1u, inv);
      }
    }
    Dft<R, +1>::run(v);
#pragma unroll
    for (int j = 0; j < R; ++j) q[j] = v[j];
  }
}

__device__ __forceinline__ void gen_last(const GenPlan& g, float2* buf, const float2* __restrict__ tab,
                                         const void* mask, int lt) {
  const float2* wk = tab + g.woff;
  const uint16_t* freq = reinterpret_cast<const uint16_t*>(tab) + g.freqoff;
  const int n = g.n;
  switch (g.R[g.np - 1]) {
    case 16: gen_last_r<16>(buf, n, wk, freq, mask, lt); break;
    case 8: gen_last_r<8>(buf, n, wk, freq, mask, lt); break;
    case 4: gen_last_r<4>(buf, n, wk, freq, mask, lt); break;
    case 2: gen_last_r<2>(buf, n, wk, freq, mask, lt); break;
    case 9: gen_last_r<9>(buf, n, wk, freq, mask, lt); break;
    case 3: gen_last_r<3>(buf, n, wk, freq, mask, lt); break;
    case 5: gen_last_r<5>(buf, n, wk, freq, mask, lt); break;
    case 7: gen_last_r<7>(buf, n, wk, freq, mask, lt); break;
    case 11: gen_last_r<11>(buf, n, wk, freq, mask, lt); break;
    default: gen_last_r<13>(buf, n, wk, freq, mask, lt); break;
  }
}

// M as a pass of its own, where the last radix is 43 (or n is 1)
__device__ __forceinline__ void gen_middle(const GenPlan& g, float2* buf, const float2* __restrict__ tab,
                                           const uint32_t* __restrict__ eb, int lt) {
  const int n = g.n;
  const float2* wk = tab + g.woff;
  const uint16_t* freq = reinterpret_cast<const uint16_t*>(tab) + g.freqoff;
  const float inv = __fdiv_rn(1.f, (float)n);
  for (int k = lt; 2 * k <= n; k += kGenThreads) {
    const int sa = __ldg(&freq[k]);
    float2 a = buf[sa];
    if (k == 0 || 2 * k == n) {
      gen_mself(a, eps_neg(eb, k), inv);
    } else {
      const int sb = __ldg(&freq[n - k]);
      float2 b = buf[sb];
      const bool ek = eps_neg(eb, k);
      gen_mpair(a, b, k, ek, ek != eps_neg(eb, n - k), inv, wk);
      buf[sb] = b;
    }
    buf[sa] = a;
  }
}

// buf <- P' buf (both packed vectors, Makhoul order in and out).  Starts with a
// barrier (callers have just written their own slots) and ends with one.
__device__ __forceinline__ void gen_apply(const float2* __restrict__ tab, const uint32_t* __restrict__ eb,
                                          const void* mask, int lt) {
  const GenPlan& g = gen_shared_plan();
  float2* buf = gen_buf();
  __syncthreads();
  const int np = g.np, full = np - g.fused;
  for (int i = 0; i < full; ++i) {
    gen_pass<-1>(g, i, buf, tab, lt);
    __syncthreads();
  }
  if (g.fused) gen_last(g, buf, tab, mask, lt);
  else gen_middle(g, buf, tab, eb, lt);
  __syncthreads();
  for (int i = full - 1; i >= 0; --i) {
    gen_pass<+1>(g, i, buf, tab, lt);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Decomposition: the steps, normalisation, centres, refinement and codes of the
// per-length kernel.  Thread t holds the positions t + 256 j, j < E (masked past n;
// EMIN 256 < n <= E 256).
// ---------------------------------------------------------------------------
template <bool TRACE, bool USM, int EMIN, int E>
__global__ void __launch_bounds__(kGenThreads, E <= 32 ? 2 : 1) gen_decompose_kernel(DecParams p, const __grid_constant__ GenPlan g) {
  constexpr int T = kGenThreads;
  const int n = g.n;
  const int lt = threadIdx.x;
  gen_stage_plan(g, lt);
  float2* buf = gen_buf();
  float2* red = buf + gen_bufn(g);
  void* mask = red + kGenRedFloats / 2;
  gen_stage_masks(g, mask, p.eps, lt);  // read after gen_apply's barriers
  uint8_t* cb = reinterpret_cast<uint8_t*>(buf);
  const int WPV = (n + 15) / 16;
  const int PS = WPV * 16;  // code bytes per plane
  const float2* tab = p.twt;
  const uint16_t* addr = reinterpret_cast<const uint16_t*>(tab) + g.addroff;
  float2* uslot;
  if constexpr (USM) uslot = red + kGenRedFloats / 2 + gen_maskn(g);
  else uslot = p.uslots + (int64_t)blockIdx.x * n;
  int parity = 0;
  const int nsteps = 4 * p.iters + 2 * p.kmeans_iters;
  // f(j, s) for every position s = lt + T j of this thread (n > EMIN T).  The thread's first
  // position is opaque: the addresses of all E positions would otherwise be computed before
  // the block loop and spilled.
  auto each = [&](auto&& f) {
    int s0 = lt;
    asm volatile("" : "+r"(s0));
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int s = s0 + j * T;
      if (j < EMIN || s < n) f(j, s);
    }
  };

  for (int64_t pr = blockIdx.x; pr < p.npairs; pr += gridDim.x) {
    const int64_t colA = 2 * pr;
    const bool hasB = (colA + 1) < p.m;
    const int64_t colB = hasB ? colA + 1 : colA;

    float2 r[E];
    float2 acc = make_float2(0.f, 0.f);
    each([&](int j, int s) {
      const int nat = gen_nat(s, n);
      const float a = load_elem(p.w, p.dtype, elem_index(p.layout, colA, nat, p.ld));
      const float b = hasB ? load_elem(p.w, p.dtype, elem_index(p.layout, colB, nat, p.ld)) : 0.f;
      r[j] = make_float2(a, b);
      acc.x = __fadd_rn(acc.x, fabsf(a));
      acc.y = __fadd_rn(acc.y, fabsf(b));
    });
    float2 sum0 = team_sum<GenTeam>(acc, red, lt, parity);
    int sA = 0, sB = 0;
    {
      const bool finA = isfinite(sum0.x), finB = isfinite(sum0.y);
      if (lt == 0 && (!finA || !finB)) atomicOr(p.status, 1u);
      const float cA = __fdiv_rn(sum0.x, (float)n), cB = __fdiv_rn(sum0.y, (float)n);
      if (finA && cA > 0.f) sA = max(-100, min(100, -ilogbf(cA)));
      if (finB && cB > 0.f) sB = max(-100, min(100, -ilogbf(cB)));
    }
    const float scA = pow2f(sA), scB = pow2f(sB);
    const float isA = pow2f(-sA), isB = pow2f(-sB);
    const bool liveA = sum0.x > 0.f, liveB = sum0.y > 0.f;
    each([&](int j, int s) {
      r[j] = make_float2(__fmul_rn(r[j].x, scA), __fmul_rn(r[j].y, scB));
      uslot[s] = make_float2(0.f, 0.f);
    });
    sum0 = make_float2(__fmul_rn(sum0.x, scA), __fmul_rn(sum0.y, scB));
    float2 coef[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) coef[q] = make_float2(0.f, 0.f);

    int8_t* trA = nullptr;
    int8_t* trB = nullptr;
    if (TRACE) {
      trA = p.trace + colA * (int64_t)nsteps * n;
      trB = p.trace + colB * (int64_t)nsteps * n;
    }

    // one atomic greedy step on the pair's residual (see the per-length kernel)
    auto greedy = [&](int step, bool have_sum, bool upd_u) -> float2 {
      float2 sm = sum0;
      if (!have_sum) {
        float2 a = make_float2(0.f, 0.f);
        each([&](int j, int) {
          a.x = __fadd_rn(a.x, fabsf(r[j].x));
          a.y = __fadd_rn(a.y, fabsf(r[j].y));
        });
        sm = team_sum<GenTeam>(a, red, lt, parity);
      }
      const float lA = __fdiv_rn(sm.x, (float)n);
      const float lB = __fdiv_rn(sm.y, (float)n);
      each([&](int j, int s) {
        if (TRACE) {
          const int64_t off = (int64_t)step * n + gen_nat(s, n);
          trA[off] = (int8_t)((r[j].x > 0.f) - (r[j].x < 0.f));
          if (hasB) trB[off] = (int8_t)((r[j].y > 0.f) - (r[j].y < 0.f));
        }
        const float dA = signed_step(r[j].x, lA);
        const float dB = signed_step(r[j].y, lB);
        r[j].x = __fsub_rn(r[j].x, dA);
        r[j].y = __fsub_rn(r[j].y, dB);
        if (upd_u) {
          float2 uj = uslot[s];
          uj.x = __fadd_rn(uj.x, dA);
          uj.y = __fadd_rn(uj.y, dB);
          uslot[s] = uj;
        }
      });
      return make_float2(lA, lB);
    };

    int step = 0;
    const int HB = 2 * p.iters;
    for (int hb = 0; hb <= HB; ++hb) {
      if (hb == HB) {
        // r -> x - u - r: its P is vhat (P^2 = I)
        each([&](int j, int s) {
          const int nat = gen_nat(s, n);
          if (p.resid) {
            p.resid[colA * n + nat] = __fmul_rn(r[j].x, isA);
            if (hasB) p.resid[colB * n + nat] = __fmul_rn(r[j].y, isB);
          }
          const float a = __fmul_rn(load_elem(p.w, p.dtype, elem_index(p.layout, colA, nat, p.ld)), scA);
          const float b = hasB ? __fmul_rn(load_elem(p.w, p.dtype, elem_index(p.layout, colB, nat, p.ld)), scB) : 0.f;
          const float2 uj = uslot[s];
          r[j] = (p.iters == 0) ? make_float2(0.f, 0.f)
                                : make_float2(__fsub_rn(__fsub_rn(a, uj.x), r[j].x), __fsub_rn(__fsub_rn(b, uj.y), r[j].y));
        });
        if (p.iters == 0) break;
      } else if ((hb & 1) == 0) {
        const float2 l1 = greedy(step++, hb == 0, true);
        const float2 l2 = greedy(step++, false, true);
        if (hb == 0) {
          coef[0] = l1;
          coef[1] = l2;
        }
      } else {
        const float2 l3 = greedy(step++, false, false);
        const float2 l4 = greedy(step++, false, false);
        if (hb == 1) {
          coef[2] = l3;
          coef[3] = l4;
        }
      }
      each([&](int j, int s) { buf[__ldg(&addr[s])] = r[j]; });
      gen_apply(tab, p.eps, mask, lt);
      each([&](int j, int s) {
        const float2 v = buf[__ldg(&addr[s])];
        r[j] = make_float2(liveA ? v.x : 0.f, liveB ? v.y : 0.f);
      });
    }
    // r now holds vhat
    if (p.u || p.vhat) {
      each([&](int j, int s) {
        const int nat = gen_nat(s, n);
        const float2 uj = uslot[s];
        if (p.u) {
          p.u[colA * n + nat] = __fmul_rn(uj.x, isA);
          if (hasB) p.u[colB * n + nat] = __fmul_rn(uj.y, isB);
        }
        if (p.vhat) {
          p.vhat[colA * n + nat] = __fmul_rn(r[j].x, isA);
          if (hasB) p.vhat[colB * n + nat] = __fmul_rn(r[j].y, isB);
        }
      });
    }

    // closed-form centres (Sec. 2.1) and boundaries, as in the per-length kernel
    float cen[2][2][4];
    float bnd[2][2][3];
    {
      const float a1[2][2] = {{coef[0].x, coef[0].y}, {coef[2].x, coef[2].y}};
      const float a2[2][2] = {{coef[1].x, coef[1].y}, {coef[3].x, coef[3].y}};
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float outer = __fadd_rn(a1[f][c], a2[f][c]);
          const float inner = fabsf(__fsub_rn(a1[f][c], a2[f][c]));
          cen[f][c][0] = -outer;
          cen[f][c][1] = -inner;
          cen[f][c][2] = inner;
          cen[f][c][3] = outer;
          const float mm = fmaxf(a1[f][c], a2[f][c]);
          bnd[f][c][0] = -mm;
          bnd[f][c][1] = 0.f;
          bnd[f][c][2] = mm;
        }
    }
    auto code_of = [](float x, const float (&b)[3]) -> int { return (x > b[0]) + (x > b[1]) + (x > b[2]); };
    for (int it = 0; it < p.kmeans_iters; ++it) {
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        // [c*8 + q]: sum above b_q; [c*8 + 3 + q]: count above b_q; [c*8 + 6]: total
        float acc16[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) acc16[i] = 0.f;
        each([&](int j, int s) {
          const float2 fv = f ? r[j] : uslot[s];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const float x = c ? fv.y : fv.x;
            if (TRACE && (c == 0 || hasB))
              (c ? trB : trA)[(int64_t)(4 * p.iters + 2 * it + f) * n + gen_nat(s, n)] = (int8_t)code_of(x, bnd[f][c]);
            acc16[c * 8 + 6] = __fadd_rn(acc16[c * 8 + 6], x);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              const bool gt = x > bnd[f][c][q];
              acc16[c * 8 + q] = __fadd_rn(acc16[c * 8 + q], gt ? x : 0.f);
              acc16[c * 8 + 3 + q] = __fadd_rn(acc16[c * 8 + 3 + q], gt ? 1.f : 0.f);
            }
          }
        });
        float tot[16];
        team_sum_k<GenTeam, 16>(acc16, tot, reinterpret_cast<float*>(red), lt);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float* t = tot + c * 8;
          const float sum[4] = {__fsub_rn(t[6], t[0]), __fsub_rn(t[0], t[1]), __fsub_rn(t[1], t[2]), t[2]};
          const float cnt[4] = {__fsub_rn((float)n, t[3]), __fsub_rn(t[3], t[4]), __fsub_rn(t[4], t[5]), t[5]};
#pragma unroll
          for (int qq = 0; qq < 4; ++qq)
            if (cnt[qq] > 0.f) cen[f][c][qq] = __fdiv_rn(sum[qq], cnt[qq]);
#pragma unroll
          for (int qq = 0; qq < 3; ++qq) bnd[f][c][qq] = __fmul_rn(0.5f, __fadd_rn(cen[f][c][qq], cen[f][c][qq + 1]));
        }
      }
    }

    // 2-bit codes: nearest centre (ties low), one byte per entry, packed 16 per word
    __syncthreads();  // everyone has read its slots of buf
    each([&](int j, int s) {
      const int nat = gen_nat(s, n);
      const float2 uj = uslot[s];
      cb[0 * PS + nat] = (uint8_t)code_of(uj.x, bnd[0][0]);
      cb[1 * PS + nat] = (uint8_t)code_of(uj.y, bnd[0][1]);
      cb[2 * PS + nat] = (uint8_t)code_of(r[j].x, bnd[1][0]);
      cb[3 * PS + nat] = (uint8_t)code_of(r[j].y, bnd[1][1]);
    });
    for (int i = n + lt; i < PS; i += T) {
#pragma unroll
      for (int plane = 0; plane < 4; ++plane) cb[plane * PS + i] = 0;
    }
    __syncthreads();
    for (int wi = lt; wi < 4 * WPV; wi += T) {
      const int plane = wi / WPV;
      const int word = wi - plane * WPV;
      const bool isB = (plane & 1) != 0;
      if (isB && !hasB) continue;
      const uint4 q = *reinterpret_cast<const uint4*>(cb + plane * PS + word * 16);
      const uint32_t qq[4] = {q.x, q.y, q.z, q.w};
      uint32_t packed = 0;
#pragma unroll
      for (int b4 = 0; b4 < 4; ++b4) {
#pragma unroll
        for (int by = 0; by < 4; ++by) packed |= ((qq[b4] >> (8 * by)) & 3u) << (2 * (4 * b4 + by));
      }
      uint32_t* dst = (plane < 2) ? p.codes_u : p.codes_v;
      dst[(isB ? colB : colA) * WPV + word] = packed;
    }
    if (lt == 0) {
      const float sc[2] = {isA, isB};
      for (int v2 = 0; v2 < (hasB ? 2 : 1); ++v2) {
        const int64_t col = v2 ? colB : colA;
        const float f = sc[v2];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq) {
          p.centres_u[col * 4 + qq] = __fmul_rn(cen[0][v2][qq], f);
          p.centres_v[col * 4 + qq] = __fmul_rn(cen[1][v2][qq], f);
        }
        if (p.coeffs) {
          float* co = p.coeffs + col * 4;
          co[0] = __fmul_rn(v2 ? coef[0].y : coef[0].x, f);
          co[1] = __fmul_rn(v2 ? coef[1].y : coef[1].x, f);
          co[2] = __fmul_rn(v2 ? coef[2].y : coef[2].x, f);
          co[3] = __fmul_rn(v2 ? coef[3].y : coef[3].x, f);
        }
      }
    }
    __syncthreads();  // buf and the code bytes are reused by the next pair
  }
}

using GenDec = void (*)(DecParams, GenPlan);
// the decompose kernels, one translation unit each (kd_gen_<E>.cu): 256 EMIN < n <= 256 E,
// u in shared memory but for the last two
GenDec gen_dec_4();
GenDec gen_dec_10();
GenDec gen_dec_20();
GenDec gen_dec_32();
GenDec gen_dec_44();
GenDec gen_dec_55();
GenDec gen_dec_64();
GenDec gen_dec_trace();

}  // namespace kd
