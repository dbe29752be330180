// The folded 2-bit layer product of App. C, straight from the code planes:
//
//     Y = X W_hat^T,   W_hat = U_q + P V_q   (vector j of W_hat = output channel j)
//       = X U_q^T + (X P) V_q^T               (P symmetric)
//     y[r][j] = sum_i cu_j[code_u(j, i)] x[r][i] + sum_i cv_j[code_v(j, i)] xp[r][i]
//
// with xp = X P from kd_apply_p.  Neither U_q nor V_q is expanded: every weight costs
// its 2-bit code in each plane (0.5 byte per weight in all), read once from HBM.
//
// This file holds the argument checks, the entry points and the table-lookup kernel for few
// batch rows; the others take kd_fold_tc.cu, on the tensor cores, 16 rows in one pass over the
// codes (by_lookup has the line and both sides' times).
//
// Mapping.  One launch serves up to KD_MAX_BATCH matrices (a layer): persistent CTAs
// of eight warps walk the work items (matrix, tile of RT = 16 / B output channels), for B
// batch rows (blockIdx.y).
// Per item each warp takes slices of 32 consecutive code words (512 inputs): it loads
// its lane's 16 inputs of x and xp (L2-resident, shared by every item of the matrix)
// into registers, then the code words of all RT channels of the tile (one coalesced
// word per channel, plane and lane, all in flight together).  Two codes at a time (4
// bits) index a per-channel table of the 16 centre pairs (c[q0], c[q1]) in shared
// memory: one 64-bit shared load and one packed FP32x2 FMA per two weights, plane
// and batch row.  The lanes' and warps' partial sums are added in a fixed order
// (deterministic results, the same for one row and for two).
#include <cuda_runtime.h>

#include "kashin.h"
#include "kd_fold_tc.h"
#include "kd_tc.cuh"

namespace kd {
namespace {

constexpr int kFoldWarps = 8;
constexpr int kFoldThreads = 32 * kFoldWarps;

struct FoldMat {
  const uint32_t* codes_u;
  const uint32_t* codes_v;
  const float* centres_u;
  const float* centres_v;
  const float* x;
  const float* xp;
  float* y;
  int64_t n, m, words, ldx, ldy;
  int64_t tile0;  // first work item of this matrix
  int vec;        // x and xp 16-byte aligned with ldx a multiple of 4: 128-bit input loads
};

struct FoldParams {
  int count;
  int rows;        // batch rows of the call
  int64_t items;   // work items of all matrices, once for each B rows (blockIdx.y)
  FoldMat mat[KD_MAX_BATCH];
};

// RT x B = 16 partial sums per lane
template <int B>
struct FoldTile {
  static constexpr int RT = 16 / B;
};

// MANY: more than B batch rows (without, the row offsets fold away: 7B layer, two rows, 131 ->
// 125 us)
template <int B, bool MANY>
__global__ void __launch_bounds__(kFoldThreads, 2) fold_kernel(const __grid_constant__ FoldParams p) {
  constexpr int RT = FoldTile<B>::RT;
  constexpr int K = RT * B;  // partial sums per lane
  static_assert(K == 16, "the reduction scatters 16 values per lane");
  __shared__ float2 tab[2 * RT * 16];
  __shared__ float red[kFoldWarps * 16];
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;

  int mi = 0;
  const int row0 = MANY ? B * blockIdx.y : 0;
  for (int64_t item = blockIdx.x; item < p.items; item += gridDim.x) {
    while (mi + 1 < p.count && item >= p.mat[mi + 1].tile0) ++mi;
    const FoldMat& a = p.mat[mi];
    const int64_t j0 = (item - a.tile0) * RT;
    __syncthreads();  // the previous item's readers of the tables are done
    // pair tables: entry q0 | q1 << 2 = (c[q0], c[q1]) for the elements 2k, 2k + 1 of a word
    for (int t = threadIdx.x; t < 2 * RT * 16; t += kFoldThreads) {
      const int plane = t / (RT * 16);
      const int r = (t / 16) % RT;
      const int e = t % 16;
      float2 v = make_float2(0.f, 0.f);
      if (j0 + r < a.m) {
        const float4 c = __ldg(reinterpret_cast<const float4*>(plane ? a.centres_v : a.centres_u) + j0 + r);
        const float cc[4] = {c.x, c.y, c.z, c.w};
        v = make_float2(cc[e & 3], cc[e >> 2]);
      }
      tab[t] = v;
    }
    __syncthreads();

    float2 acc[RT][B];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int b = 0; b < B; ++b) acc[r][b] = make_float2(0.f, 0.f);

    const int64_t nslices = (a.words + 31) / 32;
    for (int64_t s = warp; s < nslices; s += kFoldWarps) {
      const int64_t wi = s * 32 + lane;
      const bool valid = wi < a.words;
      uint32_t cu[RT], cv[RT];
#pragma unroll
      for (int r = 0; r < RT; ++r) {
        const bool ok = valid && j0 + r < a.m;
        cu[r] = ok ? __ldg(a.codes_u + (j0 + r) * a.words + wi) : 0u;
        cv[r] = ok ? __ldg(a.codes_v + (j0 + r) * a.words + wi) : 0u;
      }
      // this lane's 16 inputs of x and xp per batch row (zero past n and past the rows):
      // four 128-bit loads each when the whole word lies inside aligned rows
      float2 xv[B][8], pv[B][8];
      {
        const bool vec = a.vec && 16 * wi + 16 <= a.n;
#pragma unroll
        for (int b = 0; b < B; ++b) {
          const bool live = valid && row0 + b < p.rows;
          const int64_t o0 = (int64_t)(row0 + b) * a.ldx + 16 * wi;
          if (vec && live) {
#pragma unroll
            for (int k = 0; k < 8; k += 2) {
              const float4 u = __ldg(reinterpret_cast<const float4*>(a.x + o0 + 2 * k));
              const float4 w = __ldg(reinterpret_cast<const float4*>(a.xp + o0 + 2 * k));
              xv[b][k] = make_float2(u.x, u.y);
              xv[b][k + 1] = make_float2(u.z, u.w);
              pv[b][k] = make_float2(w.x, w.y);
              pv[b][k + 1] = make_float2(w.z, w.w);
            }
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int64_t i = 16 * wi + 2 * k;
              const bool i0 = live && i < a.n, i1 = live && i + 1 < a.n;
              xv[b][k] = make_float2(i0 ? __ldg(a.x + o0 + 2 * k) : 0.f, i1 ? __ldg(a.x + o0 + 2 * k + 1) : 0.f);
              pv[b][k] = make_float2(i0 ? __ldg(a.xp + o0 + 2 * k) : 0.f, i1 ? __ldg(a.xp + o0 + 2 * k + 1) : 0.f);
            }
          }
        }
      }
#pragma unroll
      for (int r = 0; r < RT; ++r) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float2 tu = tab[r * 16 + ((cu[r] >> (4 * k)) & 15u)];
          const float2 tv = tab[(RT + r) * 16 + ((cv[r] >> (4 * k)) & 15u)];
#pragma unroll
          for (int b = 0; b < B; ++b) {
            acc[r][b] = __ffma2_rn(tu, xv[b][k], acc[r][b]);
            acc[r][b] = __ffma2_rn(tv, pv[b][k], acc[r][b]);
          }
        }
      }
    }

    // lane sums, then a butterfly reduce-scatter: lane l ends with its warp's total of
    // value l % 16 (value index r * B + b)
    float v[K];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int b = 0; b < B; ++b) v[r * B + b] = __fadd_rn(acc[r][b].x, acc[r][b].y);
#pragma unroll
    for (int k = K / 2; k >= 1; k >>= 1) {
#pragma unroll
      for (int i = 0; i < k; ++i) {
        const bool hi = (lane & k) != 0;
        const float send = hi ? v[i] : v[i + k];
        const float keep = hi ? v[i + k] : v[i];
        v[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, k));
      }
    }
    v[0] = __fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], 16));
    if (lane < K) red[warp * 16 + lane] = v[0];
    __syncthreads();
    if (threadIdx.x < K) {
      float t = red[threadIdx.x];
#pragma unroll
      for (int w = 1; w < kFoldWarps; ++w) t = __fadd_rn(t, red[w * 16 + threadIdx.x]);
      const int r = threadIdx.x / B, b = threadIdx.x % B;
      if (j0 + r < a.m && row0 + b < p.rows) a.y[(int64_t)(row0 + b) * a.ldy + j0 + r] = t;
    }
  }
  grid_dependency_wait();  // no dependency: nothing to wait for
}

// beside: the launch ahead on the stream is the tensor-core kernel of the call's other matrices;
// this one needs nothing of it and runs beside it, and ends after it (the kernel's last wait).
template <int B, bool MANY>
cudaError_t launch_fold(const FoldParams& p, bool beside, cudaStream_t s) {
  int dev = 0, sms = 0, per = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fold_kernel<B, MANY>, kFoldThreads, 0)) != cudaSuccess)
    return e;
  if (per < 1) return cudaErrorInvalidConfiguration;
  const int64_t grid = p.items < (int64_t)per * sms ? p.items : (int64_t)per * sms;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, (unsigned)((p.rows + B - 1) / B));
  cfg.blockDim = dim3(kFoldThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = beside ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fold_kernel<B, MANY>, p);
}

bool aligned(const void* ptr, size_t a) { return reinterpret_cast<uintptr_t>(ptr) % a == 0; }

}  // namespace
}  // namespace kd

namespace kd {
namespace {

kd_status check_fold(const kd_fold_mat& a, int64_t batch) {
  if (a.n <= 0 || a.m < 0 || a.ldx < a.n || a.ldy < a.m) return KD_ERR_INVALID_ARG;
  if (a.m == 0 || batch == 0) return KD_OK;
  if (!a.codes_u || !a.codes_v || !a.centres_u || !a.centres_v || !a.x || !a.xp || !a.y) return KD_ERR_INVALID_ARG;
  if (!aligned(a.centres_u, 16) || !aligned(a.centres_v, 16) || !aligned(a.codes_u, 4) ||
      !aligned(a.codes_v, 4) || !aligned(a.x, 4) || !aligned(a.xp, 4) || !aligned(a.y, 4))
    return KD_ERR_INVALID_ARG;
  return KD_OK;
}

}  // namespace
}  // namespace kd

namespace kd {
namespace {

template <int B>
kd_status fold_run(const kd_fold_mat* mats, int count, int64_t batch, bool beside, cudaStream_t s) {
  constexpr int RT = FoldTile<B>::RT;
  FoldParams p;
  p.count = 0;
  p.rows = (int)batch;
  p.items = 0;
  for (int i = 0; i < count; ++i) {
    const kd_fold_mat& a = mats[i];
    if (a.m == 0) continue;
    FoldMat& f = p.mat[p.count++];
    f.codes_u = a.codes_u;
    f.codes_v = a.codes_v;
    f.centres_u = a.centres_u;
    f.centres_v = a.centres_v;
    f.x = a.x;
    f.xp = a.xp;
    f.y = a.y;
    f.n = a.n;
    f.m = a.m;
    f.words = (a.n + 15) / 16;
    f.ldx = a.ldx;
    f.ldy = a.ldy;
    f.tile0 = p.items;
    f.vec = aligned(f.x, 16) && aligned(f.xp, 16) && (a.ldx % 4 == 0 || batch == 1);
    p.items += (a.m + RT - 1) / RT;
  }
  if (p.items == 0) return KD_OK;
  const cudaError_t e = batch > B ? launch_fold<B, (B > 1)>(p, beside, s) : launch_fold<B, false>(p, beside, s);
  return e == cudaSuccess ? KD_OK : KD_ERR_CUDA;
}

}  // namespace
}  // namespace kd

namespace kd {
namespace {

// Whether a matrix takes the lookup kernel.  It re-reads the codes for every two rows but has
// a short chain per item; the tensor-core kernel has the same time up to 16 rows and up to about
// 9000 channels, 11 us at n = 256, 13 at 768, 17 at 2048, 23 at 4096, 44 at 11008 (nearly twice
// that with centres that are not symmetric).  Measured, lookup against tensor cores (us):
//   one row     always (7B layer 88)
//   two rows    4096 x 300 11 / 23, 4096 x 4096 19 / 23, 4096 x 11008 35 / 43, 7B layer 125 / 119
//               (125 / 217 not symmetric), 768 x 768 10 / 13; short vectors of many channels the
//               other way: 768 x 4096 15 / 13, 256 x 11008 26 / 17
//   3, 4 rows   4096 x 300 9 / 23, 4096 x 1024 13 / 23, 4096 x 2048 18 / 23, 11008 x 1024 21 / 44
//   8, 16 rows  4096 x 300 11 / 23, 12 / 24; 4096 x 1024 18 / 23, 27 / 23; 16384 x 300 18 / 59
// Alone, three rows and more would gain up to 4096 channel pairs of rows and from n = 1024 on
// (3072 x 768 at 4 rows 13 / 19), but mostly a layer is one call, where the tensor cores take such
// a matrix beside the others for less: 4096 x 1024 twice and 4096 x 4096 twice at 8 rows 55 us
// with the small ones looked up, 42 without; a layer with the former at 4 rows 138 and 128.  So
// only up to 1024, and from n = 4096 on.  By the matrix and the batch alone, so that a matrix gives the same bits alone and
// in a batched call.
bool by_lookup(const kd_fold_mat& a, int64_t batch) {
  if (batch == 1) return true;
  if (batch == 2) return a.n >= 1024 || a.m <= 3072;
  return batch <= 16 && a.n >= 4096 && a.m <= 1024 && a.m * ((batch + 1) / 2) <= 1024;
}

}  // namespace
}  // namespace kd

extern "C" kd_status kd_matmul_2bit_batch(const kd_fold_mat* mats, int count, int64_t batch, void* stream) {
  if (!mats || count < 1 || count > KD_MAX_BATCH || batch < 0) return KD_ERR_INVALID_ARG;
  for (int i = 0; i < count; ++i) {
    const kd_status st = kd::check_fold(mats[i], batch);
    if (st != KD_OK) return st;
  }
  if (batch == 0) return KD_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  kd_fold_mat sorted[KD_MAX_BATCH];
  int few = 0, rest = 0;
  bool tc = false;  // the tensor-core kernel is launched
  for (int i = 0; i < count; ++i)
    if (kd::by_lookup(mats[i], batch)) sorted[few++] = mats[i];
  for (int i = 0; i < count; ++i)
    if (!kd::by_lookup(mats[i], batch)) {
      sorted[few + rest++] = mats[i];
      tc = tc || mats[i].m > 0;
    }
  kd_status st = tc ? kd::fold_tc_run(sorted + few, rest, batch, s) : KD_OK;
  if (st == KD_OK && few)
    st = batch == 1 ? kd::fold_run<1>(sorted, few, batch, tc, s) : kd::fold_run<2>(sorted, few, batch, tc, s);
  return st;
}

extern "C" kd_status kd_matmul_2bit(const uint32_t* codes_u, const uint32_t* codes_v, const float* centres_u,
                                    const float* centres_v, int64_t n, int64_t m, const float* x, const float* xp,
                                    int64_t batch, int64_t ldx, float* y, int64_t ldy, void* stream) {
  const kd_fold_mat a{codes_u, codes_v, centres_u, centres_v, x, xp, y, n, m, ldx, ldy};
  return kd_matmul_2bit_batch(&a, 1, batch, stream);
}
