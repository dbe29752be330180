// The folded 2-bit layer product of App. C for 16-bit activations (fp16 or bf16), on the
// tensor cores:
//
//     y[r][j] = sum_i h(cu_j[code_u(j, i)]) x[r][i] + sum_i h(cv_j[code_v(j, i)]) xp[r][i]
//
// with x, xp in the 16-bit type (xp = X P from kd_apply_p, rounded by the caller), h()
// the rounding of a centre to that type, fp32 accumulation.  Neither plane is expanded
// in memory.  This file holds the mma.sync kernel for few batch rows, the argument checks and
// the entry points; the others take kd_fold16_tc.cu, whose tcgen05 form decodes every code once
// per 256 rows (7B layer: 87 us at 9 rows and 280 us at 512, where 16 rows at a time through
// mma.sync took 100 us and 3.2 ms; at 8 rows and fewer it is the slower one, 83 to 87 against 82 us).
//
// Mapping.  mma.m16n8k16 with M = the batch rows (the upper eight only in the form for more than
// 8 rows), N = 8 output channels, K = 16 inputs: each code becomes its 16-bit centre in registers
// (kd_dec16.cuh) and feeds a B fragment directly.  A work item is a tile of 32 channels (four
// n-tiles) of one matrix and one CTA; its warps split the inputs into groups of 64 (four k-steps)
// round-robin, each loading the next group's code words and inputs while it computes the
// current one, then add their partial tiles in a fixed order (deterministic results).  Items
// are numbered longest vectors first, so the hardware starts the long ones first.  Bound by
// the decode on the ALU pipe (62 % busy at 4 rows, 7B layer).
//
// K order inside a group of 64 inputs.  The product is a sum over inputs, so A and B
// may enumerate them in any common order.  In k-step j the lanes with t = lane % 4
// take inputs 16 t + 4 j + {0, 1} for k-slots 2t, 2t+1 and 16 t + 4 j + {2, 3} for
// k-slots 2t+8, 2t+9.  A lane's A fragments for the whole group are then its 16
// consecutive inputs of row g (g = lane / 4: two 16-byte loads), and
// its B fragments are code word t of the group (inputs 16 t .. 16 t + 15) of its
// channel: byte j of that word holds the four codes of k-step j.
#include <cuda_runtime.h>

#include "kashin.h"
#include "kd_dec16.cuh"
#include "kd_fold16.h"

namespace kd {
namespace {

// Warps of a CTA, which split the inputs: eight (two CTAs per SM), with four the last items
// of a 7B layer ran on a third of the SMs (86 us per layer at 4 rows, 82 with eight).  Short
// vectors of many channels (wide_short) have four: eight would have one or two groups each and
// spend their time around them (50257 x 768 at 8 rows: 31 us, 25 with four).
constexpr int kF16Warps = 8, kF16ShortWarps = 4;
constexpr int kF16Rows = 8;   // batch rows at most, 16 with the upper ones
constexpr int kF16Tile = 32;  // output channels per work item (four n-tiles)
constexpr int kRedStride = kF16Tile + 1;

struct Fold16Mat {
  const uint32_t* codes_u;
  const uint32_t* codes_v;
  const float* centres_u;
  const float* centres_v;
  const unsigned short* x;
  const unsigned short* xp;
  float* y;
  int64_t n, m, words, ldx, ldy;
  int64_t item0;  // first work item of this matrix
  int vec;        // x and xp 16-byte aligned with ldx a multiple of 8: 128-bit input loads
};

struct Fold16Params {
  int count;
  int rows;  // batch rows of the call
  int64_t items;
  DecodeMul mul;
  Fold16Mat mat[KD_MAX_BATCH];
};

// D += A B for one m16n8k16 tile; BF: the 16-bit operands are bf16 instead of fp16
template <bool BF>
__device__ __forceinline__ void mma_16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                       uint32_t b0, uint32_t b1) {
  if constexpr (BF) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  } else {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
  }
}

// A lane's 16 fp16 inputs of one row at i0 .. i0 + 15 as 8 pairs, zero past n or for a
// row outside the batch.
__device__ __forceinline__ void load_row16(uint32_t (&r)[8], const unsigned short* row, int64_t i0, int64_t n,
                                           bool live, bool vec) {
  if (!live) {
#pragma unroll
    for (int k = 0; k < 8; ++k) r[k] = 0u;
  } else if (vec && i0 + 16 <= n) {
    const uint4 a = __ldg(reinterpret_cast<const uint4*>(row + i0));
    const uint4 b = __ldg(reinterpret_cast<const uint4*>(row + i0 + 8));
    r[0] = a.x; r[1] = a.y; r[2] = a.z; r[3] = a.w;
    r[4] = b.x; r[5] = b.y; r[6] = b.z; r[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t i = i0 + 2 * k;
      const uint32_t lo = i < n ? (uint32_t)__ldg(row + i) : 0u;
      const uint32_t hi = i + 1 < n ? (uint32_t)__ldg(row + i + 1) : 0u;
      r[k] = lo | (hi << 16);
    }
  }
}

// HI: 16 batch rows (blockIdx.y counts blocks of them), else up to 8; W: warps per work item
template <bool BF, bool HI, int W>
__global__ void __launch_bounds__(32 * W, W == kF16Warps ? 2 : HI ? 3 : 4)
    fold16_kernel(const __grid_constant__ Fold16Params p) {
  constexpr int kThreads = 32 * W, kRows = HI ? 2 * kF16Rows : kF16Rows;
  __shared__ float red[W][kRows][kRedStride];
  const int row0 = HI ? kRows * blockIdx.y : 0;
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;

  int mi = 0;
  for (int64_t item = blockIdx.x; item < p.items; item += gridDim.x) {
    while (mi + 1 < p.count && item >= p.mat[mi + 1].item0) ++mi;
    const Fold16Mat& a = p.mat[mi];
    const int64_t c0 = (item - a.item0) * kF16Tile;

    // this lane's channel of each n-tile: centres as byte words, code rows
    uint2 cu[4], cv[4];
    const uint32_t* ru[4];
    const uint32_t* rv[4];
    bool live[4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const int64_t j = c0 + 8 * nt + g;
      live[nt] = j < a.m;
      cu[nt] = centre_bytes<BF>(a.centres_u, j, live[nt]);
      cv[nt] = centre_bytes<BF>(a.centres_v, j, live[nt]);
      ru[nt] = a.codes_u + (live[nt] ? j : 0) * a.words;
      rv[nt] = a.codes_v + (live[nt] ? j : 0) * a.words;
    }
    float acc[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[nt][e] = 0.f;

    const bool row_live = row0 + g < p.rows, hi_live = HI && row0 + g + 8 < p.rows;
    const unsigned short* xg = a.x + (int64_t)(row0 + g) * a.ldx;
    const unsigned short* pg = a.xp + (int64_t)(row0 + g) * a.ldx;
    const int64_t groups = (a.words + 3) / 4;
    // software pipeline: the next group's code words and inputs load while this one computes
    uint32_t wu[4], wv[4], ax[8], ap[8], axh[8], aph[8];
    auto fetch = [&](int64_t gi) {
      const int64_t wi = 4 * gi + t;  // this lane's code word of the group
      const int64_t i0 = 64 * gi + 16 * t;
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const bool ok = live[nt] && wi < a.words;
        wu[nt] = ok ? __ldg(ru[nt] + wi) : 0u;
        wv[nt] = ok ? __ldg(rv[nt] + wi) : 0u;
      }
      load_row16(ax, xg, i0, a.n, row_live, a.vec);
      load_row16(ap, pg, i0, a.n, row_live, a.vec);
      load_row16(axh, xg + 8 * a.ldx, i0, a.n, hi_live, a.vec);
      load_row16(aph, pg + 8 * a.ldx, i0, a.n, hi_live, a.vec);
    };
    if (warp < groups) fetch(warp);
    for (int64_t gi = warp; gi < groups; gi += W) {
      uint32_t cwu[4], cwv[4], cax[8], cap[8], caxh[8], caph[8];
#pragma unroll
      for (int k = 0; k < 4; ++k) { cwu[k] = wu[k]; cwv[k] = wv[k]; }
#pragma unroll
      for (int k = 0; k < 8; ++k) { cax[k] = ax[k]; cap[k] = ap[k]; caxh[k] = axh[k]; caph[k] = aph[k]; }
      if (gi + W < groups) fetch(gi + W);
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        // pairs (4 j, 4 j + 1) and (4 j + 2, 4 j + 3) of the word are k-step j's B fragment
        uint4 ul, uh, vl, vh;
        decode_word(cwu[nt], cu[nt], p.mul, ul, uh);
        decode_word(cwv[nt], cv[nt], p.mul, vl, vh);
        const uint32_t bu[8] = {ul.x, ul.y, ul.z, ul.w, uh.x, uh.y, uh.z, uh.w};
        const uint32_t bv[8] = {vl.x, vl.y, vl.z, vl.w, vh.x, vh.y, vh.z, vh.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          mma_16<BF>(acc[nt], cax[2 * j], caxh[2 * j], cax[2 * j + 1], caxh[2 * j + 1], bu[2 * j], bu[2 * j + 1]);
          mma_16<BF>(acc[nt], cap[2 * j], caph[2 * j], cap[2 * j + 1], caph[2 * j + 1], bv[2 * j], bv[2 * j + 1]);
        }
      }
    }

    // partial tiles of the warps, added in warp order
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      red[warp][g][8 * nt + 2 * t] = acc[nt][0];
      red[warp][g][8 * nt + 2 * t + 1] = acc[nt][1];
      if constexpr (HI) {
        red[warp][g + 8][8 * nt + 2 * t] = acc[nt][2];
        red[warp][g + 8][8 * nt + 2 * t + 1] = acc[nt][3];
      }
    }
    __syncthreads();
    for (int o = threadIdx.x; o < kRows * kF16Tile; o += kThreads) {
      const int r = o / kF16Tile, c = o % kF16Tile;
      if (row0 + r < p.rows && c0 + c < a.m) {
        float s = red[0][r][c];
#pragma unroll
        for (int w = 1; w < W; ++w) s = __fadd_rn(s, red[w][r][c]);
        a.y[(int64_t)(row0 + r) * a.ldy + c0 + c] = s;
      }
    }
    __syncthreads();  // red is reused by the next item
  }
}

bool aligned16(const void* ptr, size_t a) { return reinterpret_cast<uintptr_t>(ptr) % a == 0; }

kd_status check_fold16(const kd_fold_mat_f16& a, int64_t batch) {
  if (a.n <= 0 || a.m < 0 || a.ldx < a.n || a.ldy < a.m) return KD_ERR_INVALID_ARG;
  if (a.m == 0 || batch == 0) return KD_OK;
  if (!a.codes_u || !a.codes_v || !a.centres_u || !a.centres_v || !a.x || !a.xp || !a.y) return KD_ERR_INVALID_ARG;
  if (!aligned16(a.centres_u, 16) || !aligned16(a.centres_v, 16) || !aligned16(a.codes_u, 4) ||
      !aligned16(a.codes_v, 4) || !aligned16(a.x, 2) || !aligned16(a.xp, 2) || !aligned16(a.y, 4))
    return KD_ERR_INVALID_ARG;
  return KD_OK;
}

}  // namespace
}  // namespace kd

namespace kd {
namespace {

// Short vectors of many channels (an output head): the tcgen05 kernel spends its time around the
// few MMAs of its tiles.  Measured, this kernel against tcgen05 (us): 256 x 50000 18 / 37 at 9 to
// 16 rows, 31 / 38 at 17 to 32; 768 x 50257 28 / 43 and 50 / 46; 1024 x 50304 34 / 47 and 61 / 50;
// 2048 x 32000 40 / 42; 768 x 8192 11 / 13, 768 x 4096 10.4 / 10.7.  With fewer channels tcgen05
// stays, up to 2 us slower alone, because a layer that also has longer vectors would need two
// launches.  By the matrix and the batch alone, as every choice here, so that a matrix gives the
// same bits alone and in a batched call.
bool wide_short(const kd_fold_mat_f16& a, int64_t batch) {
  return batch <= 16 ? a.n <= 1024 && a.m >= 8192 : batch <= 32 && a.n <= 256 && a.m >= 16384;
}

template <bool HI, int W>
kd_status launch_fold16(const kd_fold_mat_f16* mats, int count, int64_t batch, cudaStream_t s, bool bf) {
  Fold16Params p;
  p.count = 0;
  p.rows = (int)batch;
  p.items = 0;
  for (int i = 0; i < count; ++i) {
    const kd_fold_mat_f16& a = mats[i];
    if (a.m == 0) continue;
    Fold16Mat& f = p.mat[p.count++];
    f.codes_u = a.codes_u;
    f.codes_v = a.codes_v;
    f.centres_u = a.centres_u;
    f.centres_v = a.centres_v;
    f.x = static_cast<const unsigned short*>(a.x);
    f.xp = static_cast<const unsigned short*>(a.xp);
    f.y = a.y;
    f.n = a.n;
    f.m = a.m;
    f.words = (a.n + 15) / 16;
    f.ldx = a.ldx;
    f.ldy = a.ldy;
    f.item0 = p.items;
    f.vec = aligned16(f.x, 16) && aligned16(f.xp, 16) && a.ldx % 8 == 0;
    p.items += (a.m + kF16Tile - 1) / kF16Tile;
  }
  if (p.items == 0) return KD_OK;
  // one CTA per work item (the grid-stride loop covers grids past 2^30 items)
  const int64_t most = (int64_t)1 << 30;
  const dim3 grid((unsigned)(p.items < most ? p.items : most), HI ? (unsigned)((batch + 15) / 16) : 1u);
  if (bf) fold16_kernel<true, HI, W><<<grid, 32 * W, 0, s>>>(p);
  else fold16_kernel<false, HI, W><<<grid, 32 * W, 0, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? KD_OK : KD_ERR_CUDA;
}

kd_status fold16_run(const kd_fold_mat_f16* mats, int count, int64_t batch, void* stream, bool bf) {
  if (!mats || count < 1 || count > KD_MAX_BATCH || batch < 0) return KD_ERR_INVALID_ARG;
  for (int i = 0; i < count; ++i) {
    const kd_status st = check_fold16(mats[i], batch);
    if (st != KD_OK) return st;
  }
  if (batch == 0) return KD_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // the short ones, then the others, each longest vectors first, so that the long items of a
  // layer are not the last ones started
  kd_fold_mat_f16 sorted[KD_MAX_BATCH];
  int few = 0;
  for (int i = 0; i < count; ++i) few += wide_short(mats[i], batch);
  for (int i = 0, at[2] = {0, few}; i < count; ++i) {
    const int side = wide_short(mats[i], batch) ? 0 : 1;
    int k = at[side]++;
    for (; k > (side ? few : 0) && mats[i].n > sorted[k - 1].n; --k) sorted[k] = sorted[k - 1];
    sorted[k] = mats[i];
  }
  kd_status st = KD_OK;
  if (few)
    st = batch > kF16Rows ? launch_fold16<true, kF16ShortWarps>(sorted, few, batch, s, bf)
                          : launch_fold16<false, kF16ShortWarps>(sorted, few, batch, s, bf);
  if (st == KD_OK && few < count)
    st = batch > kF16Rows ? fold16_tc_run(sorted + few, count - few, batch, s, bf)
                          : launch_fold16<false, kF16Warps>(sorted + few, count - few, batch, s, bf);
  return st;
}

}  // namespace
}  // namespace kd

extern "C" kd_status kd_matmul_2bit_f16_batch(const kd_fold_mat_f16* mats, int count, int64_t batch,
                                              void* stream) {
  return kd::fold16_run(mats, count, batch, stream, false);
}

extern "C" kd_status kd_matmul_2bit_bf16_batch(const kd_fold_mat_f16* mats, int count, int64_t batch,
                                               void* stream) {
  return kd::fold16_run(mats, count, batch, stream, true);
}

extern "C" kd_status kd_matmul_2bit_f16(const uint32_t* codes_u, const uint32_t* codes_v, const float* centres_u,
                                        const float* centres_v, int64_t n, int64_t m, const void* x,
                                        const void* xp, int64_t batch, int64_t ldx, float* y, int64_t ldy,
                                        void* stream) {
  const kd_fold_mat_f16 a{codes_u, codes_v, centres_u, centres_v, x, xp, y, n, m, ldx, ldy};
  return kd_matmul_2bit_f16_batch(&a, 1, batch, stream);
}

extern "C" kd_status kd_matmul_2bit_bf16(const uint32_t* codes_u, const uint32_t* codes_v, const float* centres_u,
                                         const float* centres_v, int64_t n, int64_t m, const void* x,
                                         const void* xp, int64_t batch, int64_t ldx, float* y, int64_t ldy,
                                         void* stream) {
  const kd_fold_mat_f16 a{codes_u, codes_v, centres_u, centres_v, x, xp, y, n, m, ldx, ldy};
  return kd_matmul_2bit_bf16_batch(&a, 1, batch, stream);
}
