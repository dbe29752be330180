// The folded 2-bit layer product of App. C in fp32 (kd_fold.cu states it, and which calls come
// here) on the tensor cores, with exact sums of the inputs.
//
//  * An input is a fixed-point number on the grid of its row (of this CTA's part of it): with
//    2^k the power of two above the row's largest magnitude, x = 2^k (d1 + d2 + d3 + d4), where
//    d1, d2, d3 are the digits of weight 2^-7, 2^-15, 2^-23 (at most 128 of each, exact in bf16)
//    and d4, below 2^-24, is cut to bf16: 32 bits below the row's largest.
//  * A weight enters as which code it has, not as its centre: with T_q the sum of the inputs
//    whose code is q, the product of one plane is c0 T0 + c1 T1 + c2 T2 + c3 T3.  The MMAs
//    multiply the inputs by planes of -1, 0 and 1, which are exact in bf16:
//        D_in = T2 - T1, D_out = T3 - T0, and where a channel of the tile has centres that are
//        not symmetric about 0 (after k-means refinement), E_in = T1 + T2, E_out = T0 + T3.
//    A pair of centres far from symmetric takes T2 and T1 (T3 and T0) themselves instead: with
//    D and E a centre's sum would come out of differences as large as the other centre's.
//    The centres stay fp32 and multiply the sums.
// The sums of d1, d2 and d3 are whole numbers of at most 24 bits for up to 2^17 inputs, so the
// tensor core, which cuts each addition off instead of rounding it, adds them exactly; kChunk
// bounds an accumulation.  Pieces taken from the floating-point bits of each input instead
// (8 + 8 + 8) lost up to 2^-24 of the running sum per addition: a row led by one input erred by
// 4.7e-6 of its norm, log-normal inputs by 2.3e-6, and inputs below 2^-110 lost their last bits.
//
// Mapping.  tcgen05.mma with M = 128 output channels, N = 4 digits per batch row (16 rows per
// block), K = the inputs in stages of 64.  A cluster owns a tile of 128 channels: half of its
// CTAs the u plane with x, half the v plane with xp, each a part of the inputs (two parts up to
// 16 rows, one beyond); their sums are added at the end over distributed shared memory.  In a
// CTA
//  * two groups of four warps decode, every other stage each: a thread turns the four code
//    words of its channel into its TMEM lane of either plane (the MMA takes A from TMEM:
//    through shared memory, the planes' writes and reads filled its bandwidth and 16 rows of
//    the 7B layer took 190 us);
//  * the rows' largest magnitudes come from a small launch ahead (row_grid_kernel); where an
//    infinity or a NaN is among a row, all warps first look through the tile's rows for them;
//  * two groups of two warps split the inputs into the B tile in shared memory, every other
//    stage each, their loads two own stages ahead (again from L2; packed additions, so that
//    the decode has the ALU pipe);
//  * one thread issues the MMAs;
//  * the decoding warps also move finished sums from TMEM to registers.
// With centres that are not symmetric the K loop runs twice, over the D and then the E planes.
// TMEM (256 of 512 columns, two CTAs per SM): the sums of two planes, and one slot of A for
// each decoding group; while one CTA waits for its slot or its sums, the other decodes.
//
// An infinity among the inputs counts as zero there and is added with its centre at the end;
// a NaN makes its row NaN.  Channels with a centre of 2^101 and more, an infinity or a NaN
// among them (their products with a plain sum could overflow), and rows of more infinities
// than are noted, are summed again by plain fp32 FMAs.
//
// Measured (7B layer, L2 cold): 119 us at 3 rows, 137 at 16, 454 at 64 (218 and 250 at 3 and 16
// with centres that are not symmetric); the table-lookup kernel takes 125 us per two rows (981
// at 16).  The ALU pipe is 64 % busy, mostly with the decode.  Error against 64 bits, 2-norm: 5e-8 to 6e-8 (8e-8
// with centres that are not symmetric) for normal, all-positive, log-normal and very small inputs
// and rows led by one, n = 256 to 16384; the table-lookup kernel has 9e-8 to 2.9e-7.
#include <cuda_runtime.h>

#include "kashin.h"
#include "kd_dec16.cuh"
#include "kd_fold_tc.h"
#include "kd_tc.cuh"
#include "kd_tc_host.h"

namespace kd {
namespace {

constexpr int kTile = 128;     // output channels per CTA (the MMA's M, the TMEM lanes)
constexpr int kRows = 16;      // batch rows per block
constexpr int kStageK = 64;    // inputs per stage
constexpr int kDigits = 4;     // bf16 digits per input
constexpr int kChunk = 1024;   // stages per TMEM accumulation (2^16 inputs)
constexpr int kDecWarps = 8;   // decoding warps: two groups of four
constexpr int kSplitWarps = 4;  // two groups of two
constexpr int kThreads = 32 * (kDecWarps + kSplitWarps + 1);
constexpr int kSlotsA = 2, kSlotsB = 4;    // A in TMEM, B in shared memory
constexpr int kBBytes = kDigits * kRows * 128;
constexpr uint32_t kCols = 256;            // TMEM: sums of plane p at 64 p, A slot s at 128 + 64 s (32 per plane)
constexpr int kSmem = tc_smem_floor(kCols);
static_assert(kSlotsB * kBBytes + 1024 <= kSmem, "the B slots fit");
constexpr uint32_t kBig = 0x72000000u;     // bits of 2^101
constexpr uint32_t kInf = 0x7F800000u;
constexpr int kTopExp = 100;               // the sums take at most 2^100 of the row's 2^k before the centres
constexpr int kInfs = 64;                  // infinities noted per CTA
constexpr int kGridThreads = 256;          // of row_grid_kernel
constexpr int kScan = 8;                   // loads in flight per thread of the search for the rows' largest

struct FoldTcMat {
  const uint32_t* codes[2];
  const float* centres[2];
  const float* x[2];
  float* y;
  int64_t n, m, words, ldx, ldy;
  int vec_codes;  // code rows 16-byte aligned
  int vec_x;      // input rows of whole 16-byte blocks
};

struct FoldTcParams {
  uint32_t tile0[KD_MAX_BATCH];  // first channel tile of each matrix
  int count;
  int rows;        // batch rows of the call
  int row_blocks;  // blocks of kRows rows
  int split;       // parts of each plane's inputs, one CTA each
  DecodeMul mul;
  FoldTcMat mat[KD_MAX_BATCH];
};

struct Ctl {
  uint64_t full_a[kSlotsA], empty_a[kSlotsA], full_b[kSlotsB], empty_b[kSlotsB], acc_full, acc_empty, drained;
  uint32_t tmem;
  int fail;   // a wait expired: the tile's outputs become NaN
  uint32_t row_max[kRows];  // bits of the largest finite magnitude
  uint32_t nan_rows, inf_rows;  // batch rows with a NaN, with an infinity (bits)
  uint32_t infs;
  int scan;  // a row of this block has an infinity or a NaN
  int inf_row[kInfs], inf_at[kInfs];
};

__device__ __forceinline__ uint32_t mag(float f) { return __float_as_uint(f) & 0x7FFFFFFFu; }

// The grid of a row whose largest magnitude has these bits: 2^k above it, k >= -126 (below, the
// inputs are multiples of 2^-149, which the grid holds).
__device__ __forceinline__ int grid_exp(uint32_t max_bits) { return (int)(max_bits >> 23) - 126; }
__device__ __forceinline__ float exp2_bits(int e) {  // 2^e, -149 <= e <= 127
  return __uint_as_float(e >= -126 ? (uint32_t)(e + 127) << 23 : 1u << (e + 149));
}

__device__ __forceinline__ bool ctl_wait(Ctl& c, uint64_t* bar, uint32_t parity) { return tc_wait(bar, parity, &c.fail); }

// Whether a pair of centres (low, high) is far from symmetric: each of its sums has its own
// plane then.  Below this line the factors of D and E are within 1.67 of each other's centre.
__device__ __forceinline__ bool far(float low, float high) {
  return !(fabsf(__fadd_rn(low, high)) <= __fmul_rn(0.25f, __fsub_rn(high, low)));
}

// code -> bf16 as (low bytes, high bytes) of codes 0..3: the inner or the outer pair's plane of
// the first or the second pass
__device__ __forceinline__ uint2 plane_bytes(bool outer, bool second, bool own) {
  const uint2 d = outer ? make_uint2(0x80000080u, 0x3F0000BFu)   // D_out: -1 0  0  1
                        : make_uint2(0x00808000u, 0x003FBF00u);  // D_in:   0 -1 1  0
  if (!own) return make_uint2(d.x, second ? d.y & 0x3F3F3F3Fu : d.y);  // E: the signs off
  const uint32_t keep = outer ? (second ? 0x000000FFu : 0xFF000000u) : (second ? 0x0000FF00u : 0x00FF0000u);
  return make_uint2(d.x & keep, d.y & keep & 0x3F3F3F3Fu);
}

// inputs [n0, n0 + n) of a part of a matrix of length len
struct Part {
  int s0, stages;
  __device__ Part(int64_t len, uint32_t part, uint32_t split) {
    const uint32_t all = (uint32_t)((len + kStageK - 1) / kStageK);
    s0 = (int)(all * part / split);
    stages = (int)(all * (part + 1) / split) - s0;
  }
  __device__ int64_t n0() const { return (int64_t)kStageK * s0; }
  __device__ int n(int64_t len) const {
    return (int)(len - n0() < (int64_t)kStageK * stages ? len - n0() : (int64_t)kStageK * stages);
  }
};

// The biased exponent of the largest magnitude of each row, plane and part (255: an infinity or
// a NaN is among them), into byte 2 plane + part of the first output of every channel tile:
// the tile's own CTAs read it before they write that output.  One CTA per row, plane and part.
// With every tile taking the maxima of the same rows itself, 16 rows of the 7B layer took
// 178 us (140 with this launch, which overlaps the tiles' set-up; 2 rows 126, now 121).
__global__ void __launch_bounds__(kGridThreads) row_grid_kernel(const __grid_constant__ FoldTcParams p) {
  __shared__ uint32_t wmax[kGridThreads / 32];
  grid_dependents_start();  // the tiles' kernel sets itself up and waits for this one's end
  const uint32_t split = (uint32_t)p.split, per = 2 * split * (uint32_t)p.rows;
  const FoldTcMat& a = p.mat[blockIdx.x / per];
  const uint32_t id = blockIdx.x % per;
  const int64_t row = id / (2 * split);
  const uint32_t pl = id / split % 2, part = id % split;
  const Part range(a.n, part, split);
  const int n = range.n(a.n);
  const float* q = a.x[pl] + row * a.ldx + range.n0();
  uint32_t m = 0u;
  if (a.vec_x) {
#pragma unroll 4
    for (int i = 4 * threadIdx.x; i < n; i += 4 * kGridThreads) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(q + i));
      m = max(m, max(max(mag(f.x), mag(f.y)), max(mag(f.z), mag(f.w))));
    }
  } else {
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kGridThreads) m = max(m, mag(__ldg(q + i)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kGridThreads / 32; ++w) m = max(m, wmax[w]);
  for (int64_t c = (int64_t)threadIdx.x * kTile; c < a.m; c += kGridThreads * kTile)
    reinterpret_cast<uint8_t*>(a.y + row * a.ldy + c)[2 * pl + part] = (uint8_t)(m >> 23);
}

__global__ void __launch_bounds__(kThreads, 2) fold_tc_kernel(const __grid_constant__ FoldTcParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ Ctl ctl;
  grid_dependents_start();  // the lookup kernel of the call's other matrices may run beside this one
  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;  // the B slots
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const int lane = threadIdx.x & 31;

  const uint32_t rank = cluster_rank(), split = (uint32_t)p.split;
  const uint32_t pl = rank >= split;  // 0: u plane and x, 1: v plane and xp
  const uint32_t part = rank - pl * split;
  const uint32_t id = blockIdx.x / (2 * split);
  const uint32_t tile = id / (uint32_t)p.row_blocks;
  const int row0 = (int)(id - tile * p.row_blocks) * kRows;
  int mi = 0;
  while (mi + 1 < p.count && tile >= p.tile0[mi + 1]) ++mi;
  const FoldTcMat& a = p.mat[mi];
  const int64_t c0 = (int64_t)(tile - p.tile0[mi]) * kTile;
  const int rows = p.rows - row0 < kRows ? p.rows - row0 : kRows;
  const int nt = (kDigits * rows + 15) / 16 * 16;
  // this CTA's part of the inputs: n inputs from n0, in L stages (none where n < 64 split)
  const Part range(a.n, part, split);
  const int s0 = range.s0, L = range.stages, n = range.n(a.n);
  const int64_t n0 = range.n0();

  // decoding threads: channel r of the tile, its centres, its first code words
  const int grp = warp >> 2;
  const int r = threadIdx.x & (kTile - 1);
  const bool live = warp < kDecWarps && c0 + r < a.m;
  const uint32_t* code_row = a.codes[pl] + (live ? c0 + r : 0) * a.words + 4 * s0;
  const int words = live ? (n + 15) / 16 : 0;
  const bool vec = a.vec_codes;
  auto fetch = [&](int st) -> uint4 {  // the words of stage st (of either pass), zero past the part and m
    const int s = st < L ? st : st - L;
    const int w0 = 4 * s;
    const int left = words - w0;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    if (vec) {
      if (left > 0) w = __ldg(reinterpret_cast<const uint4*>(code_row + w0));
    } else {
      if (left > 0) w.x = __ldg(code_row + w0);
      if (left > 1) w.y = __ldg(code_row + w0 + 1);
      if (left > 2) w.z = __ldg(code_row + w0 + 2);
      if (left > 3) w.w = __ldg(code_row + w0 + 3);
    }
    return w;
  };
  uint4 w0 = fetch(grp), w1 = fetch(grp + 2), w2 = fetch(grp + 4);
  float4 cen = make_float4(0.f, 0.f, 0.f, 0.f);
  if (live) cen = __ldg(reinterpret_cast<const float4*>(a.centres[pl]) + c0 + r);
  const bool plain_channel = max(max(mag(cen.x), mag(cen.y)), max(mag(cen.z), mag(cen.w))) >= kBig;

  if (warp == kDecWarps + kSplitWarps) {
    if (lane < kSlotsA) {
      mbar_init(&ctl.full_a[lane], 4);  // the warps of a decoding group
      mbar_init(&ctl.empty_a[lane], 1);
    }
    if (lane < kSlotsB) {
      mbar_init(&ctl.full_b[lane], kSplitWarps / 2);
      mbar_init(&ctl.empty_b[lane], 1);
    }
    if (lane == 0) {
      mbar_init(&ctl.acc_full, 1);
      mbar_init(&ctl.drained, 1);
      mbar_init(&ctl.acc_empty, kDecWarps);
      ctl.fail = 0;
      ctl.nan_rows = ctl.inf_rows = ctl.infs = 0u;
    }
    // the exponents that row_grid_kernel left in the first word of the tile's output rows
    uint32_t e = 0u;
    grid_dependency_wait();
    if (lane < rows)
      e = reinterpret_cast<const volatile uint8_t*>(a.y + (int64_t)(row0 + lane) * a.ldy + c0)[2 * pl + part];
    const bool scan = __any_sync(0xffffffffu, e == 255u);
    if (lane < kRows) ctl.row_max[lane] = scan ? 0u : e << 23;
    if (lane == 0) ctl.scan = scan;
    mbar_init_fence();
    tmem_alloc(&ctl.tmem, kCols);
  }
  __syncthreads();
  // ---- rows with an infinity or a NaN: note them and take the others' largest magnitude
  // (128 inputs of a row per warp and load) ----
  if (ctl.scan) {
    const float* x0 = a.x[pl] + (int64_t)row0 * a.ldx + n0;
    const int blocks = (n + 127) / 128, tasks = rows * blocks;
    const bool vec_x = a.vec_x;
    constexpr int kStep = kThreads / 32;
    const int drow = blocks ? kStep / blocks : 0, dblk = blocks ? kStep % blocks : 0;
    int row = blocks ? warp / blocks : 0, blk = blocks ? warp % blocks : 0;
    auto next = [&](int& r, int& b) {
      r += drow;
      b += dblk;
      if (b >= blocks) {
        b -= blocks;
        ++r;
      }
    };
    for (int t0 = warp; t0 < tasks; t0 += kScan * kStep) {
      float4 f[kScan];
      int lr = row, lb = blk;
#pragma unroll
      for (int k = 0; k < kScan; ++k) {
        const int i = 128 * lb + 4 * lane;
        const float* q = x0 + (int64_t)lr * a.ldx + i;
        f[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lr < rows && i < n) {
          if (vec_x) {
            f[k] = __ldg(reinterpret_cast<const float4*>(q));
          } else {
            f[k].x = __ldg(q);
            if (i + 1 < n) f[k].y = __ldg(q + 1);
            if (i + 2 < n) f[k].z = __ldg(q + 2);
            if (i + 3 < n) f[k].w = __ldg(q + 3);
          }
        }
        next(lr, lb);
      }
#pragma unroll
      for (int k = 0; k < kScan; ++k) {
        if (row >= rows) break;
        uint32_t m = max(max(mag(f[k].x), mag(f[k].y)), max(mag(f[k].z), mag(f[k].w)));
        if (__any_sync(0xffffffffu, m >= kInf)) {
          const float v[4] = {f[k].x, f[k].y, f[k].z, f[k].w};
          m = 0u;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t b = mag(v[e]);
            if (b > kInf) {
              atomicOr(&ctl.nan_rows, 1u << row);
            } else if (b == kInf) {
              atomicOr(&ctl.inf_rows, 1u << row);
              const uint32_t at = atomicAdd(&ctl.infs, 1u);
              if (at < (uint32_t)kInfs) {
                ctl.inf_row[at] = row;
                ctl.inf_at[at] = 128 * blk + 4 * lane + e;
              }
            } else {
              m = max(m, b);
            }
          }
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) atomicMax(&ctl.row_max[row], m);
        next(row, blk);
      }
    }
  }
  tc_fence_before();
  // centres symmetric about 0 in the whole tile: two planes suffice
  const int reps = __syncthreads_or(!(cen.x == -cen.w && cen.y == -cen.z)) ? 2 : 1;
  tc_fence_after();
  const uint32_t tmem = ctl.tmem;
  const bool own_in = far(cen.y, cen.z), own_out = far(cen.x, cen.w);
  const int V = L * reps;  // stages of all passes
  // accumulations of one pass: kChunk stages each but the last
  const int chunks = (L + kChunk - 1) / kChunk;

  float acc[8];  // batch rows 8 grp .. + 7 of this channel
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.f;
  if (warp == kDecWarps + kSplitWarps) {
    // ---- MMAs ----
    if (elect_one()) {
      const uint32_t idesc = tc_idesc(true, nt);
      const uint64_t db0 = tc_desc(ring);
      int in_pass = 0, in_chunk = 0, chunk = 0;
      for (int i = 0; i < V; ++i) {
        const int sa = i % kSlotsA, sb = i % kSlotsB;
        if ((in_chunk == 0 && chunk > 0 && !ctl_wait(ctl, &ctl.acc_empty, (chunk - 1) & 1)) ||
            !ctl_wait(ctl, &ctl.full_b[sb], (i / kSlotsB) & 1) || !ctl_wait(ctl, &ctl.full_a[sa], (i / kSlotsA) & 1))
          break;
        tc_fence_after();
        const bool end = in_chunk == kChunk - 1 || in_pass == L - 1;
        const uint32_t ta = tmem + 128 + 64 * sa;
        const uint64_t db = db0 + (uint64_t)(sb * (kBBytes >> 4));
#pragma unroll
        for (int pn = 0; pn < 2; ++pn)
#pragma unroll
          for (int q = 0; q < kStageK / 16; ++q)
            tc_mma(tmem + pn * 64, ta + pn * 32 + 8 * q, db + 2 * q, idesc, in_chunk != 0 || q != 0);
        tc_commit(&ctl.empty_a[sa]);
        tc_commit(&ctl.empty_b[sb]);
        if (end) tc_commit(&ctl.acc_full);
        ++in_chunk;
        ++in_pass;
        if (end) {
          in_chunk = 0;
          ++chunk;
          if (in_pass == L) in_pass = 0;
        }
      }
      tc_drain(&ctl.drained, &ctl.fail);
    }
    __syncwarp();
  } else if (warp >= kDecWarps) {
    // ---- B tiles: thread (row t / 8 + 8 h, inputs 8 (t % 8) .. + 7), h = 0, 1 ----
    const int sg = (warp - kDecWarps) >> 1;
    const int t = threadIdx.x & 63;
    const int seg = t & 7, br0 = t >> 3;
    const float* src = a.x[pl] + (int64_t)(row0 + br0) * a.ldx + n0 + 8 * seg;
    const bool vec_x = a.vec_x;
    float scale[2];  // 2^-k of the thread's rows
    bool clean[2];   // all finite
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      scale[h] = exp2_bits(-grid_exp(ctl.row_max[br0 + 8 * h]));
      clean[h] = (((ctl.nan_rows | ctl.inf_rows) >> (br0 + 8 * h)) & 1u) == 0u;
    }
    auto load = [&](int st, float (&v)[2][8]) {
      const int i0 = kStageK * (st < L ? st : st - L);
      const int left = n - i0 - 8 * seg;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float* q = src + 8 * h * a.ldx + i0;
        const bool in = st < V && br0 + 8 * h < rows;
        if (vec_x) {
          float4 f0 = make_float4(0.f, 0.f, 0.f, 0.f), f1 = f0;
          if (in && left >= 4) f0 = __ldg(reinterpret_cast<const float4*>(q));
          if (in && left >= 8) f1 = __ldg(reinterpret_cast<const float4*>(q) + 1);
          v[h][0] = f0.x; v[h][1] = f0.y; v[h][2] = f0.z; v[h][3] = f0.w;
          v[h][4] = f1.x; v[h][5] = f1.y; v[h][6] = f1.z; v[h][7] = f1.w;
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) v[h][e] = in && e < left ? __ldg(q + e) : 0.f;
        }
      }
    };
    auto put = [&](int s, const float (&v)[2][8]) {
      const int sb = s % kSlotsB;
      if (s >= kSlotsB) ctl_wait(ctl, &ctl.empty_b[sb], (s / kSlotsB - 1) & 1);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int br = br0 + 8 * h;
        if (br < rows) {
          uint32_t pk[kDigits][4];
          const float2 sc = make_float2(scale[h], scale[h]);
          auto digit = [](float2 t, float to) {  // nearest multiple of to's last place
            return __fadd2_rn(__fadd2_rn(t, make_float2(to, to)), make_float2(-to, -to));
          };
          auto less = [](float2 t, float2 d) { return __fadd2_rn(t, make_float2(-d.x, -d.y)); };
          auto pack = [](float2 d) { return prmt(__float_as_uint(d.x), __float_as_uint(d.y), 0x7632u); };
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            // K order inside 8 inputs as the decoded codes': 0, 4, 1, 5, 2, 6, 3, 7
            float2 x = make_float2(v[h][e], v[h][e + 4]);
            if (!clean[h]) {
              if (mag(x.x) >= kInf) x.x = 0.f;
              if (mag(x.y) >= kInf) x.y = 0.f;
            }
            const float2 t = __fmul2_rn(x, sc);
            const float2 d1 = digit(t, 0x1.8p16f), t1 = less(t, d1);
            const float2 d2 = digit(t1, 0x1.8p8f), t2 = less(t1, d2);
            const float2 d3 = digit(t2, 0x1.8p0f), t3 = less(t2, d3);
            pk[0][e] = pack(d1);
            pk[1][e] = pack(d2);
            pk[2][e] = pack(d3);
            pk[3][e] = pack(t3);
          }
#pragma unroll
          for (int q = 0; q < kDigits; ++q) {
            const uint32_t row = kDigits * br + q;
            sts128(ring + sb * kBBytes + row * 128 + ((seg ^ (row & 7)) << 4),
                   make_uint4(pk[q][0], pk[q][1], pk[q][2], pk[q][3]));
          }
        }
      }
      fence_proxy_async_smem();  // the tile's writes before the MMA's reads
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.full_b[sb]);
    };
    float va[2][8], vb[2][8];
    load(sg, va);
    load(sg + 2, vb);
#pragma unroll 1
    for (int s = sg; s < V; s += 4) {
      put(s, va);
      load(s + 4, va);
      if (s + 2 < V) put(s + 2, vb);
      load(s + 6, vb);
    }
  } else {
    // ---- decode, and the fp32 sums ----
    const uint32_t lanes = tmem + ((uint32_t)(warp & 3) << 21);  // this warp's 32 TMEM lanes
    int done = 0, done_stage = 0;  // chunks added so far, the stage that ends the next one
    auto next_end = [&]() {
      const int pass = done / chunks, c = done - pass * chunks;
      done_stage = pass * L + (c + 1 < chunks ? (c + 1) * kChunk : L);
    };
    if (chunks > 0) next_end();
    auto promote = [&]() {
      ctl_wait(ctl, &ctl.acc_full, done & 1);
      tc_fence_after();
      // factors of the inner and the outer plane: c2, c3 where the centres are symmetric,
      // else half of c2 - c1, c3 - c0 for D and of c2 + c1, c3 + c0 for E, or the centres
      float fi = cen.z, fo = cen.w;
      if (reps == 2) {
        const bool e = done >= chunks;
        fi = own_in ? (e ? cen.y : cen.z) : __fmul_rn(0.5f, __fadd_rn(cen.z, e ? cen.y : -cen.y));
        fo = own_out ? (e ? cen.x : cen.w) : __fmul_rn(0.5f, __fadd_rn(cen.w, e ? cen.x : -cen.x));
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {  // four batch rows
        if (8 * grp + 4 * half < rows) {
          float d[2][16];
#pragma unroll
          for (int pn = 0; pn < 2; ++pn)
#pragma unroll
            for (int q = 0; q < 16; q += 8) tmem_ld8(&d[pn][q], lanes + pn * 64 + 32 * grp + 16 * half + q);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            // the digits, the smallest first, then the row's 2^k (the rest beyond 2^100 at the end)
            const float s2k = exp2_bits(min(grid_exp(ctl.row_max[8 * grp + 4 * half + k]), kTopExp));
            float sum[2];
#pragma unroll
            for (int pn = 0; pn < 2; ++pn)
              sum[pn] = __fmul_rn(__fadd_rn(__fadd_rn(__fadd_rn(d[pn][4 * k + 3], d[pn][4 * k + 2]), d[pn][4 * k + 1]), d[pn][4 * k]), s2k);
            acc[4 * half + k] = __fadd_rn(acc[4 * half + k], __fmaf_rn(fo, sum[1], __fmul_rn(fi, sum[0])));
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.acc_empty);
      ++done;
      next_end();
    };
    // own stages grp, grp + 2, ..., their code words loaded three own stages ahead
    uint2 b0 = plane_bytes(false, false, own_in), b1 = plane_bytes(true, false, own_out);
#pragma unroll 1
    for (int i = grp; i < V; i += 2) {
      const uint32_t ww[4] = {w0.x, w0.y, w0.z, w0.w};
      w0 = w1;
      w1 = w2;
      w2 = fetch(i + 6);
      if (i >= L && i < L + 2) {  // the first one of the second pass
        b0 = plane_bytes(false, true, own_in);
        b1 = plane_bytes(true, true, own_out);
      }
      if (i >= kSlotsA) ctl_wait(ctl, &ctl.empty_a[grp], (i / kSlotsA - 1) & 1);
      tc_fence_after();  // the MMAs that read the slot are complete
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t sel[8];
        uint4 lo, hi;
        decode_selectors_by4(ww[q], p.mul, sel);
        decode_pick(sel, b0, lo, hi);
        tmem_st8(lanes + 128 + 64 * grp + 8 * q, lo, hi);
        decode_pick(sel, b1, lo, hi);
        tmem_st8(lanes + 160 + 64 * grp + 8 * q, lo, hi);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.full_a[grp]);
      // past the end of an accumulation: its MMAs need nothing more from this warp.  All that
      // ended: a pass may end in an accumulation of one stage, and then the other group's
      // next slot waits for this one's sums
      while (done < chunks * reps && i >= done_stage) promote();
    }
    while (done < chunks * reps) promote();
  }

  __syncthreads();  // the MMAs have completed: shared memory is free
  const float bad = *(volatile int*)&ctl.fail ? __int_as_float(0x7FC00000) : 0.f;
  if (warp < kDecWarps) {
    auto centre = [&](int i) {  // of input i
      const uint32_t code = (__ldg(code_row + (i >> 4)) >> (2 * (i & 15))) & 3u;
      return (code & 2u) ? ((code & 1u) ? cen.w : cen.z) : ((code & 1u) ? cen.y : cen.x);
    };
    const float* q = a.x[pl] + (int64_t)row0 * a.ldx + n0;
    const uint32_t of = (0xFFu << (8 * grp)) & ((1u << rows) - 1u);  // this thread's rows
    const bool many = ctl.infs > (uint32_t)kInfs;
    const uint32_t infs = live && !many ? ctl.infs : 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t row_max = ctl.row_max[8 * grp + k];
      acc[k] = __fmul_rn(acc[k], exp2_bits(max(grid_exp(row_max) - kTopExp, 0)));
    }
    for (uint32_t e = 0; e < infs; ++e) {
      const int row = ctl.inf_row[e], i = ctl.inf_at[e];
      const float add = __fmul_rn(centre(i), __ldg(q + (int64_t)row * a.ldx + i));
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (row == 8 * grp + k) acc[k] = __fadd_rn(acc[k], add);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int c = 8 * grp + k;
      const float nan = (ctl.nan_rows >> c) & 1u ? __int_as_float(0x7FC00000) : bad;
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(ring + (c * kTile + r) * 4), "f"(__fadd_rn(acc[k], nan)) : "memory");
    }
    // plain sums of this channel, a code word and its 16 inputs at a time
    const uint32_t plain = !live ? 0u : of & (plain_channel ? ~0u : many ? ctl.inf_rows : 0u);
    for (uint32_t left = plain; left; left &= left - 1) {
      const int c = __ffs(left) - 1;
      const float* x = q + (int64_t)c * a.ldx;
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      for (int w = 0; w < words; ++w) {
        const uint32_t code = __ldg(code_row + w);
        float f[16];
#pragma unroll
        for (int e = 0; e < 16; e += 4) {
          const int i = 16 * w + e;
          if (a.vec_x && i < n) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(x + i));
            f[e] = v.x; f[e + 1] = v.y; f[e + 2] = v.z; f[e + 3] = v.w;
          } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) f[e + k] = i + k < n ? __ldg(x + i + k) : 0.f;
          }
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float lo = (code >> (2 * e)) & 1u ? cen.y : cen.x, hi = (code >> (2 * e)) & 1u ? cen.w : cen.z;
          if (16 * w + e < n) sum[e & 3] = __fmaf_rn((code >> (2 * e)) & 2u ? hi : lo, f[e], sum[e & 3]);
        }
      }
      const float all = __fadd_rn(__fadd_rn(sum[0], sum[1]), __fadd_rn(sum[2], sum[3]));
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(ring + (c * kTile + r) * 4), "f"(__fadd_rn(all, bad)) : "memory");
    }
  }
  cluster_sync_all();
  // the CTAs share the batch rows; parts in order, the u plane's first
  if (live) {
    for (int c = 2 * (int)rank + grp; c < rows; c += 4 * (int)split) {
      const uint32_t at = ring + (c * kTile + r) * 4;
      float v = ld_dsmem(at, 0);
      for (uint32_t q = 1; q < 2 * split; ++q) v = __fadd_rn(v, ld_dsmem(at, q));
      a.y[(int64_t)(row0 + c) * a.ldy + c0 + r] = v;
    }
  }
  cluster_sync_all();  // the peer's reads of this CTA's shared memory are done
  if (warp == kDecWarps + kSplitWarps) tmem_dealloc(tmem, kCols);
}

bool aligned_to(const void* ptr, size_t a) { return reinterpret_cast<uintptr_t>(ptr) % a == 0; }

}  // namespace

kd_status fold_tc_run(const kd_fold_mat* mats, int count, int64_t batch, cudaStream_t s) {
  // channel tiles numbered longest vectors first, so that the long ones of a layer are not
  // the last ones started
  int order[KD_MAX_BATCH];
  for (int i = 0; i < count; ++i) order[i] = i;
  for (int i = 1; i < count; ++i)
    for (int k = i; k > 0 && mats[order[k]].n > mats[order[k - 1]].n; --k) {
      const int tmp = order[k];
      order[k] = order[k - 1];
      order[k - 1] = tmp;
    }
  cudaError_t e = cudaFuncSetAttribute(fold_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return KD_ERR_CUDA;
  constexpr int64_t kMaxRows = 1 << 16;  // batch rows per launch
  for (int64_t b0 = 0; b0 < batch; b0 += kMaxRows) {
    FoldTcParams p;
    p.rows = (int)(batch - b0 < kMaxRows ? batch - b0 : kMaxRows);
    p.row_blocks = (p.rows + kRows - 1) / kRows;
    // Up to one row block, two parts per plane: a small layer's tiles alone leave places idle
    // (16 rows, before the digits: one 4096 x 11008 matrix 78 -> 44 us, a 768-wide layer's six
    // 27 -> 19), and the 7B layer takes the same (119 -> 116 us at 2 rows, 130 at 16).  Four parts
    // were slower (7B layer 159 us at 16 rows), and with more row blocks two already are (17
    // rows: 222 -> 238).  Not by the number of tiles: a matrix's results do not depend on the others'.
    p.split = p.rows <= kRows ? 2 : 1;
    p.count = 0;
    int64_t tiles = 0;
    for (int i = 0; i < count; ++i) {
      const kd_fold_mat& a = mats[order[i]];
      if (a.m == 0) continue;
      p.tile0[p.count] = (uint32_t)tiles;
      FoldTcMat& f = p.mat[p.count++];
      f.codes[0] = a.codes_u;
      f.codes[1] = a.codes_v;
      f.centres[0] = a.centres_u;
      f.centres[1] = a.centres_v;
      f.x[0] = a.x + b0 * a.ldx;
      f.x[1] = a.xp + b0 * a.ldx;
      f.y = a.y + b0 * a.ldy;
      f.n = a.n;
      f.m = a.m;
      f.words = (a.n + 15) / 16;
      f.ldx = a.ldx;
      f.ldy = a.ldy;
      f.vec_codes = aligned_to(a.codes_u, 16) && aligned_to(a.codes_v, 16) && f.words % 4 == 0;
      f.vec_x = aligned_to(f.x[0], 16) && aligned_to(f.x[1], 16) && a.ldx % 4 == 0 && a.n % 4 == 0;
      tiles += (a.m + kTile - 1) / kTile;
    }
    if (tiles == 0) return KD_OK;
    row_grid_kernel<<<(unsigned)(p.count * p.rows * 2 * p.split), kGridThreads, 0, s>>>(p);
    if (cudaGetLastError() != cudaSuccess) return KD_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * p.row_blocks * 2 * p.split));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)(2 * p.split);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, fold_tc_kernel, p) != cudaSuccess) return KD_ERR_CUDA;
  }
  return KD_OK;
}

}  // namespace kd
