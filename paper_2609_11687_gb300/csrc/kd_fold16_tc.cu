// The folded 2-bit layer product of App. C for 16-bit activations on tcgen05, for more than
// 8 batch rows (kd_fold16.cu states the product and takes fewer rows and wide, short matrices).  The code planes
// are read and decoded once per block of up to 256 batch rows.
//
// Mapping.  tcgen05.mma with M = 128 output channels, N = the batch rows of the block,
// K = the inputs: u plane against x, then v plane against xp.  A CTA owns one tile of 128
// channels and (part of) K, cut into units of 128 inputs, each two stages of 64:
//  * two groups of eight warps decode the codes, every other unit each: a thread reads 16
//    bytes of its channel's code row, turns them into 64 16-bit centres and writes them to
//    its TMEM lane (sixteen warps: with eight, two per scheduler, the decode's dependent
//    chains left the MMAs waiting at 256 rows.  A in TMEM: through shared memory its writes
//    and reads, with B's, filled the bandwidth, and 512 rows took 304 us);
//  * one thread loads the B tiles (64 inputs of every batch row) by TMA, zero past the last
//    input and the last row; where the rows are not 16-byte aligned the decoding threads
//    fill them instead, element by element;
//  * one thread issues the MMAs.
// The accumulators live in TMEM, in two buffers where they fit beside the A slots (up to 128
// rows).  Every few units the decoding warps add the finished sums to fp32 registers,
// while the next ones go to the other buffer: the tensor core cuts its additions off instead of
// rounding them, so its chains are kept at n / 32 steps (those of the mma.sync kernel's four
// warps), between 8 and 64.  With 64 at every n, the error at n = 768 and more than 128 rows was
// 1.1e-6 of the result's norm (2.2 times the mma.sync kernel's), at n = 256 3.5 times.
//
// Split of K.  The decode of 128 x 128 weights costs 370 SM cycles of the ALU pipe at least,
// the MMAs 4 N, so up to about 90 rows the time is the decode's and every SM has to take its
// share: blocks of at most 64 rows run as clusters of four CTAs per tile (two up to 128
// rows), each with a part of K, whose partial sums are added over distributed shared memory
// in rank order.  The split follows from the batch alone, so a matrix gives the same bits
// alone and in a batched call.
//
// Measured (7B layer): 87 / 95 / 99 / 117 / 280 us at 9 / 33 / 64 / 129 / 512 rows; at
// 512 rows that is 1.45 PFLOP/s, 75 % of the measured bf16 rate.  The MMA thread branches on
// elect.sync (kd_tc.cuh): with a lane test instead, every tcgen05 instruction cost a loop
// over the lanes and 512 rows took 422 us.
#include <cuda_runtime.h>

#include "kashin.h"
#include "kd_dec16.cuh"
#include "kd_fold16.h"
#include "kd_tc.cuh"
#include "kd_tc_host.h"

namespace kd {
namespace {

constexpr int kTile = 128;        // output channels per CTA (the MMA's M, the TMEM lanes)
constexpr int kStageK = 64;       // inputs per stage: one 128-byte row of 16-bit values
constexpr int kUnitK = 128;       // inputs per unit: two stages
constexpr int kChunk = 8;         // units per TMEM accumulation at most (64 MMA steps)
constexpr int kDecWarps = 16;     // decoding warps: two groups of eight
constexpr int kThreads = 32 * (kDecWarps + 2);  // + the TMA warp and the MMA warp
constexpr int kMaxA = 4;          // A slots (units), at most
constexpr int kMaxB = 8;          // B slots, at most
constexpr int kACols = 64;        // TMEM columns of one unit of A

struct alignas(128) FoldTcMat {
  CUtensorMap map_x, map_xp;  // launches with TMA only
  const uint32_t* codes_u;
  const uint32_t* codes_v;
  const float* centres_u;
  const float* centres_v;
  const unsigned short* x;
  const unsigned short* xp;
  float* y;
  int64_t n, m, words, ldx, ldy;
  int units;       // units of one plane
  int chunk;       // units per TMEM accumulation
  int vec;        // code rows 16-byte aligned: 128-bit code loads
};

struct FoldTcParams {
  uint32_t tile0[KD_MAX_BATCH];  // first channel tile of each matrix
  int count;
  int rows;        // batch rows of the call
  int row_blocks;  // blocks of nt rows
  int nt;          // batch rows per block, a multiple of 16 (the MMA's N)
  int split;       // CTAs of the cluster that share a tile's K
  int slots_b;     // B ring depth
  DecodeMul mul;
  FoldTcMat mat[KD_MAX_BATCH];
};

// Shared state of a CTA besides the operand ring.
struct Ctl {
  uint64_t full_a[kMaxA], empty_a[kMaxA], full_b[kMaxB], empty_b[kMaxB], acc_full[2], acc_empty[2], drained;
  uint32_t tmem;
  int fail;  // a wait expired: the tile's outputs become NaN
};

__device__ __forceinline__ bool ctl_wait(Ctl* c, uint64_t* bar, uint32_t parity) { return tc_wait(bar, parity, &c->fail); }

// Resident CTAs per SM; TMEM columns of a CTA: tc_bufs accumulator buffers of ntc columns,
// then the A slots; stages of 64 inputs per B slot: with few rows a slot holds a whole unit,
// because there the MMA thread's waits and commits cost more than its MMAs; with many rows a
// slot holds one stage, which keeps more copies in flight.
__host__ __device__ constexpr int tc_ctas(int ntc) { return ntc >= 128 ? 1 : 2; }
__host__ __device__ constexpr int tc_cols(int ntc) { return 512 / tc_ctas(ntc); }
__host__ __device__ constexpr int tc_bufs(int ntc) { return ntc == 256 ? 1 : 2; }
__host__ __device__ constexpr int tc_slots_a(int ntc) {
  return (tc_cols(ntc) - tc_bufs(ntc) * ntc) / kACols < kMaxA ? (tc_cols(ntc) - tc_bufs(ntc) * ntc) / kACols : kMaxA;
}
__host__ __device__ constexpr int tc_bstages(int ntc) { return ntc >= 128 ? 1 : 2; }

// B tile of rows that TMA cannot read (not 16-byte aligned), by the 256 threads of a decoding
// group: 64 inputs from i0 of `nt` batch rows, zero past n and past `rows`.
__device__ __forceinline__ void fill_rows(uint32_t dst, const unsigned short* src, int64_t ldx, int64_t i0, int64_t n,
                                       int nt, int rows, int t) {
  for (int i = t; i < nt * 8; i += 2 * kTile) {
    const int r = i >> 3, ch = i & 7;  // batch row, 16-byte chunk
    uint32_t h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t i1 = i0 + 8 * ch + 2 * e;
      const unsigned short* q = src + r * ldx + i1;
      const uint32_t l = r < rows && i1 < n ? __ldg(q) : 0u;
      const uint32_t u = r < rows && i1 + 1 < n ? __ldg(q + 1) : 0u;
      h[e] = l | (u << 16);
    }
    sts128(dst + r * 128 + ((ch ^ (r & 7)) << 4), make_uint4(h[0], h[1], h[2], h[3]));
  }
}

// NTC: accumulator columns reserved per buffer (>= nt); TMA: B tiles by TMA
template <bool BF, int NTC, bool TMA>
__global__ void __launch_bounds__(kThreads, tc_ctas(NTC)) fold16_tc_kernel(const __grid_constant__ FoldTcParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ Ctl ctl;
  constexpr int NC = NTC / 4;  // accumulator columns per decoding warp
  constexpr uint32_t kCols = tc_cols(NTC);
  constexpr int NB = tc_bufs(NTC);
  constexpr int SA = tc_slots_a(NTC);
  constexpr int BH = tc_bstages(NTC);
  const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;  // the B slots
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const int lane = threadIdx.x & 31;
  const int S = p.slots_b;
  const int nt = p.nt;
  const uint32_t bstage = (uint32_t)nt * 128u, bbytes = BH * bstage;

  // this CTA's tile, row block and units [k0, k0 + L) of the 2 ku units of both planes
  const uint32_t split = (uint32_t)p.split;
  const uint32_t rank = split > 1 ? cluster_rank() : 0u;
  const uint32_t id = blockIdx.x / split;
  const uint32_t tile = id / (uint32_t)p.row_blocks;
  const int row0 = (int)(id - tile * p.row_blocks) * nt;
  int mi = 0;
  while (mi + 1 < p.count && tile >= p.tile0[mi + 1]) ++mi;
  const FoldTcMat& a = p.mat[mi];
  const int64_t c0 = (int64_t)(tile - p.tile0[mi]) * kTile;
  const int ku = a.units, chunk = a.chunk;
  const int k0 = (int)((uint32_t)(2 * ku) * rank / split);
  const int L = (int)((uint32_t)(2 * ku) * (rank + 1) / split) - k0;

  // the decoding threads' first code words, on their way during the set-up
  const int grp = warp >> 3, half = (warp >> 2) & 1;  // decoding group, its stage of a unit
  const int r = threadIdx.x & (kTile - 1);      // its channel of the tile, its TMEM lane
  const bool live = warp < kDecWarps && c0 + r < a.m;
  const uint32_t* ru = a.codes_u + (live ? c0 + r : 0) * a.words;
  const uint32_t* rv = a.codes_v + (live ? c0 + r : 0) * a.words;
  const int words = live ? (int)a.words : 0;
  const bool vec = a.vec;
  // the four code words of this thread's stage of unit u (zero past the row, the K range and m)
  auto fetch = [&](int u) -> uint4 {
    const int k = k0 + u;
    const uint32_t* src = k >= ku ? rv : ru;
    const int w0 = 8 * (k >= ku ? k - ku : k) + 4 * half;
    const int left = u < L ? words - w0 : 0;
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    if (vec) {  // rows of whole 16-byte blocks
      if (left > 0) w = __ldg(reinterpret_cast<const uint4*>(src + w0));
    } else {
      if (left > 0) w.x = __ldg(src + w0);
      if (left > 1) w.y = __ldg(src + w0 + 1);
      if (left > 2) w.z = __ldg(src + w0 + 2);
      if (left > 3) w.w = __ldg(src + w0 + 3);
    }
    return w;
  };
  uint4 w0 = fetch(grp), w1 = fetch(grp + 2);

  if (warp == kDecWarps) {
    if (lane < SA) {
      mbar_init(&ctl.full_a[lane], kDecWarps / 2);  // the warps of the decoding group
      mbar_init(&ctl.empty_a[lane], 1);
    }
    if (lane < S) {
      mbar_init(&ctl.full_b[lane], TMA ? 1 : kDecWarps / 2);
      mbar_init(&ctl.empty_b[lane], 1);
    }
    if (lane < 2) {
      mbar_init(&ctl.acc_full[lane], 1);
      mbar_init(&ctl.acc_empty[lane], kDecWarps);
    }
    if (lane == 0) {
      mbar_init(&ctl.drained, 1);
      ctl.fail = 0;
    }
    mbar_init_fence();
  }
  if (warp == kDecWarps + 1) tmem_alloc(&ctl.tmem, kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl.tmem;

  if (warp == kDecWarps) {
    // ---- B slots by TMA ----
    if (TMA) {
      int s = 0;
      uint32_t par = 1;  // the first round finds every slot free
      int issued = 0;
      for (int i = 0; i < L * (2 / BH); ++i) {
        if (i >= S && !__all_sync(0xffffffffu, ctl_wait(&ctl, &ctl.empty_b[s], par))) break;
        if (elect_one()) {
          const int k = k0 + (BH == 2 ? i : i >> 1);
          const CUtensorMap* map = k >= ku ? &a.map_xp : &a.map_x;
          const int x = (k >= ku ? k - ku : k) * kUnitK + (BH == 2 ? 0 : (i & 1) * kStageK);
          uint8_t* dst = smem_raw + (ring + s * bbytes - smem_u32(smem_raw));
          mbar_arrive_expect_tx(&ctl.full_b[s], bbytes);
#pragma unroll
          for (int h = 0; h < BH; ++h) tma_load_2d(dst + h * bstage, map, x + h * kStageK, row0, &ctl.full_b[s]);
        }
        __syncwarp();
        ++issued;
        if (++s == S) {
          s = 0;
          par ^= 1;
        }
      }
      // shared memory is not used otherwise, nor given back, before the copies have landed, also
      // after an expired wait (bounded as well)
      for (s = 0; s < S; ++s) {
        const int last = ring_last_parity(issued, S, s);
        if (last >= 0 && !mbar_wait_bounded(&ctl.full_b[s], last)) *(volatile int*)&ctl.fail = 1;
      }
    }
  } else if (warp == kDecWarps + 1) {
    // ---- MMAs ---- (the whole warp in the loop, so that its counters stay in uniform registers:
    // with one thread elected before it 512 rows of the 7B layer took 294 us, 283 so)
    const uint32_t idesc = tc_idesc(BF, nt);
    const uint64_t db0 = tc_desc(ring);
    int s = 0, sa = 0, left = chunk;  // units left of this accumulation
    uint32_t par = 0, par_a = 0, b = 0, par_acc = 1;
    bool ok = true, fresh = true;
    for (int u = 0; u < L && ok; ++u) {
      if (u >= NB * chunk && fresh) ok = ctl_wait(&ctl, &ctl.acc_empty[b], par_acc);
      ok = ok && ctl_wait(&ctl, &ctl.full_a[sa], par_a);
      const uint32_t ta = tmem + NB * NTC + sa * kACols;
      const uint32_t d = tmem + b * NTC;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (BH == 1 || h == 0) {
          ok = ok && ctl_wait(&ctl, &ctl.full_b[s], par);
          ok = __all_sync(0xffffffffu, ok);  // one answer for the warp (elect_one)
          tc_fence_after();
        }
        if (ok && elect_one()) {
          const uint64_t db = db0 + (uint64_t)(s * (bbytes >> 4)) + (BH == 2 ? h * (bstage >> 4) : 0u);
#pragma unroll
          for (int q = 0; q < kStageK / 16; ++q)
            tc_mma(d, ta + 32 * h + 8 * q, db + 2 * q, idesc, !fresh || h + q != 0);
          if (BH == 1 || h == 1) tc_commit(&ctl.empty_b[s]);
          if (h == 1) {
            tc_commit(&ctl.empty_a[sa]);
            if (left == 1 || u == L - 1) tc_commit(&ctl.acc_full[b]);
          }
        }
        __syncwarp();
        if ((BH == 1 || h == 1) && ++s == S) {
          s = 0;
          par ^= 1;
        }
      }
      if (++sa == SA) {
        sa = 0;
        par_a ^= 1;
      }
      fresh = --left == 0;
      if (fresh) {
        left = chunk;
        if (NB == 2) b ^= 1;
        if (b == 0) par_acc ^= 1;
      }
    }
  }
  __syncwarp();

  float acc[NC];
  if (warp < kDecWarps) {
    // ---- decode, and the fp32 sums ----
    const uint2 cu = centre_bytes<BF>(a.centres_u, c0 + r, live), cv = centre_bytes<BF>(a.centres_v, c0 + r, live);
    const uint32_t lanes = tmem + ((uint32_t)(warp & 3) << 21);  // this warp's 32 TMEM lanes
#pragma unroll
    for (int i = 0; i < NC; ++i) acc[i] = 0.f;
    int done = 0;  // chunks added so far
    auto promote = [&]() {
      const int b = NB == 2 ? done & 1 : 0;
      ctl_wait(&ctl, &ctl.acc_full[b], (NB == 2 ? done >> 1 : done) & 1);
      tc_fence_after();
      const uint32_t t = lanes + b * NTC + (warp >> 2) * NC;
#pragma unroll
      for (int q = 0; q < NC; q += 16) {
        constexpr int W = NC < 16 ? NC : 16;
        float v[W];
#pragma unroll
        for (int i = 0; i < W; i += 8) tmem_ld8(v + i, t + q + i);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < W; ++i) acc[q + i] = __fadd_rn(acc[q + i], v[i]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.acc_empty[b]);
      ++done;
    };
    // own units grp, grp + 2, ..., their code words loaded two own units ahead
#pragma unroll 1
    for (int u = grp; u < L; u += 2) {
      const uint32_t ww[4] = {w0.x, w0.y, w0.z, w0.w};
      w0 = w1;
      w1 = fetch(u + 4);
      const int s = u % SA;
      if (u >= SA) ctl_wait(&ctl, &ctl.empty_a[s], (u / SA - 1) & 1);
      tc_fence_after();  // the MMAs that read the slot are complete
      const bool v = k0 + u >= ku;
      const uint2 c = make_uint2(v ? cv.x : cu.x, v ? cv.y : cu.y);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint4 e0, e1;
        decode_word(ww[q], c, p.mul, e0, e1);
        tmem_st8(lanes + NB * NTC + s * kACols + 32 * half + 8 * q, e0, e1);
      }
      if constexpr (!TMA) {
        for (int h = 0; h < 2; ++h) {
          const int i = BH == 2 ? u : 2 * u + h, sb = i % S;
          if (i >= S) ctl_wait(&ctl, &ctl.empty_b[sb], (i / S - 1) & 1);
          fill_rows(ring + sb * bbytes + (BH == 2 ? h * bstage : 0u), (v ? a.xp : a.x) + row0 * a.ldx, a.ldx,
                    (int64_t)kUnitK * (v ? k0 + u - ku : k0 + u) + h * kStageK, a.n, nt, p.rows - row0, threadIdx.x & (2 * kTile - 1));
          if (BH == 1 || h == 1) {
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl.full_b[sb]);
          }
        }
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl.full_a[s]);
      // past the end of an accumulation (with two buffers, when its MMAs are known to be
      // complete): they need nothing more from this warp.  All that ended: an accumulation may be
      // one unit, and own units are two apart
      while (u >= (done + 1) * chunk + (NB == 2 ? SA - 1 : 0)) promote();
    }
    const int chunks = (L + chunk - 1) / chunk;
    while (done < chunks) promote();
  }
  // here and not after the MMA loop, where it cost the loop 2 to 5 % at 512 rows
  if (warp == kDecWarps + 1 && elect_one()) tc_drain(&ctl.drained, &ctl.fail);
  __syncthreads();
  const int cols = p.rows - row0 < nt ? p.rows - row0 : nt;  // batch rows of this block
  if (p.split == 1) {
    if (warp < kDecWarps) {
      const int64_t j = c0 + r;
      if (live) {
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          const int c = (warp >> 2) * NC + i;
          if (c < cols) a.y[(int64_t)(row0 + c) * a.ldy + j] = acc[i];
        }
      }
    }
  } else {
    // partial tiles into shared memory (the ring is idle), [column][channel]
    const uint32_t ch = r;
    if (warp < kDecWarps) {
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        const int c = (warp >> 2) * NC + i;
        if (c < cols) asm volatile("st.shared.f32 [%0], %1;" ::"r"(ring + (c * kTile + ch) * 4), "f"(acc[i]) : "memory");
      }
    }
    cluster_sync_all();
    if (warp < kDecWarps && c0 + ch < a.m) {
      for (int c = 4 * rank + (warp >> 2); c < cols; c += 4 * p.split) {
        float s = ld_dsmem(ring + (c * kTile + ch) * 4, 0);
        for (int q = 1; q < p.split; ++q) s = __fadd_rn(s, ld_dsmem(ring + (c * kTile + ch) * 4, q));
        a.y[(int64_t)(row0 + c) * a.ldy + c0 + ch] = s;
      }
    }
    cluster_sync_all();  // the peers' reads of this CTA's shared memory are done
  }
  if (*(volatile int*)&ctl.fail) {  // over whatever the tile's CTAs have written
    __syncthreads();
    for (int c = warp >> 2; live && c < cols; c += 4)
      a.y[(int64_t)(row0 + c) * a.ldy + c0 + r] = __int_as_float(0x7FC00000);
  }
  if (warp == kDecWarps + 1) tmem_dealloc(tmem, kCols);
}

bool aligned_to(const void* ptr, size_t a) { return reinterpret_cast<uintptr_t>(ptr) % a == 0; }

// cuTensorMapEncodeTiled, looked up once through the runtime (no link against libcuda)
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn() {
  static const EncodeFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult st;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &st) != cudaSuccess ||
        st != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeFn>(f);
  }();
  return fn;
}

// rows of 16-bit inputs as boxes of 64 inputs x nt rows, 128-byte swizzle, zero outside
bool encode_rows(CUtensorMap* map, const void* x, int64_t n, int64_t rows, int64_t ldx, int nt) {
  const EncodeFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)rows};
  // a single row's stride is never used
  const cuuint64_t strides[1] = {rows == 1 ? (cuuint64_t)(n + 7) / 8 * 16 : (cuuint64_t)ldx * 2};
  const cuuint32_t box[2] = {kStageK, (cuuint32_t)nt};
  const cuuint32_t step[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<void*>(x), dims, strides, box, step,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool BF, int NTC, bool TMA>
cudaError_t launch_tc(FoldTcParams& p, int64_t tiles, cudaStream_t s) {
  const int budget = tc_ctas(NTC) == 1 ? 224 * 1024 : 110 * 1024;
  const int slot = tc_bstages(NTC) * p.nt * 128;
  const int left = budget / slot;
  p.slots_b = left < kMaxB ? left : kMaxB;
  // at least what the partial tiles of a split take at the end
  const int used = p.slots_b * slot + 1024, least = tc_smem_floor(tc_cols(NTC));
  const size_t smem = (size_t)(used > least ? used : least);
  auto kernel = fold16_tc_kernel<BF, NTC, TMA>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles * p.row_blocks * p.split));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)p.split;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

template <bool BF>
cudaError_t launch_tc(FoldTcParams& p, int64_t tiles, bool tma, cudaStream_t s) {
  if (!tma) return p.nt <= 64 ? launch_tc<BF, 64, false>(p, tiles, s) : launch_tc<BF, 256, false>(p, tiles, s);
  if (p.nt <= 16) return launch_tc<BF, 16, true>(p, tiles, s);
  if (p.nt <= 32) return launch_tc<BF, 32, true>(p, tiles, s);
  if (p.nt <= 64) return launch_tc<BF, 64, true>(p, tiles, s);
  if (p.nt <= 128) return launch_tc<BF, 128, true>(p, tiles, s);
  return launch_tc<BF, 256, true>(p, tiles, s);
}

}  // namespace

kd_status fold16_tc_run(const kd_fold_mat_f16* mats, int count, int64_t batch, cudaStream_t s, bool bf) {
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
  constexpr int64_t kMaxRows = 1 << 16;  // batch rows per launch
  for (int64_t b0 = 0; b0 < batch; b0 += kMaxRows) {
    FoldTcParams p;
    p.rows = (int)(batch - b0 < kMaxRows ? batch - b0 : kMaxRows);
    p.row_blocks = (p.rows + 255) / 256;
    p.nt = ((p.rows + p.row_blocks - 1) / p.row_blocks + 15) / 16 * 16;
    p.split = p.nt <= 64 ? 4 : p.nt <= 128 ? 2 : 1;
    // the matrices whose rows TMA can read, then the others (16-byte alignment of the base
    // and, past one row, of the stride)
    for (int pass = 0; pass < 2; ++pass) {
      p.count = 0;
      int64_t tiles = 0;
      for (int i = 0; i < count; ++i) {
        const kd_fold_mat_f16& a = mats[order[i]];
        if (a.m == 0) continue;
        FoldTcMat& f = p.mat[p.count];
        f.x = static_cast<const unsigned short*>(a.x) + b0 * a.ldx;
        f.xp = static_cast<const unsigned short*>(a.xp) + b0 * a.ldx;
        const bool tma = aligned_to(f.x, 16) && aligned_to(f.xp, 16) && (a.ldx % 8 == 0 || p.rows == 1);
        if (tma != (pass == 0)) continue;
        f.codes_u = a.codes_u;
        f.codes_v = a.codes_v;
        f.centres_u = a.centres_u;
        f.centres_v = a.centres_v;
        f.y = a.y + b0 * a.ldy;
        f.n = a.n;
        f.m = a.m;
        f.words = (a.n + 15) / 16;
        f.ldx = a.ldx;
        f.ldy = a.ldy;
        p.tile0[p.count] = (uint32_t)tiles;
        f.units = (int)((a.n + kUnitK - 1) / kUnitK);
        f.chunk = a.n < 512 ? 1 : a.n / 256 < kChunk ? (int)(a.n / 256) : kChunk;
        f.vec = aligned_to(a.codes_u, 16) && aligned_to(a.codes_v, 16) && f.words % 4 == 0;
        if (tma && (!encode_rows(&f.map_x, f.x, a.n, p.rows, a.ldx, p.nt) ||
                    !encode_rows(&f.map_xp, f.xp, a.n, p.rows, a.ldx, p.nt)))
          return KD_ERR_CUDA;
        tiles += (a.m + kTile - 1) / kTile;
        ++p.count;
      }
      if (tiles == 0) continue;
      const cudaError_t e = bf ? launch_tc<true>(p, tiles, pass == 0, s) : launch_tc<false>(p, tiles, pass == 0, s);
      if (e != cudaSuccess) return KD_ERR_CUDA;
    }
  }
  return KD_OK;
}

}  // namespace kd
