// Decoding of 2-bit code words into 16-bit centres (fp16 or bf16), in registers.
#pragma once

#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace kd {

// a centre rounded (nearest, ties to even) to the activations' 16-bit type, as bits
template <bool BF>
__device__ __forceinline__ uint32_t bits16(float c) {
  if constexpr (BF) return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(c));
  else return (uint32_t)__half_as_ushort(__float2half_rn(c));
}

// The 16-bit centres of one channel as (low bytes, high bytes), zero past m.
template <bool BF>
__device__ __forceinline__ uint2 centre_bytes(const float* centres, int64_t j, bool ok) {
  if (!ok) return make_uint2(0u, 0u);
  const float4 c = __ldg(reinterpret_cast<const float4*>(centres) + j);
  const uint32_t p01 = bits16<BF>(c.x) | (bits16<BF>(c.y) << 16);
  const uint32_t p23 = bits16<BF>(c.z) | (bits16<BF>(c.w) << 16);
  return make_uint2(__byte_perm(p01, p23, 0x6420u), __byte_perm(p01, p23, 0x7531u));
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// Factors of decode_word.  They come from the kernel's parameters: as constants the
// compiler would turn the products into shifts and adds on the ALU pipe.
struct DecodeMul {
  uint32_t a = 65, b = 0x11;
};

// The 16 centres of one code word in order, as 16-bit pairs.  The centres' low and high
// bytes are two words, and one byte permute with the selector nibbles (q0, q0 + 4, q1,
// q1 + 4) yields the pair of codes q0, q1.  The selectors of codes 2i, 2i + 1 and 2i + 8,
// 2i + 9 are formed together: v = q0 | q1 << 2 in each half, (65 v) & 0x0303 puts q0 and q1
// into bytes, times 0x11 plus 0x4040 makes the nibbles.  Bound by the ALU pipe (two cycles
// per warp instruction): 23 of its instructions per word, the products run beside it, and
// the permute is the bare instruction because __byte_perm masks its selector first.
// Measured on all SMs: 46 cycles per word and warp, against 65 with the masks, shifts and
// __byte_perm, and 47 with the upper selectors taken from 64-bit products.
__device__ __forceinline__ void decode_selectors(uint32_t w, const DecodeMul& mul, uint32_t (&sel)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t x = (((w >> (4 * i)) & 0x000F000Fu) * mul.a) & 0x03030303u;
    sel[i] = x * mul.b + 0x40404040u;
    sel[i + 4] = sel[i] >> 16;
  }
}
// The same for an order of the codes in which the selectors need no multiplex: sel[i] gives
// codes i and i + 4, sel[i + 4] codes i + 8 and i + 12 (11 ALU instructions instead of 15).
__device__ __forceinline__ void decode_selectors_by4(uint32_t w, const DecodeMul& mul, uint32_t (&sel)[8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    sel[i] = ((w >> (2 * i)) & 0x03030303u) * mul.b + 0x40404040u;
    sel[i + 4] = sel[i] >> 16;
  }
}
__device__ __forceinline__ void decode_pick(const uint32_t (&sel)[8], uint2 c, uint4& lo, uint4& hi) {
  lo = make_uint4(prmt(c.x, c.y, sel[0]), prmt(c.x, c.y, sel[1]), prmt(c.x, c.y, sel[2]), prmt(c.x, c.y, sel[3]));
  hi = make_uint4(prmt(c.x, c.y, sel[4]), prmt(c.x, c.y, sel[5]), prmt(c.x, c.y, sel[6]), prmt(c.x, c.y, sel[7]));
}
__device__ __forceinline__ void decode_word(uint32_t w, uint2 c, const DecodeMul& mul, uint4& lo, uint4& hi) {
  uint32_t sel[8];
  decode_selectors(w, mul, sel);
  decode_pick(sel, c, lo, hi);
}

__device__ __forceinline__ void sts128(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

}  // namespace kd
