// Decode of packed RaZeR blocks to bf16 pairs for the tcgen05 matmul kernel, in registers and by table, and what the other kernels share
// of it.
//
// In registers, per pair of elements, with no comparison and no conversion instruction: the stored nibble
// is isolated in both 16-bit halves of the word, one integer multiply-add drops two shifted
// copies of it, one logic op keeps sign -> bit 15 and E1 E0 M -> bits 8:6 (a bf16 pattern worth
// value x 2^-126, subnormal for 0.5) and ORs in the special value, which one fused
// multiply-add with ReLU derives from the isolated nibble (the special value is the only
// nibble that is numerically zero); one packed bf16 multiply by +-scale x 2^126 finishes the
// exact product value x block scale (Sec. 3: dequantized element, without the tensor scale).
#pragma once

#include "razer_common.cuh"

namespace razer {

// Packed bf16 arithmetic on raw 32-bit patterns, through the compiler's own intrinsics (rather than
// inline PTX) so that it can place results directly in the consecutive registers the TMEM store or the
// MMA wants.
__device__ __forceinline__ __nv_bfloat162 as_bf162(uint32_t v) { return *reinterpret_cast<__nv_bfloat162*>(&v); }
__device__ __forceinline__ uint32_t as_u32(__nv_bfloat162 v) { return *reinterpret_cast<uint32_t*>(&v); }
__device__ __forceinline__ uint32_t fma_relu_bf16x2(uint32_t a, uint32_t b, uint32_t c) {
  return as_u32(__hfma2_relu(as_bf162(a), as_bf162(b), as_bf162(c)));
}
__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) { return as_u32(__hmul2(as_bf162(a), as_bf162(b))); }
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | c; }

// Decode table in shared memory.
//   ss[(negate << 6 | scale code)][lane] : (+-scale x 2^126) as bf16x2; one copy per lane so that a
//                                          warp's 32 lookups never collide on a bank
constexpr int DECODE_SS_ENTRIES = 128;
constexpr int DECODE_TABLE_BYTES = DECODE_SS_ENTRIES * 32 * 4;

// Fill the table (all threads of the CTA call this; a __syncthreads() must follow).
__device__ __forceinline__ void decode_tables_fill(uint8_t* base, int tid, int nthreads) {
  // every entry is computed once per quarter (four threads per entry) and written as eight of its 32 lane copies
  for (int i = tid; i < DECODE_SS_ENTRIES * 4; i += nthreads) {
    const uint32_t idx = (uint32_t)i >> 2;
    // scale x 2^126 has four significant bits: the upper half of the FP32 pattern is the exact bf16
    const float sc = scale_value(idx & 0x3Fu) * 8.50705917e37f;   // 2^126
    const uint32_t b = (__float_as_uint(sc) >> 16) | ((idx & 0x40u) << 9);
    const uint32_t v = b | (b << 16);
    uint4* dst = reinterpret_cast<uint4*>(base + idx * 128 + (i & 3) * 32);
    dst[0] = make_uint4(v, v, v, v);
    dst[1] = make_uint4(v, v, v, v);
  }
}
// (sv x 2^-126, sv x 2^-126) as bf16x2; sv has at most four significant bits.
__host__ __device__ __forceinline__ uint32_t special_value_pair(float sv) {
  union { float f; uint32_t u; } b;
  b.f = sv * 1.17549435e-38f;
  return (b.u >> 16) | (b.u & 0xFFFF0000u);
}

// Scale pair of block `blk` (0..3, compile-time) of a chunk, from the row's scale word (four packed scale bytes
// [select | negate | 6-bit scale code]); ss_lane = shared-window address of &ss[0][lane].
__device__ __forceinline__ uint32_t decode_block_scale(uint32_t ss_lane, uint32_t sw, int blk) {
  return lds32(ss_lane + ((blk == 0 ? sw << 7 : sw >> (8 * blk - 7)) & 0x3F80u));   // (byte & 0x7F) * 128
}

// Four stored nibbles of each 16-bit half of `w` -> four bf16x2 registers (elements 2p, 2p + 1 of the word in
// register p), each the exact product value x scale with the block's sign.  The special value is the one
// nibble that is numerically zero when the isolated nibble is read as a bf16 pair: relu(nibble * -2^11 + sv')
// is sv' = sv x 2^-126 for it and 0 for every other nibble (the smallest, 2^-133, times 2^11 already exceeds
// the largest sv').
// mul_lo = 2^6 + 2^12, mul_hi = 2^2 + 2^8 (run-time values so that they stay multiplies): one shifted copy of the nibble
// lands with E1 E0 M on bits 8:6, the other with S on bit 15; the mask keeps exactly those.
__device__ __forceinline__ void decode_word(uint32_t w, uint32_t ss2, uint32_t svp, uint32_t mul_lo, uint32_t mul_hi, uint32_t* out) {
  constexpr uint32_t NEG = 0xC500C500u;               // (-2048, -2048) as bf16x2
  const uint32_t w8 = w >> 8;
  const uint32_t n0 = w & 0x000F000Fu, n1 = w & 0x00F000F0u;
  const uint32_t n2 = w8 & 0x000F000Fu, n3 = w8 & 0x00F000F0u;
  const uint32_t u0 = and_or(n0 * mul_lo, 0x81C081C0u, fma_relu_bf16x2(n0, NEG, svp));
  const uint32_t u1 = and_or(n1 * mul_hi, 0x81C081C0u, fma_relu_bf16x2(n1, NEG, svp));
  const uint32_t u2 = and_or(n2 * mul_lo, 0x81C081C0u, fma_relu_bf16x2(n2, NEG, svp));
  const uint32_t u3 = and_or(n3 * mul_hi, 0x81C081C0u, fma_relu_bf16x2(n3, NEG, svp));
  out[0] = mul_bf16x2(u0, ss2);
  out[1] = mul_bf16x2(u1, ss2);
  out[2] = mul_bf16x2(u2, ss2);
  out[3] = mul_bf16x2(u3, ss2);
}


// The same pairs by table: [weight byte][special value][lane], two elements (value x 2^-126) to an entry, a copy per lane so that 32
// random lookups never meet on a bank.  A pair costs a byte permute (which forms the address), a load and the multiply by the
// scale; another permute each puts the pairs back in order, since a byte of a code word holds elements 0, 2 / 4, 6 / 1, 3 / 5, 7.
// Eight weights are 21 instructions in registers and 16 this way; in the tcgen05 kernel at 16 tokens 1032 warp instructions a chunk,
// everything included, became 856.
constexpr int PAIR_TABLE_BYTES = 65536;
__device__ __forceinline__ void pair_table_fill(uint32_t base, int tid, int nthreads, uint32_t svp0, uint32_t svp1) {
#pragma unroll 1
  for (int e = tid; e < 512; e += nthreads) {
    auto element = [&](uint32_t nib) { return nib ? ((nib & 7u) << 6) | ((nib & 8u) << 12) : ((e & 1) ? svp1 : svp0) & 0xFFFFu; };
    const uint32_t v = element(((uint32_t)e >> 1) & 0xFu) | (element((uint32_t)e >> 5) << 16);
#pragma unroll
    for (int j = 0; j < 8; ++j)                             // each lane starts elsewhere in its row
      asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(base + (uint32_t)e * 128 + (uint32_t)((j + tid) & 7) * 16), "r"(v) : "memory");
  }
}
// Byte B of a code word; `row` = select bit (bit 7) | lane * 4.
template <int B>
__device__ __forceinline__ uint32_t pair_lookup(const uint8_t* table, uint32_t w, uint32_t row) {
  return *reinterpret_cast<const uint32_t*>(table + __byte_perm(w, row, 0x7604 | (B << 4)));
}
// The pairs of two blocks, unscaled; `rows` = the chunk's select bits (bit 7 of each byte) | lane * 4 in every byte.
__device__ __forceinline__ void lookup_blocks(const uint8_t* table, uint32_t rows, int blk, const uint2 (&cw)[CHUNK_BLOCKS], uint32_t (&pairs)[16]) {
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const uint32_t row = __byte_perm(rows, 0, 0x4440 | (blk + b));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t w = h ? cw[blk + b].y : cw[blk + b].x;
      uint32_t* p = pairs + 8 * b + 4 * h;
      p[0] = pair_lookup<0>(table, w, row);                 // elements 0, 2
      p[1] = pair_lookup<2>(table, w, row);                 // 1, 3
      p[2] = pair_lookup<1>(table, w, row);                 // 4, 6
      p[3] = pair_lookup<3>(table, w, row);                 // 5, 7
    }
  }
}
// ... scaled and put in order.
__device__ __forceinline__ void finish_blocks(const uint32_t (&pairs)[16], uint32_t s0, uint32_t s1, uint32_t* out) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint32_t s = q < 4 ? s0 : s1, x = mul_bf16x2(pairs[2 * q], s), y = mul_bf16x2(pairs[2 * q + 1], s);
    out[2 * q] = __byte_perm(x, y, 0x5410);
    out[2 * q + 1] = __byte_perm(x, y, 0x7632);
  }
}

}  // namespace razer
