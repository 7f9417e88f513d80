// Quantizers: razer_quant_act / razer_quant_act_fp4 (online, bf16 activations) and razer_quant_weight (offline, FP32
// weights).  Sec. 4.2, Eq. 1-3, 6-7.
//
// Every FP32 result that decides something (block scale, scaled values, candidate errors) has the value of the correctly
// rounded IEEE operations in a fixed order, issued through intrinsics, so the compiler can neither fuse nor reorder
// them and the decisions are reproducible bit for bit.  (Not every one is computed by that one operation: the quotients below
// are corrected products.)
//
// What bounds these kernels: instruction issue until the arithmetic per element is cut down, then DRAM.  The three costs
// that mattered, and what replaced them:
//   * x / denom, 16 IEEE divisions per block: one correctly rounded reciprocal per block and Markstein's correction
//     (P. Markstein, IBM J. Res. Dev. 34, 1990): with y = RN(1/b) and q within an ulp of a/b, RN(q + RN(a - b q) y) is
//     RN(a/b).  One correction is enough for bf16 numerators (all 2^30 pairs of an 8-bit numerator with a 24-bit
//     denominator agree with the IEEE division); FP32 numerators take two, the first of which makes q faithful.
//   * rounding to FP4, seven compares and adds: the e2m1 conversion instruction (nearest, ties to even, saturating),
//     two elements at a time, and one exponent-aligned add and subtract where the value itself is needed.
//   * two errors per candidate pair: by symmetry +sv and -sv need one comparison on |x|, and each element's squared
//     distance goes to one sum or the other by its sign.
// A block that the short form cannot take (a NaN or an infinity, a step outside 2^-60 .. 2^60, a quotient beyond 2^100) goes
// through the plain procedure.  Measured on B200, everything in this file included: razer_quant_act of 2048 x 8192 54.2 -> 27.2 us,
// razer_quant_act_fp4 (no special value) 58.1 -> 19.6; razer_quant_weight of 11008 x 4096 256.6 -> 94.6, of which the maximum 32, and
// by gains instead of error sums (quant_weight_quick_kernel) 71.3.
#include <algorithm>

#include "razer_common.cuh"
#include "razer_ptx.cuh"

namespace razer {

// Round a non-negative finite float to the nearest E4M3 code (ties to even mantissa),
// saturating at `max_code`.
__device__ __forceinline__ uint32_t round_to_e4m3(float t, uint32_t max_code) {
  uint32_t code;
  if (t < 0.015625f) {                       // below 2^-6: subnormal grid, quantum 2^-9
    code = (uint32_t)__float2int_rn(__fmul_rn(t, 512.0f));   // exact product, ties to even
  } else {
    const uint32_t b = __float_as_uint(t);
    const uint32_t e = (b >> 23) - 120u;     // biased E4M3 exponent (>= 1 here)
    const uint32_t man = b & 0x7FFFFFu;
    const uint32_t keep = man >> 20, rem = man & 0xFFFFFu;
    const uint32_t up = (rem > 0x80000u) || (rem == 0x80000u && (keep & 1u));
    code = (e >= 32u) ? max_code : ((e << 3) | keep) + up;   // a mantissa carry bumps the exponent
  }
  return min(code, max_code);
}

// Saturating round-to-nearest-even onto the FP4 magnitudes 0 .5 1 1.5 2 3 4 6 (Eq. 3).
__device__ __forceinline__ uint32_t round_to_fp4_idx(float a) {
  return (uint32_t)(a > 0.25f) + (uint32_t)(a >= 0.75f) + (uint32_t)(a > 1.25f) +
         (uint32_t)(a >= 1.75f) + (uint32_t)(a > 2.5f) + (uint32_t)(a >= 3.5f) + (uint32_t)(a > 5.0f);
}

// The short form of a block's arithmetic: valid for finite inputs below 2^100, steps within 2^-60 .. 2^60 and quotients below 2^100
// (a quotient that FP32 cannot hold would be infinite and its correction a NaN).  (An element
// below 2^-100 may then miss its quotient's last bit, which is far below anything the error sums of a block whose
// candidates differ can see: such an element's share is under 2^-80, a difference between candidates over 2^-40.)
__device__ __forceinline__ bool short_form(float bmax, float denom) {
  return bmax < 1.0e30f && bmax < denom * 1.0e30f && denom > 8.6736174e-19f && denom < 1.1529215e18f;
}
// Two FP32 values in one 64-bit register: the packed instructions round each half like their scalar forms and take one issue
// slot for both, which is what the quantizers are bound by.
struct F2 { uint64_t v; };
__device__ __forceinline__ F2 f2(float a, float b) { F2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void split(F2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v)); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) { F2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) { F2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r; }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { F2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r; }
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return fma2(b, f2(-1.0f, -1.0f), a); }   // one rounding, of a - b
__device__ __forceinline__ F2 abs2(F2 x) { float a, b; split(x, a, b); return f2(fabsf(a), fabsf(b)); }

// x / d correctly rounded, nd = -d, y = RN(1/d); x has at most eight significant bits.
__device__ __forceinline__ F2 div_bf16(F2 x, F2 nd, F2 y) {
  const F2 q = mul2(x, y);
  return fma2(fma2(q, nd, x), y, q);
}
// x / d correctly rounded, nd = -d, y = RN(1/d), any x.
__device__ __forceinline__ F2 div_f32(F2 x, F2 nd, F2 y) {
  F2 q = mul2(x, y);
  q = fma2(fma2(q, nd, x), y, q);
  return fma2(fma2(q, nd, x), y, q);
}
// |x| rounded to the nearest FP4 magnitude, ties to even mantissa, saturating: adding 2^22 times the power of two at or
// below a (at least 1) leaves two significant bits (steps of 0.5 below 2, 1 below 4, 2 from there on).
__device__ __forceinline__ F2 round_to_fp4(F2 a) {
  float a0, a1;
  split(a, a0, a1);
  const F2 c = f2(__uint_as_float((max(__float_as_uint(a0), 0x3F800000u) & 0x7F800000u) + (22u << 23)),
                  __uint_as_float((max(__float_as_uint(a1), 0x3F800000u) & 0x7F800000u) + (22u << 23)));
  float r0, r1;
  split(sub2(add2(a, c), c), r0, r1);
  return f2(fminf(r0, 6.0f), fminf(r1, 6.0f));
}
// Error of two scaled magnitudes under special value m (`d_r`: their distances to FP4): squares of the smaller distance, and
// which elements are strictly closer to m.
__device__ __forceinline__ F2 special_error(F2 a, F2 d_r, F2 minus_m, bool& t0, bool& t1) {
  float r0, r1, s0, s1;
  split(d_r, r0, r1);
  split(add2(a, minus_m), s0, s1);
  t0 = fabsf(s0) < fabsf(r0);
  t1 = fabsf(s1) < fabsf(r1);
  const F2 d = f2(t0 ? s0 : r0, t1 ? s1 : r1);
  return mul2(d, d);
}
// Error sums of a positive and a negative special value, both continued by two elements (in order): an element's error is q_t under
// the special value of its own sign and q_r under the other.
__device__ __forceinline__ void add_errors(F2& e, F2 q_r, F2 q_t, bool neg0, bool neg1) {
  float r0, r1, t0, t1;
  split(q_r, r0, r1);
  split(q_t, t0, t1);
  e = add2(e, neg0 ? f2(r0, t0) : f2(t0, r0));
  e = add2(e, neg1 ? f2(r1, t1) : f2(t1, r1));
}
// Eight values to FP4 codes, v[i] in nibble i (nearest, ties to even, saturating at 6; -0 and negative values that round to
// zero give code 8).
__device__ __forceinline__ uint32_t to_fp4x8(float v0, float v1, float v2, float v3, float v4, float v5, float v6, float v7) {
  uint32_t w;
  asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};\n\t}"
      : "=r"(w)
      : "f"(v0), "f"(v1), "f"(v2), "f"(v3), "f"(v4), "f"(v5), "f"(v6), "f"(v7));
  return w;
}
// Bit 3 of every nibble whose magnitude bits are not all zero.
__device__ __forceinline__ uint32_t nonzero_nibbles(uint32_t w) { return ((w & 0x77777777u) + 0x77777777u) & 0x88888888u; }

// Nibble position (in the 64 bits of a block's codes) of element j: the interchange order, or the packed form's order
// (nibbles p and p + 4 of a word = elements 2p and 2p + 1) of the FP4 operand.
template <bool PACKED>
__device__ __forceinline__ constexpr int elem_at(int nib) {   // element whose code sits in nibble `nib` (0..15)
  return PACKED ? (nib & 8) + 2 * (nib & 3) + ((nib >> 2) & 1) : nib;
}

// Quantize one 16-element block (Eq. 2-3, 6-7 with the candidates +sv and -sv): eight code bytes and the scale byte.
// The plain procedure, one IEEE division per element; interchange order.
__device__ __noinline__ void quant_act_block_plain(const uint4 v0, const uint4 v1, float d32, float d32x6, float sv_mag,
                                                   uint32_t& w0, uint32_t& w1, uint32_t& sbyte) {
  const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
  float xv[16];
  float bmax = 0.0f;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    xv[2 * j] = __uint_as_float(w[j] << 16);
    xv[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
    bmax = fmaxf(bmax, fmaxf(fabsf(xv[2 * j]), fabsf(xv[2 * j + 1])));
  }
  w0 = 0, w1 = 0, sbyte = 0;
  if (bmax > 0.0f) {
    const float tq = __fdiv_rn(bmax, d32x6);                         // Eq. 2 argument
    uint32_t scode = round_to_e4m3(tq, 126u);
    if (scode == 0) scode = 1;                                       // keep a non-empty block alive
    const float denom = __fmul_rn(d32, scale_value(scode));
    float e_pos = 0.0f, e_neg = 0.0f;
    uint32_t std_code[16];
    uint32_t take_pos = 0, take_neg = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float xs = __fdiv_rn(xv[j], denom);                      // the scaled block of Eq. 6
      const uint32_t idx = round_to_fp4_idx(fabsf(xs));
      const uint32_t neg = __float_as_uint(xs) >> 31;
      const float r = neg ? -fp4_mag(idx) : fp4_mag(idx);
      const float d_r = fabsf(__fsub_rn(xs, r));
      const float d_p = fabsf(__fsub_rn(xs, sv_mag));
      const float d_n = fabsf(__fsub_rn(xs, -sv_mag));
      const bool tp = d_p < d_r, tn = d_n < d_r;                     // strictly closer only
      const float qp = tp ? sv_mag : r, qn = tn ? -sv_mag : r;
      const float dp = __fsub_rn(qp, xs), dn = __fsub_rn(qn, xs);
      e_pos = __fadd_rn(e_pos, __fmul_rn(dp, dp));                   // ascending j, no fusion
      e_neg = __fadd_rn(e_neg, __fmul_rn(dn, dn));
      take_pos |= (uint32_t)tp << j;
      take_neg |= (uint32_t)tn << j;
      std_code[j] = idx ? (idx | (neg << 3)) : 0u;                   // a true zero is always code 0
    }
    const bool use_neg = e_neg < e_pos;                              // ties keep metadata 0 (+sv)
    const uint32_t take = use_neg ? take_neg : take_pos;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t c = ((take >> j) & 1u) ? 8u : std_code[j];
      if (j < 8) w0 |= c << (4 * j); else w1 |= c << (4 * (j - 8));
    }
    sbyte = (use_neg ? 0x80u : 0u) | scode;
  }
}

// The same block in the short form.  SV = false: no special value (plain NVFP4).  PACKED: the order of the codes.
template <bool SV, bool PACKED>
__device__ __forceinline__ void quant_act_block(const uint4 v0, const uint4 v1, float d32, float d32x6, float sv_mag,
                                                uint32_t& w0, uint32_t& w1, uint32_t& sbyte) {
  const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
  uint32_t m2 = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) m2 = __vmaxu2(m2, w[j] & 0x7FFF7FFFu);
  const uint32_t mbits = max(m2 & 0xFFFFu, m2 >> 16);
  w0 = 0, w1 = 0, sbyte = 0;
  if (mbits == 0) return;
  const float bmax = __uint_as_float(mbits << 16);
  uint32_t scode = round_to_e4m3(__fdiv_rn(bmax, d32x6), 126u);      // Eq. 2
  if (scode == 0) scode = 1;                                         // keep a non-empty block alive
  const float denom = __fmul_rn(d32, scale_value(scode));
  if (mbits >= 0x7F80u || !short_form(bmax, denom)) {
    quant_act_block_plain(v0, v1, d32, d32x6, SV ? sv_mag : 0.0f, w0, w1, sbyte);
    if (PACKED) {
      uint32_t o[2] = {0, 0};
#pragma unroll
      for (int n = 0; n < 16; ++n) o[n >> 3] |= (((elem_at<true>(n) < 8 ? w0 : w1) >> (4 * (elem_at<true>(n) & 7))) & 0xFu) << (4 * (n & 7));
      w0 = o[0], w1 = o[1];
    }
    return;
  }
  const float y = __frcp_rn(denom);
  const F2 y2 = f2(y, y), nd2 = f2(-denom, -denom);
  float xs[16];
#pragma unroll
  for (int j = 0; j < 8; ++j)                                        // the scaled block of Eq. 6
    split(div_bf16(f2(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xFFFF0000u)), nd2, y2), xs[2 * j], xs[2 * j + 1]);
  uint32_t c[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int b = 8 * h;
    c[h] = to_fp4x8(xs[elem_at<PACKED>(b)], xs[elem_at<PACKED>(b + 1)], xs[elem_at<PACKED>(b + 2)], xs[elem_at<PACKED>(b + 3)],
                    xs[elem_at<PACKED>(b + 4)], xs[elem_at<PACKED>(b + 5)], xs[elem_at<PACKED>(b + 6)], xs[elem_at<PACKED>(b + 7)]);
  }
  bool use_neg = false;
  uint32_t take[2] = {0, 0};                                         // bit 3 of the nibbles strictly closer to sv than to FP4
  if (SV) {
    F2 e = f2(0.0f, 0.0f);
    const F2 minus_sv = f2(-sv_mag, -sv_mag);
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
      const F2 a = f2(fabsf(xs[j]), fabsf(xs[j + 1])), d_r = sub2(a, round_to_fp4(a));
      bool t0, t1;
      const F2 q_t = special_error(a, d_r, minus_sv, t0, t1);
      add_errors(e, mul2(d_r, d_r), q_t, __float_as_uint(xs[j]) >> 31, __float_as_uint(xs[j + 1]) >> 31);   // ascending j, no fusion
      const int n0 = PACKED ? (j & 8) + ((j & 7) >> 1) : j, n1 = PACKED ? n0 + 4 : j + 1;
      if (t0) take[n0 >> 3] |= 8u << (4 * (n0 & 7));
      if (t1) take[n1 >> 3] |= 8u << (4 * (n1 & 7));
    }
    float e_pos, e_neg;
    split(e, e_pos, e_neg);
    use_neg = e_neg < e_pos;                                         // ties keep metadata 0 (+sv)
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    c[h] &= nonzero_nibbles(c[h]) | 0x77777777u;                     // a true zero is always code 0
    if (SV) {
      // only elements of the special value's sign take it (their code is at least 2 in magnitude, so the sign bit is there)
      const uint32_t t = take[h] & (use_neg ? c[h] : ~c[h]);
      c[h] = (c[h] & ~((t >> 3) * 15u)) | t;
    }
  }
  w0 = c[0], w1 = c[1];
  sbyte = (use_neg ? 0x80u : 0u) | scode;
}

// One launch for the whole of razer_quant_act, one thread per 16-element block.  When the tensor scale has to be
// computed (Eq. 1), the grid first takes the tensor maximum: every CTA folds its share into sync[0] and counts
// itself in sync[1], and all of them meet there (the launch is cooperative, so every CTA is resident; the wait is
// bounded all the same).  sync[] must be zero when the kernel starts; the last CTA to finish sets it back to zero.
// A thread keeps the first block it reads for the maximum, so inputs of up to one block per resident thread are read
// once; a single CTA needs no meeting through memory (and no cooperative launch).
// Inputs of TWO_LAUNCH_BLOCKS and more take two launches instead: act_amax_kernel leaves the maximum in sync[0] and its CTA count in
// the lower half of sync[1], and this kernel (amax_ctas > 0), resident early as a dependent launch and with its first block
// in registers, reads them when that one has completed.  Its CTAs count in the upper half; the last one clears sync[].  A lower
// half that is not the first kernel's CTA count gives away a scratch that was not zero.
// Where the quantizer writes: the interchange format (PREPARED = false), or the FP4 activation operand of the
// block-scaled tensor-core kernel (Fp4ActLayout: codes padded to KP columns with each word's nibbles in the packed
// order, scale bytes in scale-factor tile order; the padding is written as zeros by this kernel too).
struct QuantActOut {
  int M, k16, kp16, spt, m_pad;      // rows; 16-element blocks per row of the input / of the padded operand; stages; padded rows
};

// Maximum magnitude of a bf16 tensor, as its bit pattern, folded into sync[0]; NaNs are skipped (patterns above 0x7F80 count as
// zero).  Four independent loads a thread and turn.
__device__ __forceinline__ void fold_bf16_max(uint32_t& m2, const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t a = w[j] & 0x7FFF7FFFu;
    m2 = __vmaxu2(m2, a & ~__vcmpgtu2(a, 0x7F807F80u));
  }
}
__global__ void __launch_bounds__(256) act_amax_kernel(const uint4* __restrict__ x, long long n_vec, uint32_t* __restrict__ sync) {
  __shared__ uint32_t warp_max[8];
  grid_dep_wait();                                        // x and sync[] may belong to the preceding kernel
  grid_dep_launch();
  uint32_t m2 = 0;
  const long long stride = (long long)gridDim.x * 256;
  long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  for (; i + 3 * stride < n_vec; i += 4 * stride) {
    const uint4 v0 = x[i], v1 = x[i + stride], v2 = x[i + 2 * stride], v3 = x[i + 3 * stride];
    fold_bf16_max(m2, v0);
    fold_bf16_max(m2, v1);
    fold_bf16_max(m2, v2);
    fold_bf16_max(m2, v3);
  }
  for (; i < n_vec; i += stride) fold_bf16_max(m2, x[i]);
  const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, max(m2 & 0xFFFFu, m2 >> 16));
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t all = __reduce_max_sync(0xFFFFFFFFu, warp_max[threadIdx.x & 7]);
    if (threadIdx.x == 0) {
      if (all) atomicMax(&sync[0], all);
      atomicAdd(&sync[1], 1u);
    }
  }
}

template <bool SV, bool PREPARED>
__global__ void __launch_bounds__(256) quant_act_fused_kernel(const uint4* __restrict__ x, long long n_blocks, float sv_mag,
                                                             const float* __restrict__ scale_in, uint32_t* sync,
                                                             uint2* __restrict__ codes, uint8_t* __restrict__ scales,
                                                             float* __restrict__ scale_out, const QuantActOut o, uint32_t amax_ctas) {
  __shared__ uint32_t warp_max[8];
  __shared__ uint32_t amax_shared;
  const long long n_work = PREPARED ? (long long)o.m_pad * o.kp16 : n_blocks;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  // work item t -> (row, block of the row) of the padded operand, and whether the input has such a block
  auto locate = [&](long long t, int& m, int& kb) -> long long {
    m = (int)(n_work < (1ll << 31) ? (uint32_t)t / (uint32_t)o.kp16 : t / o.kp16);
    kb = (int)(t - (long long)m * o.kp16);
    return (m < o.M && kb < o.k16) ? (long long)m * o.k16 + kb : -1;
  };
  uint4 f0 = make_uint4(0, 0, 0, 0), f1 = f0;                          // this thread's first block
  float d32;
  if (scale_in) {
    d32 = *scale_in;
  } else {
    uint32_t m2 = 0;
    auto fold = [&](const uint4& v) { if (amax_ctas == 0) fold_bf16_max(m2, v); };
    if (PREPARED) {
      if (t0 < n_work) {
        int m, kb;
        const long long src = locate(t0, m, kb);
        if (src >= 0) { f0 = x[2 * src]; f1 = x[2 * src + 1]; }
      }
      // beyond the first item the maximum does not care about the padded order
      fold(f0);
      fold(f1);
      if (amax_ctas == 0 && n_work > stride)
        for (long long t = t0; t < n_blocks; t += stride) { fold(x[2 * t]); fold(x[2 * t + 1]); }
    } else {
      if (t0 < n_work) { f0 = x[2 * t0]; f1 = x[2 * t0 + 1]; }
      fold(f0);
      fold(f1);
      if (amax_ctas == 0)
        for (long long t = t0 + stride; t < n_work; t += stride) { fold(x[2 * t]); fold(x[2 * t + 1]); }
    }
    if (amax_ctas > 0) {
      grid_dep_wait();
      grid_dep_launch();                                               // only now: a matmul behind reads packed weights at once
      if (threadIdx.x == 0) {
        const uint32_t a = *(volatile uint32_t*)&sync[0];
        __threadfence();
        const uint32_t prev = atomicAdd(&sync[1], 0x10000u);
        const bool clean = (prev & 0xFFFFu) == amax_ctas;
        if (clean && (prev >> 16) == gridDim.x - 1) sync[0] = sync[1] = 0;   // everyone has read the maximum
        amax_shared = clean ? a : 0xFFFFFFFFu;
      }
      __syncthreads();
    } else {
      uint32_t m = max(m2 & 0xFFFFu, m2 >> 16);
      m = __reduce_max_sync(0xFFFFFFFFu, m);
      if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) m = max(m, warp_max[i]);
        if (gridDim.x > 1) {
          if (m) atomicMax(&sync[0], m);
          __threadfence();
          atomicAdd(&sync[1], 1u);
          // all CTAs are resident (cooperative launch); the bound only guards against a dirty sync[]
          uint32_t seen = 0;
          for (uint32_t spins = 0; spins < (1u << 22); ++spins) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(sync + 1) : "memory");
            if (seen >= gridDim.x) break;
            __nanosleep(32);
          }
          uint32_t a;
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(a) : "l"(sync) : "memory");
          m = seen >= gridDim.x ? a : 0xFFFFFFFFu;                       // gave up: flagged below with a NaN scale
        } else if (sync[0] | sync[1]) {
          m = 0xFFFFFFFFu;                                               // a scratch that was not zero
        }
        amax_shared = m;
      }
      __syncthreads();
    }
    const uint32_t bits = amax_shared;
    if (bits == 0xFFFFFFFFu) {
      if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = __uint_as_float(0x7FC00000u);
      return;
    }
    const float amax = __uint_as_float(bits << 16);
    d32 = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, __fmul_rn(448.0f, 6.0f));   // Eq. 1
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = d32;
  const float d32x6 = __fmul_rn(d32, 6.0f);
  for (long long t = t0; t < n_work; t += stride) {
    int m = 0, kb = 0;
    const long long src = PREPARED ? locate(t, m, kb) : t;
    uint4 v0 = f0, v1 = f1;
    if (t != t0 || scale_in) {
      v0 = v1 = make_uint4(0, 0, 0, 0);
      if (src >= 0) { v0 = x[2 * src]; v1 = x[2 * src + 1]; }
    }
    uint32_t w0, w1, sbyte;
    quant_act_block<SV, PREPARED>(v0, v1, d32, d32x6, sv_mag, w0, w1, sbyte);
    if (!PREPARED) {
      codes[t] = make_uint2(w0, w1);
      scales[t] = (uint8_t)sbyte;
    } else {
      // one thread per block of the PADDED operand: blocks beyond K and rows beyond M are zeros
      if (m < o.M) codes[t] = make_uint2(w0, w1);
      // scale-factor tile of (128-token tile, stage, chunk); inside it word 4 * (t % 32) + t / 32, byte = block of the
      // chunk: the four lanes of a chunk (kp16 is a multiple of 4) put their bytes together
      uint32_t sw = (sbyte & 0x7Fu) << (8 * (kb & 3));
      sw |= __shfl_xor_sync(0xFFFFFFFFu, sw, 1);
      sw |= __shfl_xor_sync(0xFFFFFFFFu, sw, 2);
      const int tile = m >> 7, tm = m & 127, step = kb >> 4, c = (kb >> 2) & 3;
      const size_t at = (((size_t)tile * o.spt + step) * 4 + c) * 512 + (size_t)((tm & 31) * 4 + (tm >> 5)) * 4;
      if ((kb & 3) == 0) *reinterpret_cast<uint32_t*>(scales + at) = sw;
    }
  }
  if (!scale_in && amax_ctas == 0 && gridDim.x > 1) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const uint32_t prev = atomicAdd(&sync[1], 1u);
      if (prev + 1 == 2 * gridDim.x) {                                 // everyone has read the maximum: leave sync[] clean
        sync[0] = 0;
        sync[1] = 0;
      }
    }
  }
}

// ------------------------------------------------------------------ offline weight quantizer (Sec. 4.2)
// The same procedure as the activation quantizer above with the weight format: FP32 input, the 6-bit E3M3
// block scale (codes 0..63 of the E4M3 grid, maximum 1.875) and four candidate special values
// +m0, +m1, -m0, -m1 in metadata order (meta = sign * 2 + select, bits 7:6 of the scale byte).

// Tensor maximum of |w| over FP32 input (Eq. 1 numerator); NaNs are skipped.  Four independent loads a thread and turn:
// one load in flight per thread left two thirds of the DRAM bandwidth idle.
__global__ void __launch_bounds__(256) weight_amax_kernel(const uint4* __restrict__ w, long long n_vec, uint32_t* __restrict__ amax_bits) {
  grid_dep_launch();                                      // the quantizer behind may become resident
  uint32_t m = 0;
  auto fold = [&](const uint4& v) {
    const uint32_t b[4] = {v.x & 0x7FFFFFFFu, v.y & 0x7FFFFFFFu, v.z & 0x7FFFFFFFu, v.w & 0x7FFFFFFFu};
#pragma unroll
    for (int j = 0; j < 4; ++j) m = max(m, (b[j] > 0x7F800000u) ? 0u : b[j]);
  };
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n_vec; i += 4 * stride) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = w[i + u * stride];
#pragma unroll
    for (int u = 0; u < 4; ++u) fold(v[u]);
  }
  for (; i < n_vec; i += stride) fold(w[i]);
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  __shared__ uint32_t warp_max[8];
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < 8; ++q) m = max(m, warp_max[q]);
    if (m) atomicMax(amax_bits, m);
  }
}

// Candidates of a block: four special values in metadata order that share the scale of Eq. 2 (block maximum -> 6), and,
// where AWARE, two with a scale of their own (block maximum -> |v|) for a special value beyond 6 whose sign is that of
// the block's first largest element.
// The plain procedure for a block of 16 * sub elements, one IEEE division per element and candidate (inputs that the short
// form cannot take).  Errors of the AWARE candidates are compared in the tensor's units, fl32(fl32(d * d) * e), d = the
// candidate's step.
template <bool AWARE>
__device__ __noinline__ uint32_t quant_weight_block_plain(const float4* __restrict__ src, int sub, float d32, float m0, float m1,
                                                          uint32_t remap_code, uint2* __restrict__ codes) {
  constexpr int NC = AWARE ? 6 : 4;
  const uint32_t other_zero = remap_code ^ 8u;
  const float mags[2] = {m0, m1};
  float bmax = 0.0f;
  uint32_t top_neg = 0;                                              // sign of the first largest element
  for (int q = 0; q < 4 * sub; ++q) {
    const float4 v = src[q];
    const float xv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (fabsf(xv[j]) > bmax) { bmax = fabsf(xv[j]); top_neg = __float_as_uint(xv[j]) >> 31; }
  }
  uint32_t sbyte = 0;
  float denom = 1.0f, sv = m0;
  if (bmax > 0.0f) {
    float cv[NC], cd[NC];
    uint32_t cs[NC], cm[NC];
    bool ok[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const float qmax = c < 4 ? 6.0f : mags[c - 4];
      const float tq = __fdiv_rn(bmax, __fmul_rn(d32, qmax));        // Eq. 2 argument
      uint32_t scode = round_to_e4m3(tq, 63u);
      if (scode == 0) scode = 1;                                     // keep a non-empty block alive
      cs[c] = scode;
      cd[c] = __fmul_rn(d32, scale_value(scode));
      cm[c] = c < 4 ? (uint32_t)c : (top_neg * 2u + (uint32_t)(c - 4));
      cv[c] = (cm[c] & 2u) ? -mags[cm[c] & 1u] : mags[cm[c] & 1u];
      ok[c] = c < 4 || mags[c - 4] > 6.0f;
    }
    float err[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) err[c] = 0.0f;
#pragma unroll 1
    for (int q = 0; q < 4 * sub; ++q) {
      const float4 v = src[q];
      const float xv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // the four standard candidates share the scale of Eq. 2, hence the scaled value and its FP4 rounding
        float xs = 0.0f, r = 0.0f, d_r = 0.0f;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (c >= 4 && !ok[c]) continue;
          if (c == 0 || c >= 4) {
            xs = __fdiv_rn(xv[j], cd[c]);                            // the scaled block of Eq. 6
            const uint32_t idx = round_to_fp4_idx(fabsf(xs));
            r = (__float_as_uint(xs) >> 31) ? -fp4_mag(idx) : fp4_mag(idx);
            d_r = fabsf(__fsub_rn(xs, r));
          }
          const bool tk = fabsf(__fsub_rn(xs, cv[c])) < d_r;         // strictly closer only
          const float d = __fsub_rn(tk ? cv[c] : r, xs);
          err[c] = __fadd_rn(err[c], __fmul_rn(d, d));               // ascending element order, no fusion
        }
      }
    }
    if (AWARE) {
#pragma unroll
      for (int c = 0; c < NC; ++c) err[c] = __fmul_rn(__fmul_rn(cd[c], cd[c]), err[c]);
    }
    int pick = 0;                                                    // first minimum: ties keep the earlier candidate
    float best = err[0];
#pragma unroll
    for (int c = 1; c < NC; ++c)
      if (ok[c] && err[c] < best) { best = err[c]; pick = c; }
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (c == pick) { sbyte = (cm[c] << 6) | cs[c]; denom = cd[c]; sv = cv[c]; }
  }
#pragma unroll 1
  for (int g = 0; g < sub; ++g) {
    uint32_t wd[2] = {other_zero * 0x11111111u, other_zero * 0x11111111u};
    if (bmax > 0.0f) {
      wd[0] = wd[1] = 0;
#pragma unroll 1
      for (int q = 0; q < 4; ++q) {
        const float4 v = src[4 * g + q];
        const float xv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float xs = __fdiv_rn(xv[j], denom);
          const uint32_t idx = round_to_fp4_idx(fabsf(xs));
          const uint32_t neg = __float_as_uint(xs) >> 31;
          const float r = neg ? -fp4_mag(idx) : fp4_mag(idx);
          const bool tk = fabsf(__fsub_rn(xs, sv)) < fabsf(__fsub_rn(xs, r));
          const uint32_t c = tk ? remap_code : (idx ? (idx | (neg << 3)) : other_zero);   // a true zero is always the other zero code
          const int e = 4 * q + j;
          wd[e >> 3] |= c << (4 * (e & 7));
        }
      }
    }
    codes[g] = make_uint2(wd[0], wd[1]);
  }
  return sbyte;
}

// Sixteen elements of a block in the short form, at one step: error sums (continued from group to group).
//   e_base: no special value; e[0], e[1]: +-m0, +-m1 (candidates of an inactive magnitude keep e_base)
// KEEP: the scaled elements replace xv, and take[i] receives bit 3 of the nibbles strictly closer to magnitude i than to FP4.
template <bool ON0, bool ON1, bool KEEP>
__device__ __forceinline__ void weight_errors(float (&xv)[16], float denom, float y, float m0, float m1, float& e_base, F2 (&e)[2],
                                              uint32_t (&take)[2][2]) {
  const F2 nd2 = f2(-denom, -denom), y2 = f2(y, y), minus_m0 = f2(-m0, -m0), minus_m1 = f2(-m1, -m1);
#pragma unroll
  for (int j = 0; j < 16; j += 2) {
    const F2 xs = div_f32(f2(xv[j], xv[j + 1]), nd2, y2);            // the scaled block of Eq. 6
    float x0, x1, q0, q1;
    split(xs, x0, x1);
    const bool neg0 = __float_as_uint(x0) >> 31, neg1 = __float_as_uint(x1) >> 31;
    const F2 a = abs2(xs), d_r = sub2(a, round_to_fp4(a)), q_r = mul2(d_r, d_r);
    split(q_r, q0, q1);
    if (!(ON0 && ON1)) e_base = __fadd_rn(__fadd_rn(e_base, q0), q1);   // ascending element order, no fusion
    bool t0, t1;
    if (ON0) {
      add_errors(e[0], q_r, special_error(a, d_r, minus_m0, t0, t1), neg0, neg1);
      if (KEEP && t0) take[0][j >> 3] |= 8u << (4 * (j & 7));
      if (KEEP && t1) take[0][j >> 3] |= 8u << (4 * ((j + 1) & 7));
    }
    if (ON1) {
      add_errors(e[1], q_r, special_error(a, d_r, minus_m1, t0, t1), neg0, neg1);
      if (KEEP && t0) take[1][j >> 3] |= 8u << (4 * (j & 7));
      if (KEEP && t1) take[1][j >> 3] |= 8u << (4 * ((j + 1) & 7));
    }
    if (KEEP) xv[j] = x0, xv[j + 1] = x1;
  }
}
// One candidate alone (AWARE): magnitude m on the elements whose sign bit is `sgn`.
__device__ __forceinline__ float weight_error_one(const float (&xv)[16], float denom, float y, float m, uint32_t sgn, float e) {
  const F2 nd2 = f2(-denom, -denom), y2 = f2(y, y), minus_m = f2(-m, -m);
#pragma unroll
  for (int j = 0; j < 16; j += 2) {
    const F2 xs = div_f32(f2(xv[j], xv[j + 1]), nd2, y2), a = abs2(xs), d_r = sub2(a, round_to_fp4(a));
    float x0, x1, r0, r1, s0, s1;
    split(xs, x0, x1);
    split(d_r, r0, r1);
    split(add2(a, minus_m), s0, s1);
    const bool t0 = fabsf(s0) < fabsf(r0) && (__float_as_uint(x0) >> 31) == sgn, t1 = fabsf(s1) < fabsf(r1) && (__float_as_uint(x1) >> 31) == sgn;
    const F2 d = f2(t0 ? s0 : r0, t1 ? s1 : r1);
    split(mul2(d, d), r0, r1);
    e = __fadd_rn(__fadd_rn(e, r0), r1);
  }
  return e;
}
// Codes of sixteen scaled elements, those in `take` (bit 3 of their nibbles) that have sign bit `sgn` to the special value.
__device__ __forceinline__ uint2 codes_of_scaled(const float (&xs)[16], const uint32_t (&take)[2], uint32_t sgn, uint32_t remap_code) {
  uint32_t c[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int b = 8 * h;
    uint32_t w = to_fp4x8(xs[b], xs[b + 1], xs[b + 2], xs[b + 3], xs[b + 4], xs[b + 5], xs[b + 6], xs[b + 7]);
    const uint32_t t = take[h] & (sgn ? w : ~w);                     // elements of the special value's sign only
    const uint32_t nz = nonzero_nibbles(w);
    w &= nz | 0x77777777u;                                           // a true zero is always the other zero code
    if (remap_code == 0u) w |= ~nz & 0x88888888u;
    w &= ~((t >> 3) * 15u);
    if (remap_code != 0u) w |= t;
    c[h] = w;
  }
  return make_uint2(c[0], c[1]);
}
// Codes of sixteen elements under the winning candidate (magnitude m, sign bit sgn).
__device__ __forceinline__ uint2 weight_codes(const float (&xv)[16], float denom, float y, float m, uint32_t sgn, uint32_t remap_code) {
  const F2 nd2 = f2(-denom, -denom), y2 = f2(y, y), minus_m = f2(-m, -m);
  float xs[16];
  uint32_t take[2] = {0, 0};
#pragma unroll
  for (int j = 0; j < 16; j += 2) {
    const F2 q = div_f32(f2(xv[j], xv[j + 1]), nd2, y2), a = abs2(q);
    split(q, xs[j], xs[j + 1]);
    float r0, r1, s0, s1;
    split(sub2(a, round_to_fp4(a)), r0, r1);
    split(add2(a, minus_m), s0, s1);
    if (fabsf(s0) < fabsf(r0)) take[j >> 3] |= 8u << (4 * (j & 7));
    if (fabsf(s1) < fabsf(r1)) take[j >> 3] |= 8u << (4 * ((j + 1) & 7));
  }
  return codes_of_scaled(xs, take, sgn, remap_code);
}

// Eight floats from a 16-byte aligned address, in one 32-byte load where the tensor is aligned to that (`wide`, uniform): a block
// of its own per thread makes every load of a warp touch 32 separate sectors, and halves fetched apart cost twice the requests
// (blocks of 32 to 128 elements: 140 us for 11008 x 4096, now 88; blocks of 16: 67, now 62).
__device__ __forceinline__ void load8(const float4* p, float* v, bool wide) {
  if (wide) {
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
  } else {
    const float4 a = p[0], b = p[1];
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  }
}

// One thread's scale block of `sub` groups of 16 elements (ONE: sub == 1, the block stays in registers from its maximum
// to its codes; larger blocks are walked three times); called by whole warps, `inside`: this thread has a block.  A magnitude beyond 6 can
// win an element only where the block's scaled maximum passes halfway between 6 and it, so a warp in which no block does skips its two
// candidates: their sums would equal those without a special value.
template <bool AWARE, bool ONE>
__device__ __forceinline__ void quant_weight_block(const float4* __restrict__ src, bool inside, int sub_arg, bool wide, float d32, float m0, float m1,
                                                   uint32_t remap_code, uint2* __restrict__ codes, uint8_t* __restrict__ scale) {
  const int sub = ONE ? 1 : sub_arg;
  const uint32_t other_zero = remap_code ^ 8u;
  const float d32x6 = __fmul_rn(d32, 6.0f);
  float xv[16];
  auto load = [&](int g) {
#pragma unroll
    for (int q = 0; q < 2; ++q) load8(src + 4 * g + 2 * q, xv + 8 * q, wide);
  };
  uint32_t mbits = 0;
#pragma unroll 1
  for (int g = 0; g < sub; ++g) {
    load(g);
#pragma unroll
    for (int j = 0; j < 16; ++j) mbits = max(mbits, __float_as_uint(xv[j]) & 0x7FFFFFFFu);
  }
  const float bmax = __uint_as_float(mbits);
  uint32_t scode = round_to_e4m3(__fdiv_rn(bmax, d32x6), 63u);       // Eq. 2
  if (scode == 0) scode = 1;                                         // keep a non-empty block alive
  float denom = __fmul_rn(d32, scale_value(scode));
  bool fast = inside && mbits > 0 && mbits < 0x7F800000u && short_form(bmax, denom);
  float own_denom[2] = {1.0f, 1.0f};
  uint32_t own_scode[2] = {1u, 1u};
  uint32_t top_neg = 0;
  if (AWARE) {
    bool found = false;                                              // sign of the first largest element
#pragma unroll 1
    for (int g = 0; g < sub; ++g) {
      if (!ONE) load(g);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const bool is_top = !found && (__float_as_uint(xv[j]) & 0x7FFFFFFFu) == mbits;
        if (is_top) { top_neg = __float_as_uint(xv[j]) >> 31; found = true; }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float m = i ? m1 : m0;
      uint32_t sc = round_to_e4m3(__fdiv_rn(bmax, __fmul_rn(d32, m)), 63u);
      if (sc == 0) sc = 1;
      own_scode[i] = sc;
      own_denom[i] = __fmul_rn(d32, scale_value(sc));
      fast = fast && short_form(bmax, own_denom[i]);
    }
  }
  const float y = __frcp_rn(denom);
  const float xmax = __fmul_rn(bmax, y) * 2.001f;
  const bool on0 = __any_sync(0xFFFFFFFFu, fast && (m0 < 6.0f || xmax > 6.0f + m0));
  const bool on1 = __any_sync(0xFFFFFFFFu, fast && (m1 < 6.0f || xmax > 6.0f + m1));
  if (!inside) return;
  if (!fast) {
    if (mbits == 0) {
      for (int g = 0; g < sub; ++g) codes[g] = make_uint2(other_zero * 0x11111111u, other_zero * 0x11111111u);
      *scale = 0;
    } else {
      *scale = (uint8_t)quant_weight_block_plain<AWARE>(src, sub, d32, m0, m1, remap_code, codes);
    }
    return;
  }
  float e_base = 0.0f;
  F2 e2[2] = {f2(0.0f, 0.0f), f2(0.0f, 0.0f)};
  uint32_t take[2][2] = {{0, 0}, {0, 0}};
  constexpr bool KEEP = ONE && !AWARE;
#pragma unroll 1
  for (int g = 0; g < sub; ++g) {
    if (!ONE) load(g);
    if (on0 && on1) weight_errors<true, true, KEEP>(xv, denom, y, m0, m1, e_base, e2, take);
    else if (on0) weight_errors<true, false, KEEP>(xv, denom, y, m0, m1, e_base, e2, take);
    else if (on1) weight_errors<false, true, KEEP>(xv, denom, y, m0, m1, e_base, e2, take);
    else weight_errors<false, false, KEEP>(xv, denom, y, m0, m1, e_base, e2, take);
  }
  float e[4];                                                        // metadata order: +m0, +m1, -m0, -m1
  split(e2[0], e[0], e[2]);
  split(e2[1], e[1], e[3]);
  if (!on0) e[0] = e[2] = e_base;
  if (!on1) e[1] = e[3] = e_base;
  if (AWARE) {
#pragma unroll
    for (int c = 0; c < 4; ++c) e[c] = __fmul_rn(__fmul_rn(denom, denom), e[c]);
  }
  uint32_t meta = 0;                                                 // first minimum: ties keep the earlier candidate
  float best = e[0];
#pragma unroll
  for (int c = 1; c < 4; ++c)
    if (e[c] < best) { best = e[c]; meta = c; }
  float y_win = y;
  if (AWARE) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float m = i ? m1 : m0;
      if (m > 6.0f) {
        const float d = own_denom[i], yo = __frcp_rn(d);
        float eo = 0.0f;
#pragma unroll 1
        for (int g = 0; g < sub; ++g) {
          if (!ONE) load(g);
          eo = weight_error_one(xv, d, yo, m, top_neg, eo);
        }
        eo = __fmul_rn(__fmul_rn(d, d), eo);
        if (eo < best) { best = eo; meta = top_neg * 2u + (uint32_t)i; scode = own_scode[i]; denom = d; y_win = yo; }
      }
    }
  }
  const float m_win = (meta & 1u) ? m1 : m0;
#pragma unroll 1
  for (int g = 0; g < sub; ++g) {
    if (!ONE) load(g);
    if (KEEP) {
      const uint32_t won[2] = {(meta & 1u) ? take[1][0] : take[0][0], (meta & 1u) ? take[1][1] : take[0][1]};
      *codes = codes_of_scaled(xv, won, meta >> 1, remap_code);
    } else {
      codes[g] = weight_codes(xv, denom, y_win, m_win, meta >> 1, remap_code);
    }
  }
  *scale = (uint8_t)((meta << 6) | scode);
}

// The grid runs from the end of the tensor to its start, the reverse of the maximum's order, so that the part of the input still in L2 is
// read first.
template <bool AWARE, bool ONE>
__global__ void __launch_bounds__(256, 4) quant_weight_kernel(const float4* __restrict__ w, long long n_blocks, int sub_arg, float m0, float m1,
                                                          uint32_t remap_code, const float* __restrict__ scale_in,
                                                          const uint32_t* __restrict__ amax_bits, uint2* __restrict__ codes,
                                                          uint8_t* __restrict__ scales, float* __restrict__ scale_out) {
  const int sub = ONE ? 1 : sub_arg;
  const bool wide = aligned32(w);
  float d32;
  if (scale_in) {
    d32 = *scale_in;
  } else {
    const float amax = __uint_as_float(*amax_bits);
    d32 = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, __fmul_rn(1.875f, 6.0f));   // Eq. 1
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = d32;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long turns = (n_blocks + stride - 1) / stride;
  for (long long turn = turns - 1; turn >= 0; --turn) {
    const long long t = turn * stride + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool inside = t < n_blocks;
    const long long at = inside ? t : 0;
    quant_weight_block<AWARE, ONE>(w + 4 * at * sub, inside, sub, wide, d32, m0, m1, remap_code, codes + at * sub, scales + at);
  }
}

// What follows gives the same result for the usual magnitudes (m0 halfway between two FP4 values, m1 beyond 6) by gains instead of error
// sums.
__device__ __forceinline__ float max_nan(float a, float b) {          // a NaN stays one
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ uint32_t to_e4m3(float t) {                // nearest, ties to even, saturating; t >= 0
  uint16_t v;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(v) : "f"(0.0f), "f"(t));
  return v & 0xFFu;
}
// What a special value m takes off a block's error is a sum over the elements that take it, and those lie in one interval, of half-width
// `half_width` around m0 or beyond lo1 = (6 + m1) / 2; an element at distance -t inside it gains k t.  That needs neither the rounded
// value nor the squares, so a thread's 16 elements cost half the instructions.  The decision is that of the FP32 sums in
// ascending order unless two candidates come within `delta`, more than all roundings of both ways together.  t is exact wherever its
// sign matters (a within a factor of two of m0, v0, v1 or m1), so the elements that take the special value are the same ones.
// SUB lanes share a block of 16 * SUB elements, so every block size reads its tensor once and alike.
//
// Blocks left undecided (candidates too close, scaled elements beyond quick_max, values that the short form cannot take) are put down by
// their warp and taken by quant_weight_block, a thread each, as soon as there are 32; a CTA's warps share out what is left at the end.
// Few blocks of continuous weights are, many of weights that lie on a coarse grid (FP8, INT8, INT4 checkpoints), and nearly all large blocks at
// a given scale a hundred times too small.
//
// Bound by instruction issue.  11008 x 4096 at a given scale, us in graph replays, quant_weight_kernel / this with undecided blocks walked
// one element at a time by their whole warp and blocks beyond 9.4 steps by the plain procedure / this:
//   blocks of 16: Student-t 61.3 / 43.6 / 42.8, rounded to bf16 61.4 / 54.4 / 44.6, FP8 grid 64.2 / 80.4 / 49.1, normal at 0.1 of its scale 94 / 255 / 64
//   blocks of 128: 94.7 / 57.4 / 54.0, 94.6 / 73.7 / 55.9, 114.0 / 157.7 / 83.8, 107 / 1645 / 78
// Blocks of 32 and more at 1e-3 of their scale and below (every code saturates) are slower by up to a third.  As many CTAs as are resident: the
// undecided blocks fill warps better than with 16 to an SM (bf16, blocks of 128: 63.8).
template <int SUB>
__global__ void __launch_bounds__(256, 4) quant_weight_quick_kernel(const float4* __restrict__ w, long long n_groups, float m0, float m1,
                                                                    float half_width, uint32_t remap_code, const float* scale_in,
                                                                    const uint32_t* amax_bits, uint2* __restrict__ codes,
                                                                    uint8_t* __restrict__ scales, float* __restrict__ scale_out) {
  constexpr int WARPS = 8;
  constexpr float quick_max = 8192.0f / (SUB * SUB);                   // further out `delta` passes usual differences
  __shared__ float2 steps[64];                                         // scale code -> step, its correctly rounded reciprocal
  __shared__ long long left[WARPS][64];                                // blocks left undecided, per warp
  __shared__ int n_left[WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool wide = aligned32(w);
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long turns = (n_groups + stride - 1) / stride;
  grid_dep_wait();                                                     // for the maximum
  // volatile: while this grid starts up the maximum is still being taken, so no load of it may move up or go by the constant cache
  float d32;
  if (scale_in) {
    d32 = *(volatile const float*)scale_in;
  } else {
    const float amax = __uint_as_float(*(volatile const uint32_t*)amax_bits);
    d32 = (amax == 0.0f) ? 1.0f : __fdiv_rn(amax, __fmul_rn(1.875f, 6.0f));   // Eq. 1
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = d32;
  const float d32x6 = __fmul_rn(d32, 6.0f);
  const bool usual = d32x6 > 1.0e-18f && d32x6 < 1.0e22f;              // some step is inside short_form's range
  const float inv6 = usual ? __frcp_rn(d32x6) : __uint_as_float(0x7FC00000u);
  if (threadIdx.x < 64) {
    const float d = __fmul_rn(d32, scale_value(threadIdx.x));
    steps[threadIdx.x] = make_float2(d, usual && short_form(0.0f, d) ? __frcp_rn(d) : __uint_as_float(0x7FC00000u));   // NaN: not this way
  }
  __syncthreads();
  const float k0 = 4.0f * half_width, k1 = 2.0f * (m1 - 6.0f), lo1 = 0.5f * (m1 + 6.0f);
  int count = 0;
  for (long long turn = turns - 1; turn >= -1; --turn) {                // the last one: what is left
    bool some = true;
    long long block = 0;
    if (turn >= 0) {
      const long long t = turn * stride + (long long)blockIdx.x * blockDim.x + threadIdx.x;
      const bool inside = t < n_groups;                                  // the same for all lanes of a block: n_groups and stride are multiples of SUB
      float xs[16];
#pragma unroll
      for (int q = 0; q < 2; ++q) load8(w + 4 * (inside ? t : 0) + 2 * q, xs + 8 * q, wide);
      float bmax = 0.0f;
#pragma unroll
      for (int j = 0; j < 16; j += 2) bmax = max3_nan(bmax, fabsf(xs[j]), fabsf(xs[j + 1]));
#pragma unroll
      for (int o = 1; o < SUB; o *= 2) bmax = max_nan(bmax, __shfl_xor_sync(0xFFFFFFFFu, bmax, o));
      // Eq. 2: the quotient, correctly rounded where the code is not 0 or 1 anyway (the correction of div_f32)
      float tq = bmax * inv6;
      tq = __fmaf_rn(__fmaf_rn(tq, -d32x6, bmax), inv6, tq);
      tq = __fmaf_rn(__fmaf_rn(tq, -d32x6, bmax), inv6, tq);
      const uint32_t scode = max(min(to_e4m3(tq), 63u), 1u);             // never 0: keep a non-empty block alive
      const float2 step = steps[scode];
      const float xmax = bmax * step.y;
      bool quick = inside && bmax < 1.0e30f && xmax <= quick_max;        // false for a NaN anywhere
      if (__any_sync(0xFFFFFFFFu, quick)) {
        const bool on1 = __any_sync(0xFFFFFFFFu, quick && xmax > 0.999f * lo1);
        const F2 nd2 = f2(-step.x, -step.x), y2 = f2(step.y, step.y);
        F2 sum0 = f2(0.0f, 0.0f), dif0 = sum0, sum1 = sum0, dif1 = sum0;   // gains / -K of all elements; of the positive less the negative ones
        float far = 0.0f;                                                // the squared distances beyond 6
        uint32_t c[2], take0[2], take1[2] = {0, 0};
        auto flip = [](float g, float x) { return __uint_as_float(__float_as_uint(g) ^ (__float_as_uint(x) & 0x80000000u)); };
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float* x = xs + 8 * h;
          float t0[8];
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            split(div_f32(f2(x[j], x[j + 1]), nd2, y2), x[j], x[j + 1]);   // the scaled block of Eq. 6
            t0[j] = fabsf(fabsf(x[j]) - m0) - half_width;
            t0[j + 1] = fabsf(fabsf(x[j + 1]) - m0) - half_width;
            const float g0 = fminf(t0[j], 0.0f), g1 = fminf(t0[j + 1], 0.0f);
            sum0 = add2(sum0, f2(g0, g1));
            dif0 = add2(dif0, f2(flip(g0, x[j]), flip(g1, x[j + 1])));
          }
          c[h] = to_fp4x8(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
          take0[h] = to_fp4x8(t0[0], t0[1], t0[2], t0[3], t0[4], t0[5], t0[6], t0[7]) & 0x88888888u;
        }
        if (on1) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float* x = xs + 8 * h;
            float t1[8];
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
              t1[j] = lo1 - fabsf(x[j]);
              t1[j + 1] = lo1 - fabsf(x[j + 1]);
              const float g0 = fminf(t1[j], 0.0f), g1 = fminf(t1[j + 1], 0.0f);
              sum1 = add2(sum1, f2(g0, g1));
              dif1 = add2(dif1, f2(flip(g0, x[j]), flip(g1, x[j + 1])));
            }
            take1[h] = to_fp4x8(t1[0], t1[1], t1[2], t1[3], t1[4], t1[5], t1[6], t1[7]) & 0x88888888u;
          }
          if (__any_sync(0xFFFFFFFFu, quick && xmax > 7.0f)) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float o = fmaxf(fabsf(xs[j]) - 6.0f, 0.0f);
              far += o * o;
            }
          }
        }
        auto gains = [&](F2 sum, F2 dif, float k, float& pos, float& neg) {
          float a, b, d, f;
          split(sum, a, b);
          split(dif, d, f);
          a += b;
          d += f;
#pragma unroll
          for (int o = 1; o < SUB; o *= 2) {
            a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
            d += __shfl_xor_sync(0xFFFFFFFFu, d, o);
          }
          pos = -0.5f * k * (a + d);
          neg = -0.5f * k * (a - d);
        };
        float gain[4] = {0.0f, 0.0f, 0.0f, 0.0f};                        // metadata order: +m0, +m1, -m0, -m1
        gains(sum0, dif0, k0, gain[0], gain[2]);
        uint32_t meta = gain[2] > gain[0] ? 2u : 0u;
        // How far roundings can bring two candidates together, n = 16 SUB elements, u = 2^-24.  No element up to 7 is further than 1 from FP4,
        // none up to 3.5 than 1/2, none up to 1.75 than 1/4: with the squares beyond 6 that bounds a block's error by E.  An FP32 sum of n
        // squares is off by less than (n + 2) u E; a gain, which is part of the error, by less than 15 u E (8 packed additions, the two
        // halves', three shuffles', the scale's, one of t itself).  Two of each: (2 n + 34) u E, at most 66 u E SUB = 3.94e-6 E SUB.
        const uint32_t from2 = (c[0] & 0x44444444u) | ((c[1] & 0x44444444u) >> 1), from4 = ((c[0] >> 1) & c[0] & 0x22222222u) | ((c[1] & (c[1] << 1) & 0x44444444u));
        float bound = 1.0f + 0.25f * (float)__popc(from2) + 0.75f * (float)__popc(from4) + far;
#pragma unroll
        for (int o = 1; o < SUB; o *= 2) bound += __shfl_xor_sync(0xFFFFFFFFu, bound, o);
        const float delta = bound * (SUB * 4.0e-6f);
        bool close = fabsf(gain[0] - gain[2]) <= delta && fmaxf(gain[0], gain[2]) > 0.0f;
        if (on1) {
          gains(sum1, dif1, k1, gain[1], gain[3]);
          const float top0 = fmaxf(gain[0], gain[2]), low0 = fminf(gain[0], gain[2]);
          const float top1 = fmaxf(gain[1], gain[3]), low1 = fminf(gain[1], gain[3]);
          const float top = fmaxf(top0, top1), second = fmaxf(fminf(top0, top1), top0 > top1 ? low0 : low1);
          close = top - second <= delta && top > 0.0f;
          if (top1 > top0) meta = gain[3] > gain[1] ? 3u : 1u;
        }
        quick = quick && !close;
        if (quick) {
          uint32_t out[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t v = c[h];
            const uint32_t taken = ((meta & 1u) ? take1[h] : take0[h]) & ((meta & 2u) ? v : ~v);   // elements of the special value's sign only
            const uint32_t nz = nonzero_nibbles(v);
            v &= nz | 0x77777777u;                                       // a true zero is always the other zero code
            if (remap_code == 0u) v |= ~nz & 0x88888888u;
            v &= ~((taken >> 3) * 15u);
            if (remap_code != 0u) v |= taken;
            out[h] = v;
          }
          codes[t] = make_uint2(out[0], out[1]);
          if (threadIdx.x % SUB == 0) scales[t / SUB] = (uint8_t)(bmax > 0.0f ? (meta << 6) | scode : 0u);
        }
      }
      const uint32_t undecided = __ballot_sync(0xFFFFFFFFu, inside && !quick && threadIdx.x % SUB == 0);
      if (!undecided) continue;
      if ((undecided >> lane) & 1u) left[warp][count + __popc(undecided & ((1u << lane) - 1u))] = t / SUB;
      count += __popc(undecided);
      __syncwarp();
      if (count < 32) continue;
      count -= 32;
      block = left[warp][count + lane];
    } else {
      if (lane == 0) n_left[warp] = count;
      if (!__syncthreads_or(count)) return;
      int at = threadIdx.x, from = 0;
      while (from < WARPS && at >= n_left[from]) at -= n_left[from++];
      some = from < WARPS;
      if (!__any_sync(0xFFFFFFFFu, some)) return;
      if (some) block = left[from][at];
    }
    // (the walking form for blocks of 16 too: the other one spills here)
    quant_weight_block<false, false>(w + 4 * SUB * block, some, SUB, wide, d32, m0, m1, remap_code, codes + SUB * block, scales + block);
    __syncwarp();
  }
}

int launch_quant_weight(const float* w, int N, int K, int block, int scale_aware, float m0, float m1, int remap_code,
                        const float* scale_in,
                        uint32_t* amax_scratch, uint8_t* codes, uint8_t* scales, float* scale_out, cudaStream_t st) {
  const int sub = block / 16;
  const long long n_blocks = (long long)N * (K / block);
  const long long n_vec = (long long)N * (K / 4);
  const int threads = 256;
  if (!scale_in) {
    RAZER_TRY(check_cuda(cudaMemsetAsync(amax_scratch, 0, sizeof(uint32_t), st), "amax memset"));
    const long long b = (n_vec + threads * 4 - 1) / (threads * 4);
    const int g2 = (int)(b < 1 ? 1 : (b > 148 * 8 ? 148 * 8 : b));
    weight_amax_kernel<<<g2, threads, 0, st>>>((const uint4*)w, n_vec, amax_scratch);
    count_launches(1);
    RAZER_TRY(check_cuda(cudaGetLastError(), "weight_amax_kernel launch"));
  }
  const bool halfway = m0 == 2.5f || m0 == 3.5f || m0 == 5.0f;         // between FP4 neighbours 2, 3 / 3, 4 / 4, 6
  if (!scale_aware && halfway && m1 > 6.0f) {
    const long long n_groups = n_blocks * sub, b = (n_groups + threads - 1) / threads;
    const int g = (int)(b < 1 ? 1 : (b > 148LL * 4 ? 148LL * 4 : b));    // as many as are resident
    auto kern = sub == 1 ? quant_weight_quick_kernel<1> : sub == 2 ? quant_weight_quick_kernel<2> : sub == 4 ? quant_weight_quick_kernel<4>
                                                                                                   : quant_weight_quick_kernel<8>;
    // dependent: with a maximum ahead it starts up while that drains
    return launch_dependent("quant_weight_quick_kernel launch", kern, g, threads, 0, st, (const float4*)w, n_groups, m0, m1,
                            m0 == 5.0f ? 0.5f : 0.25f, (uint32_t)remap_code, scale_in, (const uint32_t*)amax_scratch, (uint2*)codes, scales,
                            scale_out);
  }
  const long long b = (n_blocks + threads - 1) / threads;
  const int g = (int)(b < 1 ? 1 : (b > 148LL * 16 ? 148LL * 16 : b));
  auto kern = scale_aware ? (sub == 1 ? quant_weight_kernel<true, true> : quant_weight_kernel<true, false>)
                          : (sub == 1 ? quant_weight_kernel<false, true> : quant_weight_kernel<false, false>);
  kern<<<g, threads, 0, st>>>((const float4*)w, n_blocks, sub, m0, m1, (uint32_t)remap_code, scale_in, amax_scratch, (uint2*)codes,
                              scales, scale_out);
  count_launches(1);
  return check_cuda(cudaGetLastError(), "quant_weight_kernel launch");
}

// One cooperative launch or two dependent ones: a meeting of the whole grid costs more on the GPU (us, replayed: 256 x 8192 8.5 against
// 6.3 for the FP4 operand, 9.9 against 7.1 with a special value; 1000 x 4096 10.1 against 8.6; 64 x 8192 5.4 against 4.2), the second
// launch 1 us on the host.  Level for a caller that launches from the host at 128 x 8192 (7.8 against 8.0, and 256 x 8192 10.3
// against 7.8), where the line is drawn.
constexpr long long TWO_LAUNCH_BLOCKS = 65536;

template <bool SV, bool PREPARED>
static int launch_quant_act_any(const void* x, int M, int K, float sv_mag, const float* scale_in, uint32_t* sync_scratch,
                                uint8_t* codes, uint8_t* scales, float* scale_out, const QuantActOut& o, cudaStream_t st) {
  const long long n_blocks = (long long)M * (K / 16);
  const long long n_work = PREPARED ? (long long)o.m_pad * o.kp16 : n_blocks;
  const int threads = 256;
  auto kern = quant_act_fused_kernel<SV, PREPARED>;
  static int max_ctas = 0;                                             // CTAs that are resident together
  if (!max_ctas) {
    int dev = 0, sms = 0, per_sm = 0;
    RAZER_TRY(check_cuda(cudaGetDevice(&dev), "cudaGetDevice"));
    RAZER_TRY(check_cuda(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "cudaDeviceGetAttribute"));
    RAZER_TRY(check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0),
                         "cudaOccupancyMaxActiveBlocksPerMultiprocessor"));
    max_ctas = sms * (per_sm < 1 ? 1 : per_sm);
  }
  const long long b = (n_work + threads - 1) / threads;
  const int grid = (int)(b < 1 ? 1 : (b > max_ctas ? max_ctas : b));
  const bool two = !scale_in && grid > 1 && n_blocks >= TWO_LAUNCH_BLOCKS;
  if (two) {
    const long long n_vec = 2 * n_blocks, amax_ctas = std::min((n_vec + 4 * threads - 1) / (4 * threads), 8 * 148LL);
    RAZER_TRY(launch_dependent("act_amax_kernel launch", act_amax_kernel, amax_ctas, threads, 0, st, (const uint4*)x, n_vec, sync_scratch));
    return launch_dependent("quant_act_fused_kernel launch", kern, grid, threads, 0, st, (const uint4*)x, n_blocks, sv_mag, scale_in,
                            sync_scratch, (uint2*)codes, scales, scale_out, o, (uint32_t)amax_ctas);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = scale_in || grid == 1 ? 0 : 1;                        // the grid only meets when it computes the scale
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, (const uint4*)x, n_blocks, sv_mag, scale_in, sync_scratch, (uint2*)codes,
                                           scales, scale_out, o, 0u);
  count_launches(1);
  return check_cuda(e, "quant_act_fused_kernel launch");
}

int launch_quant_act(const void* x, int M, int K, float sv_mag, const float* scale_in,
                     uint32_t* sync_scratch, uint8_t* codes, uint8_t* scales, float* scale_out,
                     cudaStream_t st) {
  const QuantActOut o = {};
  if (sv_mag != 0.0f)
    return launch_quant_act_any<true, false>(x, M, K, sv_mag, scale_in, sync_scratch, codes, scales, scale_out, o, st);
  return launch_quant_act_any<false, false>(x, M, K, 0.0f, scale_in, sync_scratch, codes, scales, scale_out, o, st);
}

// Plain NVFP4 quantization (no special value) straight into the FP4 activation operand of the block-scaled kernel.
int launch_quant_act_fp4(const void* x, int M, int K, const float* scale_in, uint32_t* sync_scratch, void* act_fp4,
                         float* scale_out, cudaStream_t st) {
  const Fp4ActLayout L = make_fp4_act_layout(M, K);
  QuantActOut o;
  o.M = M;
  o.k16 = K / 16;
  o.kp16 = L.KP / 16;
  o.spt = L.spt;
  o.m_pad = L.tiles128 * 128;
  uint8_t* codes = (uint8_t*)act_fp4;
  return launch_quant_act_any<false, true>(x, M, K, 0.0f, scale_in, sync_scratch, codes, codes + L.codes_bytes, scale_out, o, st);
}

}  // namespace razer
