// Decode GEMV (M <= 8) against packed RaZeR weights for sm_100a: TMA-fed register-fragment kernel.
//
//   y[m, n] = bf16( ts * sum_k x[m, k] * D1[n, k] ),   D1 = block_scale * element (exact bf16)
//
// The path is bound by the decode of the 4.5-bit weights, so everything around the decode is kept off the decoding warps: one
// producer warp each moves packed weights and activations into a shared-memory ring with bulk copies (cp.async.bulk +
// mbarrier), two epilogue warps add the warps' partial sums, write y and run the cross-CTA combination, and the CW consumer
// warps only wait for a stage, decode their slice of it in registers and feed it to warp-level m16n8k16 MMAs as the A fragment
// (B fragment = the activation slice, 8 tokens along n; FP32 accumulators).  Sec. 4.3 of the paper describes this
// fragment-matched style for its weight-only kernel; App. E its partition.
//
// Decode: a table in shared memory maps a byte of the code word (two elements) and the block's special value to a bf16 pair; it
// holds a copy per lane, so that 32 random lookups never meet on a bank.  A pair costs one byte permute (which forms the
// address), one load and one multiply by the block scale, where isolating, shifting and blending it in registers
// (razer_decode.cuh) costs five and a quarter, two of them on the half-rate FMA pipe: 61 instructions per 16 weights came down to
// 47, and what binds is now the shared-memory pipe (14 wavefronts per warp and 16 weights a lane, 94 % of it busy while a launch
// streams).  Decoding an eighth to a half of the words in registers instead, to even the two out, measured 1 to 13 % slower;
// 20 or 24 consumer warps 6 to 10 %.
// Unit: SW * TM strips; a warp that takes more strips of a chunk (TM) reads its activation fragment less often.
// Each producer issues from one lane elected once: with the issue of both in one lane chosen by its index, a copy cost 200 to 300
// cycles of that warp, and at 8 tokens (10 copies a stage) the launch waited for the issue: 8 x 28672 x 8192 60.4 us, now 33.9.
// Measured (us, launches back to back, weights from HBM; before = register decode, two CTAs per SM): 1 x 28672 x 8192 37.6 ->
// 29.3, 4 x 28672 x 8192 38.9 -> 31.2, 8 x 4096 x 4096 7.0 -> 5.9, 7 x 3333 x 2064 5.9 -> 4.7, 1 x 11008 x 4096 10.3 -> 9.5,
// 1 x 1024 x 1024 2.5 -> 2.2.  Of a launch, 1 us is the release of the dependent launch, 0.6 to 1.3 the activations' way
// in, 0.5 the epilogue; the SMs end within 2 us of each other.
//
// Work: a unit is SW * TM strips of 16 weight rows over the whole of K; a slice is one unit x one 64-column chunk.
// A stage of the ring holds KW * SPW consecutive slices of one unit and the matching activation columns.  A CTA has an SM to
// itself (the tables are large); the CTAs of the next launch in the stream start as those of this one exit (programmatic
// dependent launch), fill their tables and rings and wait.  Two CTAs per SM, so that the next launch is resident
// earlier, would leave each a ring of 36 KB beside its tables.
// Partition (host, stream_plan): either every CTA takes whole units only, or every CTA takes q whole units
// and the remaining units are cut along K into equal slice ranges, one range per CTA, processed FIRST: a
// unit shared by several CTAs is combined through FP32 slots in the workspace by the last CTA to arrive (one
// counter per unit and epilogue warp, slots added in CTA order: a fixed summation order), which then happens in the shadow of
// the whole units that follow.  This is the stripe partition with a global reduction of Sec. 4.3 / App. E,
// arranged so that the reduction is off the critical path.
//
// Every wait is bounded: on expiry the thread records a code in the workspace status word and the CTA drains
// its copies and exits.
#include "razer_stream_common.cuh"

namespace razer {

namespace stream_path {

// Per-lane constants of the consumer's reads from a stage.
struct LaneView {
  uint32_t h0, h1;           // code words of rows g and g + 8 of block t (offset inside the warp's piece)
  uint32_t sc;               // the two scale bytes of those blocks
  uint32_t xo;               // the lane's 16 activation columns of token g (offset from the stage's first column)
  uint32_t row;              // lane * 4: the lane's copy in the tables
};

// Table reads: nothing writes the tables any more once a stage is decoded, so these may move freely.
extern __shared__ __align__(1024) uint8_t smem_raw[];
template <int OFF>
__device__ __forceinline__ uint32_t table32(uint32_t at) { return *reinterpret_cast<const uint32_t*>(smem_raw + OFF + at); }
// The two elements of byte B of a code word, times their block's scale.  `row` = lut | select bit (bit 7).
template <int B>
__device__ __forceinline__ uint32_t decode_byte(uint32_t w, uint32_t row, uint32_t scale) {
  return mul_bf16x2(table32<0>(__byte_perm(w, row, 0x7604 | (B << 4))), scale);
}

// One word of rows g and g + 8: eight elements each, two MMAs.  Bytes 0, 1 of a code word hold elements (0, 2) and (4, 6),
// bytes 2, 3 hold (1, 3) and (5, 7); the activations are paired alike.
__device__ __forceinline__ void word_step(float (&acc)[4], uint32_t w0, uint32_t w1, uint32_t r0, uint32_t r1, uint32_t s0, uint32_t s1,
                                          const uint32_t (&xq)[4]) {
  mma_16816(acc, decode_byte<0>(w0, r0, s0), decode_byte<0>(w1, r1, s1), decode_byte<2>(w0, r0, s0), decode_byte<2>(w1, r1, s1), xq[0], xq[1]);
  mma_16816(acc, decode_byte<1>(w0, r0, s0), decode_byte<1>(w1, r1, s1), decode_byte<3>(w0, r0, s0), decode_byte<3>(w1, r1, s1), xq[2], xq[3]);
}
// One strip (16 rows) of one slice: decode the lane's two blocks, four MMAs (into one accumulator: separate
// accumulators per MMA measured no faster).
template <int OFF>
__device__ __forceinline__ void strip_step(float (&acc)[4], uint32_t piece, const LaneView& v, const uint32_t (&xq)[2][4]) {
  const uint2 c0 = lds64_at<OFF>(piece + v.h0), c1 = lds64_at<OFF>(piece + v.h1);
  const uint32_t sb = lds16_at<OFF>(piece + v.sc);
  const uint32_t s0 = table32<LUT_BYTES>(((sb << 7) & 0x3F80u) | v.row), s1 = table32<LUT_BYTES>(((sb >> 1) & 0x3F80u) | v.row);
  const uint32_t r0 = (sb & 0x80u) | v.row, r1 = ((sb >> 8) & 0x80u) | v.row;
  word_step(acc, c0.x, c1.x, r0, r1, s0, s1, xq[0]);
  word_step(acc, c0.y, c1.y, r0, r1, s0, s1, xq[1]);
}

// The warp's slices J, J + 1, .. SPW - 1 of a stage (slice j is chunk c + j * KW): activation fragment, then decode
// + MMA for each of the unit's strips, fully unrolled with every shared-memory offset an immediate (a rolled
// loop over the slices, with or without loading a slice ahead, measured 6 to 15 % slower).
// CHECKED: the stage is the last of a segment and may hold fewer slices.
template <class C, int J, bool CHECKED>
__device__ __forceinline__ void slice_steps(float (&acc)[C::TM][4], uint32_t st, uint32_t xs, const LaneView& v, int c, int c1) {
  if constexpr (J < C::SPW) {
    constexpr int TM = C::TM, KW = C::KW;
    if (!CHECKED || c + J * KW < c1) {
      const uint4 xa = lds128_at<J * KW * 128>(xs + v.xo), xb = lds128_at<J * KW * 128 + 16>(xs + v.xo);
      const uint32_t xq[2][4] = {
          {__byte_perm(xa.x, xa.y, 0x5410), __byte_perm(xa.x, xa.y, 0x7632), __byte_perm(xa.z, xa.w, 0x5410), __byte_perm(xa.z, xa.w, 0x7632)},
          {__byte_perm(xb.x, xb.y, 0x5410), __byte_perm(xb.x, xb.y, 0x7632), __byte_perm(xb.z, xb.w, 0x5410), __byte_perm(xb.z, xb.w, 0x7632)}};
      constexpr int W = J * KW * PIECE_BYTES, S = C::STRIP_BYTES;
      strip_step<W>(acc[0], st, v, xq);
      if constexpr (TM >= 2) strip_step<W + S>(acc[1], st, v, xq);
      if constexpr (TM >= 4) {
        strip_step<W + 2 * S>(acc[2], st, v, xq);
        strip_step<W + 3 * S>(acc[3], st, v, xq);
      }
    }
    slice_steps<C, J + 1, CHECKED>(acc, st, xs, v, c, c1);
  }
}

template <class C>
__global__ void __launch_bounds__(THREADS, 1) razer_stream_kernel(const Args a) {
  constexpr int TM = C::TM, CPS = C::CPS, XS = C::XS, KW = C::KW, RED_STRIDE = C::RED_STRIDE;
  __shared__ uint32_t abort_word, never_set;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x;
  const Work work = make_work(a, b);

  // ---- dynamic shared memory: decode tables, barriers, partial sums, ring stages ----
  const uint32_t base = smem_addr(smem_raw);
  const uint32_t lut = base, scales = base + LUT_BYTES, fixed_at = scales + SCALES_BYTES;
  const uint32_t red_bytes = (uint32_t)(a.red_bufs * KW) * a.M * RED_STRIDE * 4u;
  const uint32_t ring = fixed_at + ((BAR_BYTES + red_bytes + 127u) & ~127u);
  const uint32_t stage_bytes = (uint32_t)C::W_BYTES + (uint32_t)a.M * XS;
  const int stages = min(MAX_STAGES, (int)((base + SMEM_BYTES - ring) / stage_bytes));
  auto stage_addr = [&](int s) -> uint32_t { return ring + (uint32_t)s * stage_bytes; };
  const uint32_t bar_full = fixed_at, bar_empty = bar_full + 8 * MAX_STAGES;
  const uint32_t bar_red_full = bar_empty + 8 * MAX_STAGES, bar_red_free = bar_red_full + 16;
  const uint32_t red = fixed_at + BAR_BYTES;                 // [red_bufs][KW][M][RED_STRIDE] floats
  volatile uint32_t* abort_flag = &abort_word;

  // ---- stage k of this CTA's work (k counts stages over all segments) is (segment, first chunk) ----
  const size_t strip_run = (size_t)a.kc * PIECE_BYTES;        // bytes of one strip's K run
  struct Walk { int seg_i, c, c1, unit, slot, phase; };
  auto walk_start = [&](Walk& w) {
    w.seg_i = 0; w.slot = 0; w.phase = 0; w.c = w.c1 = w.unit = 0;
    if (work.n_seg > 0) { const Seg s = work.seg(0); w.c = s.c0; w.c1 = s.c1; w.unit = s.unit; }
  };
  auto walk_next = [&](Walk& w) {
    w.c += CPS;
    if (w.c >= w.c1 && ++w.seg_i < work.n_seg) { const Seg s = work.seg(w.seg_i); w.c = s.c0; w.c1 = s.c1; w.unit = s.unit; }
    if (++w.slot == stages) { w.slot = 0; w.phase ^= 1; }
  };
  auto issue_w = [&](const Walk& w) {
    const uint32_t bar = bar_full + 8 * w.slot, wb = (uint32_t)min(CPS, w.c1 - w.c) * PIECE_BYTES;
    uint32_t dst = stage_addr(w.slot);
    mbar_expect_tx(bar, C::STRIPS * wb);
    const uint8_t* src = a.packed + (size_t)(w.unit * C::STRIPS) * strip_run + (size_t)w.c * PIECE_BYTES;
#pragma unroll
    for (int i = 0; i < C::STRIPS; ++i, src += strip_run, dst += C::STRIP_BYTES) bulk_copy_g2s(dst, src, wb, bar);
  };

  // ---- warp 0 sets up the barriers and sends out the first ring of weight copies before the CTA meets: they depend on
  // nothing, and the first HBM round trip is the longest wait of a short launch; the consumers fill the tables meanwhile ----
  Walk head;                                                  // warp 0: the next stage to issue
  int issued = 0;
  if (warp == 0) {
    walk_start(head);
    if (elect_one()) {
      abort_word = never_set = 0;
      for (int i = 0; i < MAX_STAGES; ++i) {
        mbar_init(bar_full + 8 * i, 2);
        mbar_init(bar_empty + 8 * i, CW);
      }
      for (int i = 0; i < 2; ++i) {
        mbar_init(bar_red_full + 8 * i, CW);
        mbar_init(bar_red_free + 8 * i, EW);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      if (stages >= 2)
        for (; issued < stages && head.seg_i < work.n_seg; ++issued, walk_next(head)) issue_w(head);
    }
  } else if (warp > EW && warp <= EW + CW) {
    const int tid = threadIdx.x - 32 * (EW + 1);
#pragma unroll 1
    for (int e = tid; e < 512 + 128; e += CW * 32) {
      uint32_t v, dst;
      if (e < 512) {                                          // [weight byte][special value]
        const float sv = (e & 1) ? a.sv1 : a.sv0;
        const uint32_t lo = __float_as_uint(packed_elem(((uint32_t)e >> 1) & 0xFu, sv)), hi = __float_as_uint(packed_elem((uint32_t)e >> 5, sv));
        v = __byte_perm(lo, hi, 0x7632);                      // elements have few significant bits: the upper halves are exact
        dst = lut + (uint32_t)e * 128;
      } else {
        const uint32_t c = (uint32_t)e - 512;                 // scale byte without the select bit: [negate | code]
        const float sc = scale_value(c & 0x3Fu);
        v = __byte_perm(__float_as_uint((c & PACKED_NEGATE) ? -sc : sc), 0, 0x3232);
        dst = scales + c * 128;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)                             // 32 lane copies; each lane starts elsewhere in its row
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(dst + (uint32_t)((j + lane) & 7) * 16), "r"(v) : "memory");
    }
  }
  grid_dep_launch();                                          // the next launch of the stream may become resident
  __syncthreads();
  if (stages < 2) {                                           // cannot happen with the sizes the host admits
    if (threadIdx.x == 0) { grid_dep_wait(); atomicCAS(a.status, 0u, 20u); show_status(a.status_host, 20u); }
    return;
  }

  auto fail = [&](uint32_t code) {
    *abort_flag = 1;
    grid_dep_wait();                                          // the status word lives in the (possibly shared) workspace
    atomicCAS(a.status, 0u, code);
    show_status(a.status_host, code);
  };

  if (warp == 0) {
    // ===================== weights: bulk copies into the ring.  One lane, elected once: the issuing code runs on uniform registers =====================
    if (elect_one()) {
      for (; head.seg_i < work.n_seg; ++issued, walk_next(head)) {
        if (!wait_phase(bar_empty + 8 * head.slot, (uint32_t)head.phase ^ 1u, abort_flag, 40)) { fail(1); break; }
        issue_w(head);
      }
      // Drain: copies still in flight must land before this CTA's shared memory is released.  Waiting for the
      // last `stages` issued stages covers everything that can still be in flight.
      int slot = 0, phase = 0;
      const int skip = issued > stages ? issued - stages : 0;
      for (int i = 0; i < issued; ++i) {
        if (i >= skip) wait_phase(bar_full + 8 * slot, (uint32_t)phase, &never_set, 100);
        if (++slot == stages) { slot = 0; phase ^= 1; }
      }
    }
  } else if (warp == EW + CW + 1) {
    // ===================== activations: bulk copies into the ring =====================
    grid_dep_wait();                                          // they may belong to the preceding kernel
    if (elect_one()) {
      Walk w;
      int k = 0;
      for (walk_start(w); w.seg_i < work.n_seg; ++k, walk_next(w)) {
        if (k >= stages && !wait_phase(bar_empty + 8 * w.slot, (uint32_t)w.phase ^ 1u, abort_flag, 40)) { fail(4); break; }
        const uint32_t bar = bar_full + 8 * w.slot;
        uint32_t dst = stage_addr(w.slot) + C::W_BYTES;
        const uint32_t full = (uint32_t)min(CPS, w.c1 - w.c) * 128u, bytes = min(full, (uint32_t)(a.K - w.c * CHUNK_K) * 2u);
        if (bytes < full) {
          // K ends inside the stage's last chunk: the columns beyond it multiply zero blocks, but must be finite.
          // Written before this thread's arrival on the barrier, which publishes them to the consumers.
          for (int m = 0; m < a.M; ++m)
            for (uint32_t o = bytes; o < full; o += 16) sts128_zero(dst + m * XS + o);   // K % 16 == 0: a multiple of 32
          fence_proxy_async();
        }
        mbar_expect_tx(bar, (uint32_t)a.M * bytes);
        const __nv_bfloat16* src = a.x + (size_t)w.c * CHUNK_K;
        for (int m = 0; m < a.M; ++m, src += a.K, dst += XS) bulk_copy_g2s(dst, src, bytes, bar);
      }
    }
  } else if (warp <= EW) {
    // ===================== epilogue warps: add the consumer warps' partial sums, write y, combine split units =====================
    grid_dep_wait();                                          // y, workspace and the scale scalar may belong to the preceding kernel
    if (b == 0 && warp == 1 && lane == 0 && a.status_host) show_status(a.status_host, *(volatile uint32_t*)a.status);   // what an earlier call left
    float ts = a.tensor_scale;
    if (a.extra_scale) ts *= *a.extra_scale;
    epilogue_loop<C>(a, work, b, warp - 1, lane, red, bar_red_full, bar_red_free, abort_flag, ts, fail);
  } else {
    // ===================== consumers: decode + MMA =====================
    const int cw = warp - 1 - EW, ks = cw % KW, sg = cw / KW;      // place among the chunks and among the strips
    // The activations of the first stages arrive only after the preceding kernel has finished; waiting for that
    // here (the producer has the weights in flight meanwhile) keeps it out of the bounded waits below.
    grid_dep_wait();
    const int g = lane >> 2, t = lane & 3;
    LaneView v;
    {
      const uint32_t slot = (uint32_t)(g ^ (4 * t));          // row g of block t; row g + 8 sits in slot ^ 8
      const uint32_t piece = (uint32_t)(sg * TM * C::STRIP_BYTES + ks * PIECE_BYTES);
      v.h0 = piece + t * 128 + slot * 8;
      v.h1 = piece + t * 128 + (slot ^ 8u) * 8;
      v.sc = piece + PIECE_CODE_BYTES + g * 8 + t * 2;
      // B-fragment column g is token g; a lane without a token reads the last token's columns instead: its
      // products land in accumulator columns that are never stored
      v.xo = (uint32_t)min(g, a.M - 1) * XS + ks * 128 + t * 32;
      v.row = (uint32_t)lane * 4;
    }
    const bool t_ok0 = 2 * t < a.M, t_ok1 = 2 * t + 1 < a.M;    // which of the lane's two accumulator columns are tokens
    float acc[TM][4];
#pragma unroll
    for (int tm = 0; tm < TM; ++tm)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[tm][j] = 0.0f;
    int slot = 0;
    uint32_t phase = 0;
    bool alive = true;
    for (int i = 0; alive && i < work.n_seg; ++i) {
      const Seg s = work.seg(i);
      // stages of CPS chunks; in a stage that starts at chunk c0 this warp's slices are chunks c0 + ks, c0 + ks + KW, ...
      const int n_full = (s.c1 - s.c0) / CPS;
      const bool ragged = (s.c1 - s.c0) % CPS != 0;
#pragma unroll 1
      for (int k = 0; k < n_full + (ragged ? 1 : 0); ++k) {
        if (!wait_phase(bar_full + 8 * slot, phase, abort_flag)) { fail(2); alive = false; }
        if (!__all_sync(0xFFFFFFFFu, alive)) { alive = false; break; }
        const uint32_t st = stage_addr(slot), xs = st + C::W_BYTES;
        if (k < n_full) slice_steps<C, 0, false>(acc, st, xs, v, 0, 0);
        else slice_steps<C, 0, true>(acc, st, xs, v, s.c0 + k * CPS + ks, s.c1);
        __syncwarp();                                         // every lane has read the stage
        if (lane == 0) mbar_arrive(bar_empty + 8 * slot);
        if (++slot == stages) { slot = 0; phase ^= 1u; }
      }
      if (!alive) break;
      // ---- end of a segment: leave this warp's partial sums for the epilogue warp ----
      const int buf = a.red_bufs == 2 ? i & 1 : 0;
      const uint32_t round = (uint32_t)(a.red_bufs == 2 ? i >> 1 : i);
      if (!wait_phase(bar_red_free + 8 * buf, (round & 1u) ^ 1u, abort_flag)) { fail(3); alive = false; }
      if (!__all_sync(0xFFFFFFFFu, alive)) { alive = false; break; }
      // element (token m, row r) of the warps at chunk place ks at ((buf * KW + ks) * M + m) * RED_STRIDE + r
      const uint32_t dst = red + (uint32_t)((buf * KW + ks) * a.M * RED_STRIDE + sg * TM * 16) * 4u;
#pragma unroll
      for (int tm = 0; tm < TM; ++tm) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int m = 2 * t + (j & 1), row = 16 * tm + 8 * (j >> 1) + g;
          if ((j & 1) ? t_ok1 : t_ok0)
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst + (uint32_t)(m * RED_STRIDE + row) * 4u), "f"(acc[tm][j]) : "memory");
          acc[tm][j] = 0.0f;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_red_full + 8 * buf);
    }
  }
  __syncthreads();
}

}  // namespace stream_path

static StreamPlan remembered_plan(const razer_desc* d, int M) {
  return remembered<StreamPlan>(d->N, d->K, M, 0, [&] { return stream_plan(d, M); });
}

bool gemv_stream_supported(const razer_desc* d, int M) {
  (void)d;
  return M >= 1 && M <= stream_path::MAX_M;
}

size_t gemv_stream_workspace_bytes(const razer_desc* d, int M) {
  const StreamPlan p = remembered_plan(d, M);
  return WS_ZERO_BYTES + p.slots_bytes;
}

template <int SW, int TM, int SPW>
static int launch_stream_cfg(const stream_path::Args& a, int grid, cudaStream_t st) {
  auto kern = stream_path::razer_stream_kernel<stream_path::Cfg<SW, TM, SPW>>;
  static bool attr_set = false;
  if (!attr_set) {
    RAZER_TRY(check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, stream_path::SMEM_BYTES),
                         "cudaFuncSetAttribute(max dynamic shared memory)"));
    attr_set = true;
  }
  return launch_dependent("razer_stream_kernel launch", kern, grid, stream_path::THREADS, stream_path::SMEM_BYTES, st, a);
}

int launch_gemv_stream(const razer_desc* d, const void* packed, const void* x, int M, float extra_scale,
                       const float* extra_scale_dev, void* y, void* ws, size_t ws_bytes, cudaStream_t st, uint32_t* status_host) {
  const StreamPlan p = remembered_plan(d, M);
  const size_t need = WS_ZERO_BYTES + p.slots_bytes;
  if (!ws || ws_bytes < need)
    return set_error(RAZER_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, ws_bytes);
  stream_path::Args a;
  a.packed = (const uint8_t*)packed;
  a.x = (const __nv_bfloat16*)x;
  a.y = (__nv_bfloat16*)y;
  a.status = (uint32_t*)ws;
  a.counters = (uint32_t*)((char*)ws + WS_STATUS_BYTES);
  a.slots = (float*)((char*)ws + WS_ZERO_BYTES);
  a.status_host = status_host;
  a.extra_scale = extra_scale_dev;
  a.N = d->N;
  a.K = d->K;
  a.kc = p.kc;
  a.M = M;
  a.red_bufs = p.red_bufs;
  a.units = p.units;
  a.whole_base = p.whole_base;
  a.whole_per_cta = p.whole_per_cta;
  a.rem_ctas = p.rem_ctas;
  a.pieces_per_unit = p.pieces_per_unit;
  a.sv0 = d->sv_mag[0];
  a.sv1 = d->sv_mag[1];
  a.tensor_scale = d->tensor_scale * extra_scale;
  switch (p.SW * 100 + p.TM * 10 + p.SPW) {
    case 111: return launch_stream_cfg<1, 1, 1>(a, p.grid, st);
    case 112: return launch_stream_cfg<1, 1, 2>(a, p.grid, st);
    case 121: return launch_stream_cfg<1, 2, 1>(a, p.grid, st);
    case 122: return launch_stream_cfg<1, 2, 2>(a, p.grid, st);
    case 141: return launch_stream_cfg<1, 4, 1>(a, p.grid, st);
    case 211: return launch_stream_cfg<2, 1, 1>(a, p.grid, st);
    case 212: return launch_stream_cfg<2, 1, 2>(a, p.grid, st);
    case 221: return launch_stream_cfg<2, 2, 1>(a, p.grid, st);
    default: return launch_stream_cfg<2, 2, 2>(a, p.grid, st);
  }
}

}  // namespace razer
