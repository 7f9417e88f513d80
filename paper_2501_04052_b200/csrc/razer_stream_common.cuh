// Declarations of the decode kernel (razer_gemv_stream.cu): configuration,
// kernel arguments, the list of a CTA's work segments, bounded barrier waits, shared-memory access helpers, the
// epilogue warp's loop and the host-side partition plan.
#pragma once

#include <cuda.h>
#include <algorithm>
#include <cstdlib>

#include "razer_common.cuh"
#include "razer_decode.cuh"
#include "razer_ptx.cuh"

namespace razer {

namespace stream_path {

constexpr int CW = 16;                              // consumer warps
constexpr int EW = 2;                               // epilogue warps, each with its half of a unit's outputs
constexpr int THREADS = 32 * (CW + EW + 2);         // + a producer warp each for weights and activations
constexpr int MAX_STAGES = 8;
constexpr int MAX_M = 8;
constexpr int LUT_BYTES = PAIR_TABLE_BYTES;         // [weight byte][special value][lane]: two elements as bf16x2 (here not times 2^-126)
constexpr int SCALES_BYTES = 128 * 32 * 4;                  // [scale byte without the select bit][lane]: +-scale as bf16x2
constexpr int MAX_ROWS = 64;
constexpr int SLOT_FLOATS = MAX_ROWS * MAX_M;       // one CTA's partial result of a unit
constexpr int SMEM_BYTES = 226 * 1024;              // one CTA per SM
constexpr int BAR_BYTES = (2 * MAX_STAGES + 4) * 8;

// SW x KW = CW consumer warps: SW side by side over the unit's strips (TM strips each), KW over its chunks; a warp takes
// SPW chunks of a stage.
template <int SW_, int TM_, int SPW_>
struct Cfg {
  static constexpr int SW = SW_, TM = TM_, SPW = SPW_, KW = CW / SW_;
  static constexpr int STRIPS = SW * TM, ROWS = 16 * STRIPS;
  static constexpr int CPS = KW * SPW;                     // chunks per stage
  static constexpr int STRIP_BYTES = CPS * PIECE_BYTES;    // one strip's pieces of a stage
  static constexpr int W_BYTES = STRIPS * STRIP_BYTES;     // weights of a stage
  static constexpr int XS = CPS * 128 + 16;                // bytes between tokens in a stage (16 mod 128: no bank conflicts)
  static constexpr int RED_STRIDE = ROWS + 4;              // floats per (warp, token) in the partial-sum buffers
  static_assert(XS % 16 == 0, "bulk copies land on 16-byte boundaries");
  static_assert(ROWS <= MAX_ROWS, "a unit's partial result fits its slot");
};

struct Args {
  const uint8_t* packed;
  const __nv_bfloat16* x;    // [M][K]
  __nv_bfloat16* y;          // [M][N]
  float* slots;              // [grid][2][SLOT_FLOATS]
  uint32_t* counters;        // [split unit][epilogue warp], zero between calls
  uint32_t* status;          // device status word
  uint32_t* status_host;     // the same for a host that waits for this call (pinned memory), or NULL
  const float* extra_scale;  // optional device scalar multiplied into the tensor scale
  int N, K, kc, M;
  int red_bufs;              // partial-sum buffers: 1 or 2
  int units;                 // units (Cfg::STRIPS strips) that hold rows < N
  int whole_base, whole_per_cta;   // CTA b owns the whole units whole_base + b * whole_per_cta .. (clipped to units)
  int rem_ctas;              // CTAs that share the split units [0, whole_base); 0 = nothing is split
  int pieces_per_unit;       // a split unit is cut along K into this many equal pieces; the pieces of all split units,
                             // in unit order, are dealt out to the rem_ctas CTAs in equal contiguous ranges
  float sv0, sv1, tensor_scale;
};

// D (+)= A(16 x 16, row) * B(16 x 8, col), bf16 inputs, FP32 accumulation.
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
template <int OFF>
__device__ __forceinline__ uint32_t lds16_at(uint32_t base) {
  uint32_t v;
  asm volatile("ld.shared.u16 %0, [%1+%2];" : "=r"(v) : "r"(base), "n"(OFF) : "memory");
  return v;
}
template <int OFF>
__device__ __forceinline__ uint2 lds64_at(uint32_t base) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(base), "n"(OFF) : "memory");
  return v;
}
template <int OFF>
__device__ __forceinline__ uint4 lds128_at(uint32_t base) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+%5];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(base), "n"(OFF)
               : "memory");
  return v;
}
__device__ __forceinline__ void sts128_zero(uint32_t addr) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(addr), "r"(0u) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// One segment of a CTA's work: chunks [c0, c1) of one unit.
struct Seg {
  int unit, c0, c1;
};

// A CTA's list of segments: its range of pieces of split units (at most two units), then its whole units.
struct Work {
  int n_rem, n_seg;
  int u0, a0, a1;            // first split segment: unit, chunk range
  int u1, b1;                // second split segment: unit, chunks [0, b1)
  int wu0;                   // first whole unit
  int kc;
  __device__ __forceinline__ Seg seg(int i) const {
    Seg s;
    if (i < n_rem) {
      if (i == 0) { s.unit = u0; s.c0 = a0; s.c1 = a1; }
      else { s.unit = u1; s.c0 = 0; s.c1 = b1; }
    } else {
      s.unit = wu0 + (i - n_rem);
      s.c0 = 0;
      s.c1 = kc;
    }
    return s;
  }
};

// Piece range of CTA c: pieces [P c / ctas, P (c + 1) / ctas) of the P = units * pieces_per_unit pieces
// (P * ctas stays far below 2^32: at most a few hundred units, eight pieces each, a few hundred CTAs).
__device__ __forceinline__ int piece_begin(const Args& a, int c) {
  const uint32_t P = (uint32_t)(a.whole_base * a.pieces_per_unit);
  if (P == (uint32_t)a.rem_ctas) return c;                   // one piece per CTA
  return (int)((P * (uint32_t)c) / (uint32_t)a.rem_ctas);
}
// CTA that owns piece i (the inverse of piece_begin).
__device__ __forceinline__ int cta_of_piece(const Args& a, int i) {
  const uint32_t P = (uint32_t)(a.whole_base * a.pieces_per_unit);
  if (P == (uint32_t)a.rem_ctas) return i;
  return (int)((((uint32_t)(i + 1) * (uint32_t)a.rem_ctas) - 1u) / P);
}

__device__ __forceinline__ Work make_work(const Args& a, int b) {
  Work w;
  w.kc = a.kc;
  w.n_rem = 0;
  w.u0 = w.a0 = w.a1 = w.u1 = w.b1 = 0;
  if (b < a.rem_ctas) {
    // piece j of a unit: chunks [kc j / p, kc (j + 1) / p)
    const int p = a.pieces_per_unit;
    const int i0 = piece_begin(a, b), i1 = piece_begin(a, b + 1);       // i1 > i0: there are at least as many pieces as CTAs
    w.u0 = i0 / p;
    w.u1 = (i1 - 1) / p;
    w.n_rem = w.u1 > w.u0 ? 2 : 1;
    w.a0 = (a.kc * (i0 - w.u0 * p)) / p;
    w.a1 = w.n_rem == 2 ? a.kc : (a.kc * (i1 - w.u0 * p)) / p;
    w.b1 = (a.kc * (i1 - w.u1 * p)) / p;
  }
  w.wu0 = a.whole_base + b * a.whole_per_cta;
  int n_whole = a.units - w.wu0;
  n_whole = n_whole < 0 ? 0 : (n_whole > a.whole_per_cta ? a.whole_per_cta : n_whole);
  w.n_seg = w.n_rem + n_whole;
  return w;
}

// Wait for a barrier phase.  One cheap poll first; the slow path looks at the clock and the abort flag only once
// per 32 polls and, for the service warps (sleep_ns > 0), sleeps between polls, so that a waiting warp costs the
// decoding warps few issue slots.
static __device__ __noinline__ bool wait_phase_slow(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t sleep_ns) {
  const uint64_t t0 = global_ns();
  for (uint32_t i = 0; i < (WAIT_LIMIT >> 5); ++i) {
#pragma unroll 1
    for (int j = 0; j < 32; ++j) {
      if (mbar_try_wait(bar, parity)) return true;
      if (sleep_ns > 0) __nanosleep(sleep_ns);
    }
    if (*abort_flag) return false;
    if (global_ns() - t0 > WAIT_LIMIT_NS) return false;
  }
  return false;
}
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t sleep_ns = 0) {
  if (mbar_try_wait(bar, parity)) return true;
  return wait_phase_slow(bar, parity, abort_flag, sleep_ns);
}

// An epilogue warp's loop over the CTA's segments: add the consumer warps' partial sums of its outputs of a segment in
// warp order, then either write y (whole unit) or publish the piece, count, and let the last arrival add the pieces in CTA
// order (the warps of a CTA count apart).  `ts` multiplies every output.  `fail(code)` records a wait that gave up.
template <class C, class Fail>
__device__ __forceinline__ void epilogue_loop(const Args& a, const Work& work, int b, int ew, int lane, uint32_t red,
                                              uint32_t bar_red_full, uint32_t bar_red_free, volatile uint32_t* abort_flag,
                                              float ts, Fail fail) {
  constexpr int ROWS = C::ROWS, KW = C::KW, RED_STRIDE = C::RED_STRIDE;
  constexpr int STEP = 32 * EW, PER_LANE = ROWS * MAX_M / STEP;
  const int outputs = ROWS * a.M;                           // output o = token (o / ROWS), row (o % ROWS)
  const int first = lane + 32 * ew;                         // this lane's outputs: first, first + STEP, ..
  for (int i = 0; i < work.n_seg; ++i) {
    const Seg s = work.seg(i);
    const uint32_t sleep_ns = min(256, 32 * ((s.c1 - s.c0) / C::CPS + 1));   // a stage takes the consumers several hundred ns
    const int buf = a.red_bufs == 2 ? i & 1 : 0;
    const bool got = wait_phase(bar_red_full + 8 * buf, (uint32_t)(a.red_bufs == 2 ? i >> 1 : i) & 1u, abort_flag, sleep_ns);
    if (!got) fail(10);
    if (!__all_sync(0xFFFFFFFFu, got)) break;
    float v[PER_LANE];
#pragma unroll
    for (int j = 0; j < PER_LANE; ++j) {
      const int o = first + STEP * j;
      float sum = 0.0f;
      if (o < outputs) {
        const int m = o / ROWS, row = o % ROWS;
        const uint32_t src = red + (uint32_t)((buf * KW * a.M + m) * RED_STRIDE + row) * 4u;
#pragma unroll
        for (int w = 0; w < KW; ++w) sum += __uint_as_float(lds32(src + (uint32_t)(w * a.M * RED_STRIDE) * 4u));   // warp order
      }
      v[j] = sum;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bar_red_free + 8 * buf);
    const int n0 = s.unit * ROWS;
    const bool whole = s.c0 == 0 && s.c1 == a.kc;
    if (whole) {
#pragma unroll
      for (int j = 0; j < PER_LANE; ++j) {
        const int o = first + STEP * j;
        if (o < outputs) {
          const int m = o / ROWS, n = n0 + o % ROWS;
          if (n < a.N) a.y[(size_t)m * a.N + n] = __float2bfloat16_rn(ts * v[j]);
        }
      }
      continue;
    }
    // ---- a piece of a split unit: publish, count, the last arrival adds the pieces in CTA order ----
    float* mine = a.slots + ((size_t)b * 2 + i) * SLOT_FLOATS;          // split segments come first: i is 0 or 1
#pragma unroll
    for (int j = 0; j < PER_LANE; ++j)
      if (first + STEP * j < outputs) mine[first + STEP * j] = v[j];
    __syncwarp();
    const int c_first = cta_of_piece(a, s.unit * a.pieces_per_unit);
    const int c_last = cta_of_piece(a, (s.unit + 1) * a.pieces_per_unit - 1);
    uint32_t* count = a.counters + EW * s.unit + ew;
    uint32_t last = 0;
    if (lane == 0) {
      uint32_t prev;
      // release: this warp's slot stores (ordered before by the warp barrier) become visible with the count;
      // acquire: the last arrival sees every earlier arrival's slot stores
      asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(prev) : "l"(count) : "memory");
      last = (prev + 1 == (uint32_t)(c_last - c_first + 1)) ? 1u : 0u;
      if (last) *count = 0;                     // leave the counter ready for the next call
    }
    last = __shfl_sync(0xFFFFFFFFu, last, 0);
    if (!last) continue;
    float acc[PER_LANE];
#pragma unroll
    for (int j = 0; j < PER_LANE; ++j) acc[j] = 0.0f;
    // CTA order (a fixed summation order); the loads of four CTAs' slots for two of the lane's outputs are in flight together.  (One
    // output after another, a unit of 64 rows and 8 tokens took eight round trips to L2 for every four CTAs: 8 x 2500 x 6992 in such
    // units 17.5 us, now 9.2; all eight outputs at once cost the decoding warps' code more than it gave, 1 x 28672 x 8192 29.6 -> 30.9.)
    for (int cb = c_first; cb <= c_last; cb += 4) {
      const float* src[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = min(cb + u, c_last);
        const int sl = piece_begin(a, c) / a.pieces_per_unit == s.unit ? 0 : 1;   // the unit is that CTA's first or second segment
        src[u] = a.slots + ((size_t)c * 2 + sl) * SLOT_FLOATS;
      }
#pragma unroll
      for (int j = 0; j < PER_LANE; j += 2) {
        if (first + STEP * j < outputs) {
          constexpr int LAST = PER_LANE - 1;
          const int o[2] = {first + STEP * j, min(first + STEP * min(j + 1, LAST), outputs - 1)};   // where there is no second one: any other
          float part[2][4];
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int u = 0; u < 4; ++u) part[i][u] = __ldcg(src[u] + o[i]);
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (cb + u <= c_last) {
              acc[j] += part[0][u];
              if (j < LAST) acc[j + 1] += part[1][u];
            }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < PER_LANE; ++j) {
      const int o = first + STEP * j;
      if (o < outputs) {
        const int m = o / ROWS, n = n0 + o % ROWS;
        if (n < a.N) a.y[(size_t)m * a.N + n] = __float2bfloat16_rn(ts * acc[j]);
      }
    }
  }
}

}  // namespace stream_path

// ------------------------------------------------------------------ host side
static inline int stream_sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
  }
  return n;
}

static inline int force_spw() {   // tuning aid
  static const int v = [] { const char* e = getenv("RAZER_STREAM_SPW"); return e ? atoi(e) : 0; }();
  return v;
}

struct StreamPlan {
  int SW, TM, SPW, grid, units, kc, red_bufs;
  int whole_base, whole_per_cta, rem_ctas, pieces_per_unit;
  double cost;
  size_t slots_bytes;
};

// One candidate: units of SW * TM strips; every CTA takes whole units only (split == false), or q whole units after a
// piece of one of the remaining units, each of which is cut along K into equal pieces (processed first, combined
// through the workspace).  The cost is about the busiest CTA's time in SM cycles.  A round (each consumer warp takes TM strips of one
// chunk) costs the shared-memory wavefronts of its loads, 23 per strip and 8 per chunk and warp, which is what the decode is
// bound by; a stage 400 more, a segment 450; the launch 200 for every strip of its first stage and, at its end, 5 for every
// partial sum that an epilogue lane adds.  Combining the parts of a unit costs the more the more outputs a lane has and the more CTAs
// share it; where whole units follow, units are cut only if it is over before they are.  (Fitted to 336 sizes timed in every unit
// shape, M 1 .. 8, N and K 256 .. 28672: the choice is within 1 % of the best of them in the mean, 11 % at worst.  Charged as 1700
// whatever its size, the combination made it 4 % and 67 %, and slower than the kernel that decoded in registers (last figure):
// 8 x 2500 x 6992 17.5 -> 7.1 us (11.7), 8 x 600 x 16000 11.0 -> 6.3 (8.1), 4 x 1024 x 11008 8.7 -> 6.1 (7.2), 8 x 1024 x 4096 7.5 -> 3.9 (6.7).)
constexpr double STAGE_COST = 400, SEGMENT_COST = 450, STRIP_COST = 200, SUM_COST = 5;
constexpr double SPLIT_COST = 100, COMBINE_COST = 1900, UNEVEN_COST = 300, TRIP_COST = 1400, OUTPUT_COST = 450;

static inline StreamPlan stream_candidate(const razer_desc* d, int M, int G, int SW, int TM, bool split) {
  using namespace stream_path;
  StreamPlan p;
  const Geometry g = make_geometry(d->N, d->K);
  const int strips = (d->N + STRIP_ROWS - 1) / STRIP_ROWS, KW = CW / SW;
  p.SW = SW;
  p.TM = TM;
  p.units = (strips + SW * TM - 1) / (SW * TM);
  p.kc = g.k_chunks;
  // two chunks per warp and stage where that leaves three stages in what a CTA has for its ring, and two partial-sum
  // buffers where that leaves as many
  const int red1 = KW * M * (16 * SW * TM + 4) * 4;
  const int ring = SMEM_BYTES - LUT_BYTES - SCALES_BYTES - BAR_BYTES - red1 - 128;
  const int stage1 = SW * TM * KW * PIECE_BYTES + M * (KW * 128 + 16);
  p.SPW = TM <= 2 && 6 * stage1 <= ring ? 2 : 1;
  if (force_spw() == 1 || (force_spw() == 2 && TM <= 2 && 4 * stage1 <= ring)) p.SPW = force_spw();
  const int stages = ring / (p.SPW * stage1);
  p.red_bufs = (ring - red1) / (p.SPW * stage1) >= std::min(stages, 3) ? 2 : 1;
  const int per_lane = (16 * SW * TM * M + 32 * EW - 1) / (32 * EW);   // outputs of an epilogue lane
  const double round = 16.0 * (23 * TM + 8) * (stages < 3 ? 1.3 : 1.0) + STAGE_COST / p.SPW, sums = SUM_COST * KW * per_lane;
  auto cycles = [&](int chunks) { return ((chunks + KW - 1) / KW) * round + SEGMENT_COST; };
  p.cost = STRIP_COST * SW * TM + sums;
  const int q = p.units / G, rem = p.units - q * G;
  if (split && rem > 0) {
    // pieces per unit: the count that costs the busiest CTA the least
    int best_p = 1;
    double best_cost = 0;
    const int max_p = std::max(1, std::min(8, p.kc / KW));              // a piece is at least one chunk per warp
    for (int pc = 1; pc <= max_p; ++pc) {
      const int pieces = rem * pc, ctas = std::min(G, pieces);
      const int most = (pieces + ctas - 1) / ctas;                      // pieces of the busiest CTA
      double c = cycles(most * ((p.kc + pc - 1) / pc)) + (most > 1 ? SEGMENT_COST : 0);
      if (pc > 1) {
        const bool even = pieces == ctas;                               // a piece per CTA
        const int parts = even ? pc : std::min(pc, (pc * ctas + pieces - 1) / pieces + 1);   // CTAs that share a unit
        const double combine = COMBINE_COST + (even ? 0 : UNEVEN_COST) + TRIP_COST * ((parts + 3) / 4) + OUTPUT_COST * per_lane + sums;
        if (q == 0) c += combine;
        else if (combine > q * cycles(p.kc)) continue;
      }
      if (pc == 1 || c < best_cost) { best_cost = c; best_p = pc; }
    }
    p.whole_base = rem;
    p.whole_per_cta = q;
    p.pieces_per_unit = best_p;
    p.rem_ctas = std::min(G, rem * best_p);
    p.grid = q > 0 ? G : p.rem_ctas;
    p.cost += q * cycles(p.kc) + best_cost + SPLIT_COST;
  } else {
    const int qa = (p.units + G - 1) / G;
    p.whole_base = 0;
    p.whole_per_cta = qa;
    p.pieces_per_unit = 1;
    p.rem_ctas = 0;
    p.grid = (p.units + qa - 1) / qa;
    p.cost += qa * cycles(p.kc);
  }
  p.slots_bytes = (size_t)G * 2 * SLOT_FLOATS * sizeof(float);
  return p;
}

// The cheapest candidate (one, two or four strips per unit, with or without a split).
static inline StreamPlan stream_plan(const razer_desc* d, int M) {
  using namespace stream_path;
  static const char force_split = [] { const char* e = getenv("RAZER_STREAM_SPLIT"); return e ? e[0] : '\0'; }();   // tuning aids
  static const char force_tm = [] { const char* e = getenv("RAZER_STREAM_TM"); return e ? e[0] : '\0'; }();
  static const char force_sw = [] { const char* e = getenv("RAZER_STREAM_SW"); return e ? e[0] : '\0'; }();
  const int G = stream_sm_count();
  StreamPlan best;
  bool have = false;
  for (int SW = 1; SW <= 2; ++SW) {
    if (force_sw && force_sw != '0' + SW) continue;
    for (int TM = 1; TM * SW <= 4; TM *= 2) {
      if (force_tm && force_tm != '0' + TM) continue;
      for (int split = 0; split <= 1; ++split) {
        if (force_split == '0' && split) continue;
        const StreamPlan c = stream_candidate(d, M, G, SW, TM, split != 0);
        if (force_split == '1' && !split && c.units % G != 0) continue;
        if (!have || c.cost < best.cost) { best = c; have = true; }
      }
    }
  }
  if (!have) best = stream_candidate(d, M, G, 1, 1, false);
  return best;
}

}  // namespace razer
