// Pieces shared by the tcgen05 matmul kernels: tcgen05 / TMEM instruction wrappers, the cursor over a CTA's
// stripe of work items, and the host helpers for tensor maps.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "razer_ptx.cuh"

namespace razer {

static inline size_t align256(size_t v) { return (v + 255) / 256 * 256; }

// ------------------------------------------------------------------ tcgen05 wrappers
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem], the shared-memory descriptor given as two 32-bit halves (only the low half changes
// from one MMA to the next) and the accumulate flag known at compile time.
template <bool ACCUMULATE>
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_desc_lo, uint32_t b_desc_hi,
                                           uint32_t idesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 bd;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "mov.b64 bd, {%2, %3};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], bd, %4, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "r"(b_desc_lo), "r"(b_desc_hi), "r"(idesc), "n"(ACCUMULATE ? 1 : 0)
      : "memory");
}
__device__ __forceinline__ void tc_st8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, "
      "%9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, "
      "%21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
      "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
      "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}

__device__ __forceinline__ int cta_of_item(long long item, int grid, long long total) {
  return (int)((((item + 1) * grid) - 1) / total);
}

// ------------------------------------------------------------------ end of a CTA's part of an output tile
// What both tcgen05 kernels do with the accumulator of a segment (the items of one output tile inside a CTA's stripe): a
// tile the CTA covers completely is scaled, rounded and stored; of a partial tile every CTA but the first publishes its
// part (FP32 slot in the workspace, then a release-add on the tile's counter, which is its first CTA's), and the CTA that holds the tile's FIRST
// items (for it the tile is the end of its stripe, for the others the beginning, so their parts were published long
// before) adds the parts in CTA order, a fixed summation order, and stores.
// A complete tile's accumulator goes into registers whole (rounded, two columns to a register) and is handed back to the
// MMAs before the stores.  Nothing here may spill: with all of the SM's memory configured as shared memory a spilled
// register is an L2 round trip (64 FP32 registers a thread, a few of them spilled, instead of 32 packed ones: 157
// against 118 us at 2048 x 8192 x 8192 on the FP4 kernel; 124 us with the stores before the hand-back).
struct EpilogueCtx {
  uint32_t bar_accfull, bar_accempty, bar_epi;   // barriers (shared-window addresses)
  uint32_t tmem;             // accumulator, with the warp's lane quarter
  int row, group;            // the thread's weight row inside the tile; which share of the columns
  bool leader;
};

// a: kernel arguments (y, slots, counters, g, M, token_tiles, steps_per_tile, total_items, split).  at_end: the segment reaches the
// end of its tile.  GROUPS sets of four warps share the columns in units of 16.  wait(barrier, parity, which) is a bounded
// wait of the whole warp, fail(which) records one that gave up: which = 0 accumulator, 1 rendezvous, 2 other CTAs.
// The tile's sum is spread over SETS sets of PER_SET accumulators, of which those in `live` hold something (set 0 does where SETS
// is 1).
template <int NT, int PER_SET, int SETS, int GROUPS, class KernelArgs, class Wait, class Fail>
__device__ __forceinline__ bool segment_epilogue(const KernelArgs& a, const EpilogueCtx& x, int tile, bool at_end, uint32_t live, float ts,
                                                 uint32_t seg, uint32_t& epi_phase, volatile uint32_t* abort_flag, Wait wait, Fail fail) {
  constexpr int UNITS = NT / 16, MAXC = 16 * ((UNITS + GROUPS - 1) / GROUPS);
  constexpr size_t SLOT = (size_t)NT * 128;                  // [NT / 4][128 rows][4] floats: a thread reads and writes 16 bytes at a time
  const int grid = gridDim.x, cta = blockIdx.x, spt = a.steps_per_tile;
  const int col_lo = 16 * ((x.group * UNITS) / GROUPS), n_cols = 16 * (((x.group + 1) * UNITS) / GROUPS) - col_lo;
  const int tile_begin = tile * spt;
  const bool complete = (int)((a.total_items * cta) / grid) <= tile_begin && at_end;
  const int rt = tile / a.token_tiles, m0 = (tile - rt * a.token_tiles) * NT + col_lo;
  const int valid = min(n_cols, a.M - m0);                   // columns that are tokens
  const int n_out = rt * 128 + x.row;
  __nv_bfloat16* dst = a.y + (size_t)m0 * a.g.N + n_out;
  // sixteen columns of the accumulator, summed over the accumulators used in turn
  auto load16 = [&](int c, float (&v)[16]) {
    uint32_t w[16];
    tc_ld16(x.tmem + col_lo + c, w);
    tc_wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = SETS == 1 || (live & 1u) ? __uint_as_float(w[j]) : 0.0f;
#pragma unroll
    for (int q = 1; q < SETS * PER_SET; ++q) {
      if (SETS > 1 && !((live >> (q / PER_SET)) & 1u)) continue;
      tc_ld16(x.tmem + q * NT + col_lo + c, w);
      tc_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] += __uint_as_float(w[j]);
    }
  };
  auto add16 = [](float (&v)[16], const float4 (&p)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[4 * j] += p[j].x;
      v[4 * j + 1] += p[j].y;
      v[4 * j + 2] += p[j].z;
      v[4 * j + 3] += p[j].w;
    }
  };
  if (complete) {
    if (!wait(x.bar_accfull, seg & 1u, 0)) return false;
    tc_fence_after();
    uint32_t packed[MAXC / 2];
#pragma unroll
    for (int c = 0; c < MAXC; c += 16) {
      if (c < n_cols) {
        float v[16];
        load16(c, v);
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          const __nv_bfloat162 p = __floats2bfloat162_rn(ts * v[j], ts * v[j + 1]);
          packed[(c + j) / 2] = *reinterpret_cast<const uint32_t*>(&p);
        }
      }
    }
    tc_fence_before();
    mbar_arrive(x.bar_accempty);
    if (n_out < a.g.N) {
#pragma unroll
      for (int j = 0; j < MAXC; ++j) {
        if (j < valid) *dst = __ushort_as_bfloat16((unsigned short)(packed[j / 2] >> (16 * (j & 1))));
        dst += a.g.N;
        asm volatile("" : "+l"(dst));                        // one running pointer, not MAXC addresses held ready
      }
    }
    return true;
  }
  if (NT >= 64 && a.split > 1) {                               // (narrower: one CTA adds the few columns faster than all meet again)
    // The tile's `split` CTAs all work on it at the same time and on nothing else: each finishes a share of the columns (units
    // of 16), so that publishing and adding up take (split - 1) / split of the tile per CTA instead of split - 1 tiles on one.
    // Measured beyond the items' own time, 256 columns: two CTAs 9.3 us with one of them finishing the tile, 5.4 so; eight 18
    // and 8.
    const int first = cta - cta % a.split, mine = cta - first;
    const int own_lo = (mine * UNITS) / a.split, own_hi = ((mine + 1) * UNITS) / a.split;
    const int m_tile = m0 - col_lo;                            // token of the tile's first column
    float4* base = reinterpret_cast<float4*>(a.slots) + x.row;
    if (!wait(x.bar_accfull, seg & 1u, 0)) return false;
    tc_fence_after();
#pragma unroll 1
    for (int u = x.group; u < UNITS; u += GROUPS) {
      if ((u >= own_lo && u < own_hi) || m_tile + 16 * u >= a.M) continue;
      float v[16];
      load16(16 * u - col_lo, v);
      float4* to = base + (size_t)cta * (SLOT / 4) + 4 * u * 128;
#pragma unroll
      for (int j = 0; j < 4; ++j) __stcg(to + j * 128, make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
    }
    mbar_arrive(x.bar_epi);                                    // every thread has stored its part
    if (!wait(x.bar_epi, epi_phase & 1u, 1)) return false;
    ++epi_phase;
    // release: the CTA's slot stores (ordered before this by the rendezvous) become visible with the count
    if (x.leader) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.counters + first) : "memory");
    // acquire: every counted CTA's slot stores are visible to this thread's loads below
    uint32_t seen = 0;
    const uint64_t t0 = global_ns();
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.counters + first) : "memory");
      if (seen >= (uint32_t)a.split || *abort_flag || global_ns() - t0 > WAIT_LIMIT_NS) break;
    }
    const bool ready = seen >= (uint32_t)a.split;
    if (!ready) fail(2);
    if (!__all_sync(0xFFFFFFFFu, ready)) return false;
#pragma unroll 1
    for (int u = own_lo + x.group; u < own_hi; u += GROUPS) {
      const int m = m_tile + 16 * u;
      if (m >= a.M) continue;
      float own[16], v[16];
      load16(16 * u - col_lo, own);
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = 0.0f;
      for (int c = first; c < first + a.split; c += 2) {       // ascending CTA order, two CTAs' slots in flight together
        float4 part[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            part[h][j] = (c + h < first + a.split && c + h != cta) ? __ldcg(base + (size_t)(c + h) * (SLOT / 4) + (4 * u + j) * 128)
                                                                  : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          add16(v, part[h]);
          if (c + h == cta) {
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += own[j];
          }
        }
      }
      __nv_bfloat16* to = a.y + (size_t)m * a.g.N + n_out;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (m + j < a.M && n_out < a.g.N) *to = __float2bfloat16_rn(ts * v[j]);
        to += a.g.N;
      }
    }
    tc_fence_before();
    mbar_arrive(x.bar_accempty);
    mbar_arrive(x.bar_epi);                                    // every thread has read the counter
    if (!wait(x.bar_epi, epi_phase & 1u, 1)) return false;
    ++epi_phase;
    // the last of the tile's CTAs to get here leaves the counter ready for the next call
    if (x.leader && atomicAdd(a.counters + first, 1u) == 2u * a.split - 1u) a.counters[first] = 0;
    return true;
  }
  const int c_first = cta_of_item(tile_begin, grid, a.total_items);
  const bool owner = cta == c_first;
  int c_last = c_first;
  if (owner) {
    // acquire: every counted CTA's slot stores are visible to this thread's loads below
    c_last = cta_of_item(tile_begin + spt - 1, grid, a.total_items);
    const uint32_t others = (uint32_t)(c_last - c_first);
    uint32_t seen = 0;
    const uint64_t t0 = global_ns();
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.counters + c_first) : "memory");
      if (seen >= others || *abort_flag || global_ns() - t0 > WAIT_LIMIT_NS) break;
      __nanosleep(100);
    }
    const bool ready = seen >= others;
    if (!ready) fail(2);
    if (!__all_sync(0xFFFFFFFFu, ready)) return false;
  }
  if (!wait(x.bar_accfull, seg & 1u, 0)) return false;
  tc_fence_after();
  float4* slots = reinterpret_cast<float4*>(a.slots) + (col_lo / 4) * 128 + x.row;
#pragma unroll 1
  for (int c = 0; c < n_cols; c += 16) {
    float v[16];
    load16(c, v);
    if (owner) {
      // ascending CTA order; the loads of two CTAs' slots are in flight together
      for (int cb = c_first + 1; cb <= c_last; cb += 2) {
        float4 part[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            part[u][j] = (cb + u <= c_last && c + 4 * j < valid) ? __ldcg(slots + (size_t)(cb + u) * (SLOT / 4) + (c / 4 + j) * 128)
                                                                 : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int u = 0; u < 2; ++u) add16(v, part[u]);
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (c + j < valid && n_out < a.g.N) *dst = __float2bfloat16_rn(ts * v[j]);
        dst += a.g.N;
      }
    } else {
      float4* mine = slots + (size_t)cta * (SLOT / 4);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (c + 4 * j < valid) __stcg(mine + (c / 4 + j) * 128, make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
    }
  }
  tc_fence_before();
  mbar_arrive(x.bar_accempty);
  mbar_arrive(x.bar_epi);                                    // every thread has read the counter / stored its part
  if (!wait(x.bar_epi, epi_phase & 1u, 1)) return false;
  ++epi_phase;
  if (x.leader) {
    if (owner) a.counters[cta] = 0;                          // leave the counter ready for the next call
    // release: the CTA's slot stores (ordered before this by the rendezvous) become visible with the count
    else asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.counters + c_first) : "memory");
  }
  return true;
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// What a token-tile width costs, in microseconds, fitted to sweeps over sizes, widths and grids (razer_gemm_umma.cu,
// razer_gemm_fp4.cu).  `start`: a launch, growing by `busy` with a CTA on every SM.  `chunk`: one 64-column chunk of a 128-row tile; it
// grows by `load` likewise.  `whole`: storing a tile; `cut`, `part`: combining one cut evenly among several CTAs, and each CTA of it;
// `stripe`: the two partial tiles of a stripe, `extra`: each CTA beyond three that shares one.  `late`: a grid of more than half of the
// SMs, whose successor cannot start up beside it (with several tiles to a CTA that start-up is not what is waited for); `spread`: the same with a tile or more to every CTA, the more of them there are.
struct TileCost { int NT, CH, CHX; bool table; float start, busy, chunk, load, whole, cut, part, stripe, extra, late, spread; };

// The cheapest grid for `tiles` output tiles of `steps` items: every tile on one CTA, every tile cut evenly among 2 .. 16 CTAs, or
// equal stripes on all SMs.  Returns the modelled time.
static inline float best_grid(const TileCost& t, long long tiles, int steps, int sms, int& grid) {
  float best = 0.0f;
  const long long total = tiles * steps;
  auto consider = [&](long long g, int tiles_per_cta, int cut) {            // whole tiles per CTA, or CTAs per tile, or stripes (0, 0)
    const float busy = (float)g / sms;
    float c = t.start + t.busy * busy + (float)((total + g - 1) / g * t.CH) * t.chunk * (1.0f + t.load * busy);
    if (2 * g > sms || tiles_per_cta > 1) c += t.late;
    if (tiles_per_cta > 0) {
      c += t.whole * (0.6f + 0.4f * tiles_per_cta) + (2 * g > sms ? t.spread * (busy - 0.5f) : 0.0f);
    } else if (cut > 0) {
      c += t.cut + t.part * cut;
    } else {
      const float per_cta = (float)total / g / steps, parts = 1.0f / per_cta + 1.0f;
      c += t.stripe + 0.4f * t.whole * per_cta + (parts > 3.0f ? (parts - 3.0f) * t.extra : 0.0f);
    }
    if (best == 0.0f || c < best) { best = c; grid = (int)g; }
  };
  if (tiles <= sms) {
    consider(tiles, 1, 0);
    for (int cut = 2; cut <= 16 && tiles * cut <= sms && cut <= steps; ++cut) consider(tiles * cut, 0, cut);
  } else {
    for (int q = (int)((tiles + sms - 1) / sms), n = 0; n < 2 && q <= 8; ++q, ++n)
      if (tiles % q == 0) consider(tiles / q, q, 0);
  }
  consider(total < sms ? total : sms, 0, 0);
  return best;
}

static inline int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
  }
  return n;
}

}  // namespace razer
