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
// D[tmem] (+)= A[tmem] * B[smem descriptor]
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Same with the shared-memory descriptor given as two 32-bit halves (only the low half changes
// from one MMA to the next) and the accumulate flag known at compile time.
template <bool ACCUMULATE>
__device__ __forceinline__ void tc_mma_ts2(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_desc_lo, uint32_t b_desc_hi,
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

// Position of a CTA inside its stripe of work items; advanced one item at a time so that
// the hot loops need no division.
struct ItemCursor {
  int tile, step;          // output tile and k-stage inside it
  int stage, phase;        // ring slot of the shared-memory stage and its parity
  int astage, aphase;      // ring slot of the TMEM A stage and its parity
  template <int STAGES, int ASTAGES>
  __device__ __forceinline__ void next(int steps_per_tile) {
    if (++step == steps_per_tile) { step = 0; ++tile; }
    if (++stage == STAGES) { stage = 0; phase ^= 1; }
    if (++astage == ASTAGES) { astage = 0; aphase ^= 1; }
  }
};

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

// a: kernel arguments (y, slots, counters, g, M, token_tiles, steps_per_tile, total_items).  at_end: the segment reaches the
// end of its tile.  GROUPS sets of four warps share the columns in units of 16.  wait(barrier, parity, which) is a bounded
// wait of the whole warp, fail(which) records one that gave up: which = 0 accumulator, 1 rendezvous, 2 other CTAs.
template <int NT, int NACC, int GROUPS, class KernelArgs, class Wait, class Fail>
__device__ __forceinline__ bool segment_epilogue(const KernelArgs& a, const EpilogueCtx& x, int tile, bool at_end, float ts, uint32_t seg,
                                                 uint32_t& epi_phase, volatile uint32_t* abort_flag, Wait wait, Fail fail) {
  constexpr int UNITS = NT / 16, MAXC = 16 * ((UNITS + GROUPS - 1) / GROUPS);
  constexpr size_t SLOT = (size_t)2 * NT * 128;
  const int grid = gridDim.x, cta = blockIdx.x, spt = a.steps_per_tile;
  const int col_lo = 16 * ((x.group * UNITS) / GROUPS), n_cols = 16 * (((x.group + 1) * UNITS) / GROUPS) - col_lo;
  const int tile_begin = tile * spt;
  const bool complete = (int)((a.total_items * cta) / grid) <= tile_begin && at_end;
  const int rt = tile / a.token_tiles, m0 = (tile - rt * a.token_tiles) * NT + col_lo;
  const int valid = min(n_cols, a.M - m0);                   // columns that are tokens
  const int n_out = rt * 128 + x.row;
  __nv_bfloat16* dst = a.y + (size_t)m0 * a.g.N + n_out;
  // sixteen columns of the accumulator, summed over the NACC accumulators used in turn
  auto load16 = [&](int c, float (&v)[16]) {
    uint32_t w[16];
    tc_ld16(x.tmem + col_lo + c, w);
    tc_wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(w[j]);
#pragma unroll
    for (int q = 1; q < NACC; ++q) {
      tc_ld16(x.tmem + q * NT + col_lo + c, w);
      tc_wait_ld();
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] += __uint_as_float(w[j]);
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
  float* mine = a.slots + (size_t)cta * SLOT + col_lo * 128 + x.row;
#pragma unroll 1
  for (int c = 0; c < n_cols; c += 16) {
    float v[16];
    load16(c, v);
    if (owner) {
      // ascending CTA order; the loads of two CTAs' slots are in flight together
      for (int cb = c_first + 1; cb <= c_last; cb += 2) {
        float part[2][16];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float* src = a.slots + (size_t)min(cb + u, c_last) * SLOT + (col_lo + c) * 128 + x.row;
#pragma unroll
          for (int j = 0; j < 16; ++j) part[u][j] = (cb + u <= c_last && c + j < valid) ? __ldcg(src + j * 128) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] += part[u][j];
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (c + j < valid && n_out < a.g.N) *dst = __float2bfloat16_rn(ts * v[j]);
        dst += a.g.N;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (c + j < valid) mine[(c + j) * 128] = v[j];
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
