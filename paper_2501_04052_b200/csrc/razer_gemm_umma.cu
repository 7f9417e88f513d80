// Tensor-core matmul against packed RaZeR weights for sm_100a (tcgen05 + TMEM + TMA).
//
//   y[m, n] = bf16( ts * sum_k x[m, k] * D1[n, k] ),   D1 = block_scale * element (exact bf16)
//
// Mapping onto the 5th-generation tensor core: the weight tile is the MMA's A operand
// (128 weight rows = 128 TMEM lanes), the activation tile is the B operand (NT tokens,
// K-major in shared memory, 128-byte swizzle, written by TMA), the accumulator D[128 x NT]
// lives in TMEM.  Weights never exist as bf16 in shared or global memory: TMA boxes bring the packed 4.5-bit chunks into
// shared memory, the "dequant" warps (thread = weight row) decode a chunk of 64 columns at a time, in registers or by table, and write
// the bf16 pairs straight into TMEM with tcgen05.st, and the MMA reads A from TMEM.
//
// Warp roles (96 + 32 * NDW threads): warp 0 = weight producer, warp 1 = TMEM owner + MMA issuer, warps 2 .. 1 + NDW = dequant
// and epilogue, the last = activation producer.  A warp reaches only the TMEM lanes 32 * (warp % 4) .. + 31; four warps form a
// group that decodes an item, and the groups take the items in turn.
//
// Both decodes are described in razer_decode.cuh.  Up to 32 tokens by table where a launch is long enough (make_plan): 16 x 8192 x 28672 41.3 (registers) -> 36.0 us, 16 x 4096 x 11008
// 14.2 -> 13.1, 32 x 28672 x 8192 43.2 -> 38.7.  From 64 tokens on in registers: the table takes 64 KB from the rings, and its loads
// meet the activations' in shared memory (64 x 8192 x 28672 45.3 us in registers, 49.7 by table, 48 half and half).
//
// What bounds it: up to 32 tokens shared memory (270 wavefronts a chunk of about 305 cycles, copies and MMAs counted from the layout)
// and issue (214 of 305 slots), then the decode (about 3.4 instructions a weight) up to 128 tokens, from there on the MMAs (512 cycles
// per 128 x 256 x 64) together with shared-memory bandwidth (571 cycles), and the combination of cut tiles.  Device times on B200, first for one
// ring of weights and activations and items of one chunk at 256 tokens, then for rings apart, two-chunk items and groups that
// walk only their own items: 2048 x 14336 x 4096 204 -> 171 us (149 with the decode left out), 256 x 8192 x 8192 38.4 -> 32.7,
// 64 x 8192 x 28672 50.1 -> 45.0, 16 x 8192 x 28672 45.7 -> 40.8.  At 16 tokens, decoded in registers: half-item operand stages, two
// to a group, 45.7 us (the MMA warp's waits double), all groups on one item with two stages 44.3, four groups with items of three
// chunks 44.7 (by table 41.8), without the MMAs 40.4; the chunk loop rolled, by table, 44.5.  In a prefill the tensor pipe is active
// 81 % of a CTA's cycles; the shared-memory figure is counted from the layout.
//
// Work partition (Sec. 4.3 / App. E of the paper: stripes of about equal length that may span
// several output tiles, partial results reduced through global memory): the grid is
// persistent, work items are (output tile, k-stage) pairs in tile-major order and every CTA
// takes one contiguous stripe of items; the host picks the grid (make_plan), so that a stripe is whole tiles, an even share of
// one tile, or neither.  A stripe's first and last tile may be partial: razer_tcgen05.cuh says how those are combined.  Tiles a
// stripe covers completely are written directly.
//
// Every wait (mbarrier, counter) is bounded: on expiry the thread records a code in the
// workspace status word and the kernel drains and exits instead of hanging the GPU.
#include <cuda.h>
#include <cstdlib>

#include "razer_common.cuh"
#include "razer_decode.cuh"
#include "razer_ptx.cuh"
#include "razer_tcgen05.cuh"

namespace razer {

// Instruction descriptor: bf16 x bf16 -> f32, both operands K-major, M = 128, N = NT.
__host__ __device__ constexpr uint32_t make_idesc(int nt) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(nt >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// ------------------------------------------------------------------ kernel
struct UmmaArgs {
  __nv_bfloat16* y;
  float* slots;              // [grid] FP32 partial tiles of NT x 128
  uint32_t* counters;        // one per CTA: that of the partial tile it finishes; zero between calls
  uint32_t* status;          // device status word
  uint32_t* status_host;     // the same for a host that waits for this call (pinned memory), or NULL
  const float* extra_scale;  // optional device scalar multiplied into the tensor scale
  Geometry g;
  uint32_t svp0, svp1;       // special-value pairs for select 0 / 1 (razer_decode.cuh)
  float tensor_scale;
  uint32_t mul_lo, mul_hi;   // 2^6 + 2^12 and 2^2 + 2^8, passed at run time so that they stay multiplies
  int M, token_tiles, steps_per_tile;
  int x_map_3d;              // the activation tensor map is the 3-D (64 k, tokens, k chunk) view: one load per stage
  int split;                 // > 1: every tile is cut evenly among this many CTAs (grid = tiles x split)
  long long total_items;
};


// Rings: packed weights (WST stages, released by the dequant warps as soon as they have read one), activations (XST stages,
// released by the MMAs), decoded weights in TMEM (AST stages).  Apart from one another, so that the decode can run ahead of the
// MMAs by all of AST: with weights and activations in one ring it could start on an item only once the MMAs of the item
// a ring's length before had completed and both operands had been loaded again.  A work item is CH chunks, an activation
// stage CHX of them: every item costs a group two barrier waits, a drained TMEM store and its bookkeeping, so items of one
// chunk decode about a quarter slower than items of four, while activation boxes of 256 tokens fit only singly.
template <int NT, int CH, int CHX, int WST, int XST, int AST, int NDW, int NACC, bool TABLE>
struct UmmaCfg {
  static constexpr int GROUPS = NDW / 4;                       // four warps (all TMEM lane quarters) decode one item together
  static constexpr int THREADS = 64 + 32 * NDW + 32;           // + W producer, MMA warp, X producer
  static constexpr int W_BYTES = CH * CHUNK_BYTES;
  static constexpr int X_BOX_BYTES = NT * 128;                 // NT tokens x 64 k x 2 B
  static constexpr int X_BYTES = CHX * X_BOX_BYTES;
  static constexpr int ACC_COLS = NACC * NT < 32 ? 32 : NACC * NT;   // NACC accumulators, used round robin
  // More than two accumulators: a set for each operand slot, so that an item's products meet only those of every AST-th item.  The
  // tensor core's FP32 additions truncate, and their error grows with the length of a chain: with six accumulators instead of
  // two, which 16 tokens leave TMEM for, it is a third (16 x 8192 x 28672: 3.7e-9 of |x||w| instead of 1.24e-8, outputs off the
  // correctly rounded value 5 in 10^4 instead of 15), at 42.3 instead of 41.8 us a pass.
  static constexpr int SETS = NACC > 2 ? AST : 1, PER_SET = NACC / SETS;
  static constexpr int A_STAGE_COLS = CH * 32;                 // 4 blocks x 8 columns per chunk
  static constexpr int TMEM_COLS_NEEDED = ACC_COLS + AST * A_STAGE_COLS;
  static constexpr int TMEM_COLS = TMEM_COLS_NEEDED <= 64 ? 64 : TMEM_COLS_NEEDED <= 128 ? 128
                                   : TMEM_COLS_NEEDED <= 256 ? 256 : 512;
  static constexpr int NUM_BARS = 2 * (WST + XST + AST) + 4;
  static constexpr int PAIR_BYTES = TABLE ? PAIR_TABLE_BYTES : 0;   // at the start of shared memory
  static constexpr int TABLE_BYTES = DECODE_TABLE_BYTES;        // scale table
  static constexpr size_t SMEM_BYTES =
      1024 /*alignment slack*/ + PAIR_BYTES + (size_t)XST * X_BYTES + (size_t)WST * W_BYTES + NUM_BARS * 8 + 16 + 64 + TABLE_BYTES;
  static_assert(TMEM_COLS_NEEDED <= 512, "TMEM budget exceeded");
  static_assert(SMEM_BYTES <= 232448, "shared memory budget exceeded");
  static_assert(CH % CHX == 0, "an item is whole activation stages");
  static_assert(NACC % SETS == 0 && PER_SET <= 4, "a set is within an item's first chunk, which every item has");
  static_assert(NT % 16 == 0 && NT >= 16 && NT <= 256, "UMMA N for M = 128");
  // A parity wait is only sound for a waiter that knows the barrier's previous phase to be complete.  The groups take the
  // items in turn, so a stage has to come round to the same group every time: then that group has seen all its phases.
  static_assert(NDW % 4 == 0 && WST % GROUPS == 0 && AST % GROUPS == 0, "a stage always serves the same group");
};

template <int STAGES>
struct Ring {
  int slot = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next() {
    if (++slot == STAGES) { slot = 0; phase ^= 1u; }
  }
};

extern __shared__ __align__(1024) uint8_t umma_smem[];      // a link-time address: the pair table is indexed from it without an addition

// The MMA warp issues every item's MMAs.  (Letting the group that decoded an item issue it, once level at 16 tokens, lost
// when the MMA warp came to elect its lane once: 8192 x 28672 at 16 tokens 49.3 against 45.9 us.)
template <int NT, int CH, int CHX, int WST, int XST, int AST, int NDW, int NACC, bool TABLE>
__global__ void __launch_bounds__(96 + 32 * NDW, 1)
razer_umma_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                  const __grid_constant__ UmmaArgs a) {
  using Cfg = UmmaCfg<NT, CH, CHX, WST, XST, AST, NDW, NACC, TABLE>;
  constexpr int GROUPS = Cfg::GROUPS;
  constexpr int X_WARP = 2 + NDW;                       // the activation producer
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(umma_smem) + Cfg::PAIR_BYTES + 1023) & ~(uintptr_t)1023);
  const uint32_t smem_x = smem_u32(smem), smem_w = smem_x + XST * Cfg::X_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)XST * Cfg::X_BYTES + (size_t)WST * Cfg::W_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(        // 16-byte aligned: the table behind it is written as uint4
      (reinterpret_cast<uintptr_t>(bars + Cfg::NUM_BARS) + 15) & ~(uintptr_t)15);
  volatile uint32_t* abort_flag = tmem_slot + 1;
  uint8_t* tables = reinterpret_cast<uint8_t*>(tmem_slot + 16);   // decode table (razer_decode.cuh)

  const uint32_t bar_wfull = smem_u32(bars);            // [WST] TMA -> dequant
  const uint32_t bar_wempty = bar_wfull + 8 * WST;      // [WST] dequant -> TMA
  const uint32_t bar_xfull = bar_wempty + 8 * WST;      // [XST] TMA -> MMA
  const uint32_t bar_xempty = bar_xfull + 8 * XST;      // [XST] MMA commit -> TMA
  const uint32_t bar_afull = bar_xempty + 8 * XST;      // [AST] dequant -> MMA
  const uint32_t bar_aempty = bar_afull + 8 * AST;      // [AST] MMA commit -> dequant
  const uint32_t bar_accfull = bar_aempty + 8 * AST;
  const uint32_t bar_accempty = bar_accfull + 8;
  const uint32_t bar_epi = bar_accempty + 8;            // rendezvous of the epilogue threads
  const uint32_t bar_drain = bar_epi + 8;               // the MMA warp's own MMAs have all completed

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grid = gridDim.x, cta = blockIdx.x;
  const int it_begin = (int)((a.total_items * cta) / grid);
  const int it_end = (int)((a.total_items * (cta + 1)) / grid);
  const int n_items = it_end - it_begin;
  const int spt = a.steps_per_tile;
  int tile = it_begin / spt, step = it_begin - tile * spt;   // the item at hand
  const int last_tile = (it_end - 1) / spt;                   // tile of the CTA's last item
  auto next_item = [&]() {
    if (++step == spt) { step = 0; ++tile; }
  };

  if (threadIdx.x == 0) {
    for (int i = 0; i < WST; ++i) {
      mbar_init(bar_wfull + 8 * i, 1);
      mbar_init(bar_wempty + 8 * i, 4);
    }
    for (int i = 0; i < XST; ++i) {
      mbar_init(bar_xfull + 8 * i, 1);
      mbar_init(bar_xempty + 8 * i, 1);
    }
    for (int i = 0; i < AST; ++i) {
      mbar_init(bar_afull + 8 * i, 128);
      mbar_init(bar_aempty + 8 * i, 1);
    }
    mbar_init(bar_accfull, 1);
    mbar_init(bar_accempty, 32 * NDW);                    // threads that read the accumulator in the epilogue
    mbar_init(bar_epi, 32 * NDW);
    mbar_init(bar_drain, 1);
    *abort_flag = 0;
    tmem_slot[3] = 0;                                   // a flag nobody sets (used by the drain waits)
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Weight producer state (one elected thread of warp 0).  The first ring of weight loads goes out before the rest of the prologue
  // (table, TMEM allocation): the packed weights depend on nothing, and the first HBM round trip then overlaps it.
  int issued = 0;
  int p_rt = tile / a.token_tiles, p_tt = tile - p_rt * a.token_tiles;
  Ring<WST> wr;
  auto produce_w = [&]() {
    // The packed buffer as a (piece bytes, k chunk, strip) tensor: one box brings chunks c0 .. c0 + CH - 1 of the
    // row tile's eight strips, [strip][chunk][piece] in shared memory (chunks past the end of K arrive as zeros).
    mbar_expect_tx(bar_wfull + 8 * wr.slot, (uint32_t)Cfg::W_BYTES);
    tma_load_3d(smem_w + wr.slot * Cfg::W_BYTES, &tmap_w, 0, step * CH, p_rt * TILE_STRIPS, bar_wfull + 8 * wr.slot);
    if (step == spt - 1 && ++p_tt == a.token_tiles) { p_tt = 0; ++p_rt; }
    next_item();
    wr.next();
  };
  __syncwarp();
  if (warp == 0 && elect_one()) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_w) : "memory");
    grid_dep_launch();                                    // the next kernel may start its own prologue
    for (; issued < n_items && issued < WST; ++issued) produce_w();
  }
  if (warp >= 2) {
    decode_tables_fill(tables, threadIdx.x - 64, Cfg::THREADS - 64);
    if (TABLE) pair_table_fill(smem_addr(umma_smem), threadIdx.x - 64, Cfg::THREADS - 64, a.svp0, a.svp1);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)Cfg::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tmem_a0 = tmem_base + Cfg::ACC_COLS;

  auto fail = [&](uint32_t code) {
    *abort_flag = 1;
    grid_dep_wait();                                      // the status word lives in the (possibly shared) workspace
    atomicCAS(a.status, 0u, code);
    show_status(a.status_host, code);
  };

  if (warp == 0) {
    // ===================== weight producer =====================
    if (elect_one()) {                                    // as for the MMAs; 128 x 14336 x 4096 20.0 -> 18.7 us with both producers elected
      for (; issued < n_items; ++issued) {
        if (!mbar_wait(bar_wempty + 8 * wr.slot, wr.phase ^ 1u, abort_flag)) { fail(1); break; }
        produce_w();
      }
      // Drain: copies still in flight must land before this CTA's shared memory is released.
      const int pending = issued < WST ? issued : WST;
      for (int f = issued - pending; f < issued; ++f)
        mbar_wait(bar_wfull + 8 * (f % WST), (uint32_t)((f / WST) & 1), tmem_slot + 3);
    }
  } else if (warp == X_WARP) {
    // ===================== activation producer =====================
    if (elect_one()) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_x) : "memory");
      grid_dep_wait();                                    // activations may belong to the preceding kernel
      if (cta == 0 && a.status_host) show_status(a.status_host, *(volatile uint32_t*)a.status);   // what an earlier call left
      Ring<XST> xr;
      int done = 0;                                       // stages
      bool alive = true;
      for (int i = 0; alive && i < n_items; ++i) {
        for (int c0 = step * CH; alive && c0 < min((step + 1) * CH, a.g.k_chunks); c0 += CHX) {
          if (!mbar_wait(bar_xempty + 8 * xr.slot, xr.phase ^ 1u, abort_flag)) { fail(2); alive = false; break; }
          const uint32_t st = smem_x + xr.slot * Cfg::X_BYTES, bar = bar_xfull + 8 * xr.slot;
          if (a.x_map_3d) {                               // the 3-D box always spans CHX chunks (zero-filled past K)
            mbar_expect_tx(bar, (uint32_t)Cfg::X_BYTES);
            tma_load_3d(st, &tmap_x, 0, p_tt * NT, c0, bar);
          } else {
            const int nch = min(CHX, a.g.k_chunks - c0);
            mbar_expect_tx(bar, (uint32_t)(nch * Cfg::X_BOX_BYTES));
            for (int c = 0; c < nch; ++c) tma_load_2d(st + c * Cfg::X_BOX_BYTES, &tmap_x, (c0 + c) * CHUNK_K, p_tt * NT, bar);
          }
          xr.next();
          ++done;
        }
        if (step == spt - 1 && ++p_tt == a.token_tiles) p_tt = 0;
        next_item();
      }
      const int pending = done < XST ? done : XST;
      for (int f = done - pending; f < done; ++f)
        mbar_wait(bar_xfull + 8 * (f % XST), (uint32_t)((f / XST) & 1), tmem_slot + 3);
    }
  } else if (warp == 1) {
    // ===================== MMA issuer =====================
    constexpr uint32_t idesc = make_idesc(NT);
    // Shared-memory descriptor of a K-major bf16 tile in the 128-byte swizzle (rows of 128 bytes, 64 elements): upper half = 1024 bytes
    // from one group of eight rows to the next, descriptor version, swizzle mode
    constexpr uint32_t bd_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    // One elected lane walks the items.  Electing once around the whole loop lets the compiler keep descriptors and
    // addresses in uniform registers; electing anew for every item cost about 37 cycles per tcgen05 instruction.
    if (elect_one()) {
      uint32_t seg = 0;
      int seg_items = 0;                                  // of the segment, issued
      bool alive = true;
      Ring<XST> xr;
      Ring<AST> ar;
      // What is there first is waited for first (a wait that finds its stage full still takes 150 cycles): the first item's weights, since
      // its activations may belong to the preceding kernel, and from then on the activations.  16 x 256 x 256 2.35 us with the activations
      // first throughout, 2.14 this way; the two barriers are chosen an item ahead, since choosing them here cost 2 % at 192 tokens.
      uint32_t bar0 = bar_afull, phase0 = 0, bar1 = bar_xfull, phase1 = 0;
      for (int i = 0; i < n_items; ++i) {
        const bool seg_first = (i == 0) || step == 0;
        const bool seg_last = (i + 1 == n_items) || step == spt - 1;
        const int nch = min(CH, a.g.k_chunks - step * CH);
        if (!mbar_wait(bar0, phase0, abort_flag)) { fail(i > 0 ? 10 : 3); break; }
        if (seg_first && !mbar_wait(bar_accempty, (seg & 1u) ^ 1u, abort_flag)) { fail(4); break; }
        if (!mbar_wait(bar1, phase1, abort_flag)) { fail(i > 0 ? 3 : 10); break; }
        tc_fence_after();
        const uint32_t a_t = tmem_a0 + ar.slot * Cfg::A_STAGE_COLS;
        if (seg_first) seg_items = 0;
        const bool fresh = seg_items++ < Cfg::SETS;       // the item's set of accumulators holds nothing of this segment yet
        const uint32_t d_0 = tmem_base + (Cfg::SETS > 1 ? ar.slot * (Cfg::PER_SET * NT) : 0);
        // Consecutive MMAs go to different accumulators (summed in the epilogue): MMAs on one
        // accumulator execute one after the other, and a narrow MMA is far shorter than its latency.
#pragma unroll
        for (int h = 0; h < CH / CHX; ++h) {
          if (h * CHX < nch) {
            if (h > 0) {
              if (!mbar_wait(bar_xfull + 8 * xr.slot, xr.phase, abort_flag)) { fail(10); alive = false; break; }
              tc_fence_after();
            }
            const uint32_t bd_lo = ((smem_x + xr.slot * Cfg::X_BYTES) >> 4) | (1u << 16);   // start address and (unused) leading offset fields
#pragma unroll
            for (int k = 0; k < CHX * 4; ++k) {
              const int j = h * CHX * 4 + k;
              // 16 k further along: +32 bytes inside a chunk's 128-byte rows, next chunk's box after four
              if (j < nch * 4) {
                const uint32_t bd = bd_lo + (uint32_t)(((k >> 2) * Cfg::X_BOX_BYTES + (k & 3) * 32) >> 4);
                const uint32_t d_t = d_0 + (j % Cfg::PER_SET) * NT;
                if (j < Cfg::PER_SET && fresh) tc_mma_ts<false>(d_t, a_t + j * 8, bd, bd_hi, idesc);
                else tc_mma_ts<true>(d_t, a_t + j * 8, bd, bd_hi, idesc);
              }
            }
            tc_commit(bar_xempty + 8 * xr.slot);
            xr.next();
          }
        }
        if (!alive) break;
        tc_commit(bar_aempty + 8 * ar.slot);
        if (seg_last) { tc_commit(bar_accfull); ++seg; }
        next_item();
        ar.next();
        bar0 = bar_xfull + 8 * xr.slot, phase0 = xr.phase;
        bar1 = bar_afull + 8 * ar.slot, phase1 = ar.phase;
      }
    }
    // The MMAs issued so far read shared memory and TMEM and write TMEM until they complete: commit them to a barrier
    // and wait for it (bounded, not watching the abort flag) before the CTA may release either.
    __syncwarp();
    if (elect_one()) tc_commit(bar_drain);
    __syncwarp();
    mbar_wait(bar_drain, 0u, tmem_slot + 3);
  } else {
    // ===================== dequant (32 * NDW threads, thread = weight row) + epilogue =====================
    const int row = 32 * (warp & 3) + lane;              // TMEM lane this thread owns
    const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
    const int group = (warp - 2) >> 2;                   // item i is decoded by group i % GROUPS
    // all 32 lanes take the same branch after a wait, so the .aligned tcgen05 instructions stay convergent
    auto wait_all = [&](uint32_t bar, uint32_t parity, uint32_t code) -> bool {
      const bool got = mbar_wait(bar, parity, abort_flag);
      if (!got) fail(code);
      return __all_sync(0xFFFFFFFFu, got);
    };
    const uint32_t ss_lane = smem_addr(tables) + lane * 4;
    const uint32_t mul_lo = a.mul_lo, mul_hi = a.mul_hi, lanes = (uint32_t)lane * 0x04040404u;
    // where this thread's weight row sits inside a stage ([strip 0..7][chunk 0..CH-1] pieces): strip row / 16, row r = row % 16 of it
    const int r16 = row % STRIP_ROWS;
    const uint32_t strip_at = smem_w + (uint32_t)(row / STRIP_ROWS) * (CH * PIECE_BYTES);
    const uint32_t scale_off = (uint32_t)PIECE_CODE_BYTES + (uint32_t)(r16 & 7) * 8;
    const uint32_t scale_sel = (r16 >> 3) ? 0x7531u : 0x6420u;
    const uint32_t code_off = (uint32_t)r16 * 8;         // ^ 32 blk: row r of block blk sits in slot r ^ (4 blk)
    // The epilogue of a finished segment runs after the group has decoded as far ahead as its operand stages allow, so that
    // the MMAs go on meanwhile.
    struct Pending { int tile; bool at_end; } pending = {-1, false};
    int ahead = 0;                                       // items of the group's own since then
    const EpilogueCtx ctx = {bar_accfull, bar_accempty, bar_epi, tmem_base + lane_off, row, group, threadIdx.x == 64};
    uint32_t seg = 0, epi_phase = 0;
    auto epilogue = [&]() -> bool {
      grid_dep_wait();                                     // outputs, workspace and the scale scalar may belong to the preceding kernel
      const float ts = a.extra_scale ? a.tensor_scale * *a.extra_scale : a.tensor_scale;
      const int done_tile = pending.tile;
      pending.tile = -1;
      uint32_t live = 1u;                                  // sets of accumulators that an item of the segment went to
      if (Cfg::SETS > 1) {
        const int first = max(done_tile * spt - it_begin, 0), count = min((done_tile + 1) * spt, it_end) - it_begin - first;
        live = 0;
#pragma unroll
        for (int q = 0; q < Cfg::SETS; ++q) live |= (uint32_t)((q + Cfg::SETS - first % Cfg::SETS) % Cfg::SETS < count) << q;
      }
      return segment_epilogue<NT, Cfg::PER_SET, Cfg::SETS, GROUPS>(
          a, ctx, done_tile, pending.at_end, live, ts, seg++, epi_phase, abort_flag,
          [&](uint32_t bar, uint32_t parity, uint32_t which) { return wait_all(bar, parity, 7u + which); },
          [&](uint32_t which) { fail(7u + which); });
    };
    // The group walks its own items only: bookkeeping for the others' cost as much as a third of a decode.
    bool all_closed = n_items == 0;
    step += group;
    uint32_t turn = 0;                                   // the group's items so far
    constexpr uint32_t WTURNS = WST / GROUPS, ATURNS = AST / GROUPS;   // stages and slots that serve a group
    for (int i = group;;) {
      const bool crossed = step >= spt && tile < last_tile;   // a segment ends before the group's next item
      if (pending.tile >= 0 && (crossed || i >= n_items || ahead == AST / GROUPS)) {   // (one call: it is large when inlined)
        if (!epilogue()) break;
        continue;
      }
      if (crossed) {
        pending = {tile, true};
        ahead = 0;
        step -= spt;
        ++tile;
        continue;
      }
      if (i >= n_items) {
        if (all_closed) break;
        all_closed = true;
        pending = {tile, it_end == (last_tile + 1) * spt};
        continue;
      }
      {
        const int nch = min(CH, a.g.k_chunks - step * CH);
        const uint32_t wslot = group + GROUPS * (turn % WTURNS), aslot = group + GROUPS * (turn % ATURNS);
        const uint32_t st = strip_at + wslot * Cfg::W_BYTES;
        const uint32_t a_t = tmem_a0 + aslot * Cfg::A_STAGE_COLS + lane_off;
        // a chunk's scale word and codes
        auto load = [&](uint32_t ck, uint32_t& sw, uint2 (&cw)[CHUNK_BLOCKS]) {
          const uint2 sq = lds64(ck + scale_off);           // the eight scale bytes of rows r % 8 and r % 8 + 8
#pragma unroll
          for (int blk = 0; blk < CHUNK_BLOCKS; ++blk) cw[blk] = lds64(ck + blk * (STRIP_ROWS * 8) + (code_off ^ (32u * blk)));
          sw = __byte_perm(sq.x, sq.y, scale_sel);          // this row's four, in block order
        };
        if (!wait_all(bar_wfull + 8 * wslot, (turn / WTURNS) & 1u, 5)) break;
        uint32_t sw;
        uint2 cw[CHUNK_BLOCKS];
        load(st, sw, cw);
        uint32_t pairs[2][16];
        if (TABLE) lookup_blocks(umma_smem, (sw & 0x80808080u) | lanes, 0, cw, pairs[0]);
        if (!wait_all(bar_aempty + 8 * aslot, ((turn / ATURNS) & 1u) ^ 1u, 6)) break;
        tc_fence_after();
        if constexpr (TABLE) {
          // half a chunk's lookups are on their way while the half before is scaled and put in order
#pragma unroll
          for (int c = 0; c < CH; ++c) {
            if (c < nch) {
              uint32_t ss2[CHUNK_BLOCKS], v[8 * CHUNK_BLOCKS];
#pragma unroll
              for (int blk = 0; blk < CHUNK_BLOCKS; ++blk) ss2[blk] = decode_block_scale(ss_lane, sw, blk);
              lookup_blocks(umma_smem, (sw & 0x80808080u) | lanes, 2, cw, pairs[1]);
              if (c + 1 < CH) load(st + (c + 1) * PIECE_BYTES, sw, cw);   // beyond the last chunk, or past the end of K: unused or zeros
              finish_blocks(pairs[0], ss2[0], ss2[1], v);
              if (c + 1 < CH) lookup_blocks(umma_smem, (sw & 0x80808080u) | lanes, 0, cw, pairs[0]);
              finish_blocks(pairs[1], ss2[2], ss2[3], v + 16);
              tc_st32(a_t + c * 32, v);
            }
          }
        } else {
#pragma unroll
          for (int c = 0; c < CH; ++c) {
            if (c < nch) {
              uint32_t ss2[CHUNK_BLOCKS];
#pragma unroll
              for (int blk = 0; blk < CHUNK_BLOCKS; ++blk) ss2[blk] = decode_block_scale(ss_lane, sw, blk);
              // the next chunk is fetched while this one is decoded (beyond the last one, or past the end of K: unused or zeros)
              uint32_t sw_next = 0;
              uint2 cw_next[CHUNK_BLOCKS];
              if (c + 1 < CH) load(st + (c + 1) * PIECE_BYTES, sw_next, cw_next);
              // (One store for the chunk lets the four blocks' decodes mix.)
              uint32_t v[8 * CHUNK_BLOCKS];
#pragma unroll
              for (int blk = 0; blk < CHUNK_BLOCKS; ++blk) {
                const uint32_t svp = (sw & (PACKED_SELECT << (8 * blk))) ? a.svp1 : a.svp0;
                decode_word(cw[blk].x, ss2[blk], svp, mul_lo, mul_hi, v + 8 * blk);
                decode_word(cw[blk].y, ss2[blk], svp, mul_lo, mul_hi, v + 8 * blk + 4);
              }
              tc_st32(a_t + c * 32, v);
              if (c + 1 < CH) {
                sw = sw_next;
#pragma unroll
                for (int blk = 0; blk < CHUNK_BLOCKS; ++blk) cw[blk] = cw_next[blk];
              }
            }
          }
        }
        __syncwarp();                                       // every lane has read the stage
        if (lane == 0) mbar_arrive(bar_wempty + 8 * wslot);
        ++ahead;
        ++turn;
        i += GROUPS;
        step += GROUPS;
        tc_wait_st();
        tc_fence_before();
        mbar_arrive(bar_afull + 8 * aslot);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();                                       // lane 0 ran the issue loop alone; dealloc is warp-wide
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)Cfg::TMEM_COLS)
                 : "memory");
  }
}

// ------------------------------------------------------------------ host side
struct UmmaPlan {
  int NT, CH, CHX;             // token tile; chunks per item, per activation stage
  bool table;                  // weights decoded by table
  int token_tiles, steps_per_tile, grid;
  long long tiles, total_items;
  size_t slots_bytes;
};

// Token tile, decode and grid: the cheapest by the cost model (razer_tcgen05.cuh), fitted to 63,000 times of 3823 sizes (M 9 .. 2048, N and K
// 256 .. 28672, all widths and grids, launches back to back; 900 of them with weights, activations and workspaces all in turn, under
// sustained load).  Of the best of a size's grids the choice is 0.6 % off in the mean; by fewer constants per width (one start for all,
// no `late`, no `spread`) it was 2.2 % off: 53 x 512 x 4352 7.06 us instead of 6.37, 93 x 512 x 2816 6.88 (6.22), 239 x 1590 x 1648 7.69 (6.75),
// 64 x 2341 x 816 3.79 (3.46).
// Up to 32 tokens the table costs a start (every CTA fills it) and gains by the chunk: at 16 tokens it is level with the registers at
// 1 to 3 items of four chunks a CTA (1 item +1.3 %) and faster from there (6 -4.5 %, 16 -11 %), at 32 tokens from 6 on (1 to 5 +3 to +6 %, 8 -5 %,
// 16 -7 %).
static const TileCost tile_costs[] = {
    {16, 4, 4, true, 0.321f, 0.135f, 0.114f, 0.408f, 1.423f, 3.535f, 0.207f, 4.69f, 0.172f, 0.191f, 4.131f},
    {16, 4, 4, false, 0.315f, 0.0f, 0.119f, 0.638f, 1.345f, 3.239f, 0.24f, 4.975f, 0.161f, 0.147f, 4.499f},
    {32, 4, 2, true, 0.922f, 0.164f, 0.129f, 0.467f, 0.894f, 2.883f, 0.172f, 3.902f, 0.229f, 0.306f, 4.087f},
    {32, 4, 4, false, 0.552f, 0.001f, 0.128f, 0.707f, 1.118f, 3.026f, 0.173f, 4.346f, 0.183f, 0.204f, 4.581f},
    {64, 4, 4, false, 0.637f, 0.727f, 0.139f, 0.542f, 1.172f, 3.179f, 0.205f, 4.394f, 0.346f, 0.827f, 0.953f},
    {96, 4, 2, false, 0.447f, 1.219f, 0.155f, 0.375f, 1.584f, 3.506f, 0.225f, 4.894f, 0.469f, 0.606f, 0.541f},
    {128, 4, 1, false, 0.122f, 1.194f, 0.183f, 0.362f, 1.981f, 4.037f, 0.333f, 5.988f, 0.895f, 0.707f, 0.295f},
    {192, 2, 1, false, 0.0f, 1.329f, 0.221f, 0.366f, 2.816f, 5.203f, 0.378f, 6.982f, 1.055f, 0.533f, 0.0f},
    {256, 2, 1, false, 0.0f, 0.949f, 0.257f, 0.44f, 3.516f, 5.896f, 0.48f, 7.576f, 1.685f, 0.652f, 0.213f}};

static bool admissible(const TileCost& t, int M) { return t.NT <= 16 || t.NT < 2 * M; }   // not half of the tile or more padding

static UmmaPlan work_out_plan(const razer_desc* d, int M) {
  UmmaPlan best;
  float best_cost = 0.0f;
  const Geometry g = make_geometry(d->N, d->K);
  for (const TileCost& t : tile_costs) {
    if (!admissible(t, M)) continue;
    UmmaPlan p;
    p.NT = t.NT;
    p.CH = t.CH;
    p.CHX = t.CHX;
    p.table = t.table;
    p.token_tiles = (M + p.NT - 1) / p.NT;
    p.steps_per_tile = (g.k_chunks + p.CH - 1) / p.CH;
    p.tiles = (long long)g.row_tiles * p.token_tiles;
    p.total_items = p.tiles * p.steps_per_tile;
    const float cost = best_grid(t, p.tiles, p.steps_per_tile, sm_count(), p.grid);
    if (best_cost == 0.0f || cost < best_cost) { best_cost = cost; best = p; }
  }
  best.slots_bytes = (size_t)best.grid * best.NT * TILE_ROWS * sizeof(float);
  return best;
}

static UmmaPlan make_plan(const razer_desc* d, int M) {
  return remembered<UmmaPlan>(d->N, d->K, M, 0, [&] { return work_out_plan(d, M); });
}

bool umma_supported(const razer_desc* d, int M) {
  (void)d;
  (void)M;
  // RAZER_KERNEL=simt routes every matmul to the CUDA-core kernel (debugging aid)
  const char* e = getenv("RAZER_KERNEL");
  return !(e && e[0] == 's' && e[1] == 'i');
}

size_t umma_workspace_bytes(const razer_desc* d, int M) { return WS_ZERO_BYTES + make_plan(d, M).slots_bytes; }
// No call against up to M tokens needs more, whatever its shape.
size_t umma_workspace_bound(int M) {
  int widest = 0;
  for (const TileCost& t : tile_costs)
    if (admissible(t, M) && t.NT > widest) widest = t.NT;
  return WS_ZERO_BYTES + (size_t)sm_count() * widest * TILE_ROWS * sizeof(float);
}

template <int NT, int CH, int CHX, int WST, int XST, int AST, int NDW, int NACC, bool TABLE>
static int launch_cfg(const CUtensorMap& tmap, const CUtensorMap& tmap_w, const UmmaArgs& args, int grid, cudaStream_t st) {
  using Cfg = UmmaCfg<NT, CH, CHX, WST, XST, AST, NDW, NACC, TABLE>;
  auto kern = razer_umma_kernel<NT, CH, CHX, WST, XST, AST, NDW, NACC, TABLE>;
  static bool attr_set = false;
  if (!attr_set) {
    RAZER_TRY(check_cuda(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM_BYTES),
                         "cudaFuncSetAttribute(max dynamic shared memory)"));
    attr_set = true;
  }
  return launch_dependent("razer_umma_kernel launch", kern, grid, Cfg::THREADS, Cfg::SMEM_BYTES, st, tmap, tmap_w, args);
}

int launch_gemm_umma(const razer_desc* d, const void* packed, const void* x, int M, int ldx_K, float extra_scale,
                     const float* extra_scale_dev, void* y, void* ws, size_t ws_bytes, cudaStream_t st, uint32_t* status_host) {
  const Geometry g = make_geometry(d->N, d->K);
  const UmmaPlan p = make_plan(d, M);
  const size_t need = WS_ZERO_BYTES + p.slots_bytes;
  if (!ws || ws_bytes < need)
    return set_error(RAZER_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, ws_bytes);
  EncodeTiledFn enc = encode_fn();
  if (!enc) return set_error(RAZER_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  CUtensorMap tmap;
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = CUDA_ERROR_UNKNOWN;
  int map_3d = 0;
  if (d->K % CHUNK_K == 0 && ldx_K == d->K) {
    // (64 k, tokens, k chunk) view of x: one box brings the activations of all CHX chunks of a stage
    const cuuint64_t dims[3] = {(cuuint64_t)CHUNK_K, (cuuint64_t)M, (cuuint64_t)(d->K / CHUNK_K)};
    const cuuint64_t strides[2] = {(cuuint64_t)ldx_K * 2, (cuuint64_t)CHUNK_K * 2};
    const cuuint32_t box[3] = {(cuuint32_t)CHUNK_K, (cuuint32_t)p.NT, (cuuint32_t)p.CHX};
    r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(x), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    map_3d = (r == CUDA_SUCCESS);
  }
  if (!map_3d) {
    const cuuint64_t dims[2] = {(cuuint64_t)d->K, (cuuint64_t)M};
    const cuuint64_t strides[1] = {(cuuint64_t)ldx_K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)CHUNK_K, (cuuint32_t)p.NT};
    r = enc(&tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(x), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  if (r != CUDA_SUCCESS) return set_error(RAZER_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
  // packed weights: (72 x 8 bytes of a piece, k chunk, strip), box = (whole piece, CH chunks, the tile's 8 strips)
  CUtensorMap tmap_w;
  {
    const cuuint64_t dims[3] = {(cuuint64_t)(PIECE_BYTES / 8), (cuuint64_t)g.k_chunks, (cuuint64_t)g.strips()};
    const cuuint64_t strides[2] = {(cuuint64_t)PIECE_BYTES, (cuuint64_t)g.strip_bytes()};
    const cuuint32_t box[3] = {(cuuint32_t)(PIECE_BYTES / 8), (cuuint32_t)p.CH, (cuuint32_t)TILE_STRIPS};
    r = enc(&tmap_w, CU_TENSOR_MAP_DATA_TYPE_INT64, 3, const_cast<void*>(packed), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(RAZER_ERR_CUDA, "cuTensorMapEncodeTiled (weights) failed with code %d", (int)r);
  }

  UmmaArgs a;
  a.y = (__nv_bfloat16*)y;
  a.status = (uint32_t*)ws;
  a.counters = (uint32_t*)((char*)ws + WS_STATUS_BYTES);
  a.slots = (float*)((char*)ws + WS_ZERO_BYTES);
  a.status_host = status_host;
  a.extra_scale = extra_scale_dev;
  a.g = g;
  a.svp0 = special_value_pair(d->sv_mag[0]);
  a.svp1 = special_value_pair(d->sv_mag[1]);
  a.mul_lo = (1u << 6) + (1u << 12);
  a.mul_hi = (1u << 2) + (1u << 8);
  a.tensor_scale = d->tensor_scale * extra_scale;
  a.M = M;
  a.token_tiles = p.token_tiles;
  a.steps_per_tile = p.steps_per_tile;
  a.split = p.grid % p.tiles == 0 ? (int)(p.grid / p.tiles) : 0;
  a.total_items = p.total_items;
  a.x_map_3d = map_3d;
  switch (p.NT) {
    case 16: return p.table ? launch_cfg<16, 4, 4, 6, 4, 3, 12, 6, true>(tmap, tmap_w, a, p.grid, st) : launch_cfg<16, 4, 4, 6, 4, 3, 12, 6, false>(tmap, tmap_w, a, p.grid, st);
    case 32: return p.table ? launch_cfg<32, 4, 2, 6, 4, 3, 12, 2, true>(tmap, tmap_w, a, p.grid, st) : launch_cfg<32, 4, 4, 6, 4, 3, 12, 2, false>(tmap, tmap_w, a, p.grid, st);
    case 64: return launch_cfg<64, 4, 4, 6, 3, 3, 12, 2, false>(tmap, tmap_w, a, p.grid, st);
    case 96: return launch_cfg<96, 4, 2, 6, 4, 3, 12, 1, false>(tmap, tmap_w, a, p.grid, st);
    case 128: return launch_cfg<128, 4, 1, 6, 6, 3, 12, 1, false>(tmap, tmap_w, a, p.grid, st);
    case 192: return launch_cfg<192, 2, 1, 8, 5, 4, 16, 1, false>(tmap, tmap_w, a, p.grid, st);
    default: return launch_cfg<256, 2, 1, 8, 4, 4, 16, 1, false>(tmap, tmap_w, a, p.grid, st);
  }
}

}  // namespace razer
