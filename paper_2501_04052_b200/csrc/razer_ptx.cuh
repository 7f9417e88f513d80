// Inline-PTX wrappers shared by the matmul kernels: mbarriers with bounded waits, TMA bulk copies and tensor
// loads, warp election, programmatic dependent launch.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace razer {

constexpr uint32_t WAIT_LIMIT = 1u << 26;             // try_wait rounds before a wait gives up, and
constexpr uint64_t WAIT_LIMIT_NS = 2000000000ull;     // its wall-clock bound (2 s)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// One poll of a barrier phase.  The hint lets the hardware park the thread until the phase
// completes (or about the hinted time passes) instead of spinning in the issue slots that
// the decoding warps need.
constexpr uint32_t WAIT_SLICE_NS = 1000000u;
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(WAIT_SLICE_NS)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait; false = gave up (or another thread already flagged a failure).  In line and without a call, so that the issuing
// loops keep their uniform registers; the clock is read only once per WAIT_POLLS polls, of up to WAIT_SLICE_NS each: the first look
// starts the count, and the wait gives up at the first one after the rest of WAIT_LIMIT_NS.
constexpr uint32_t WAIT_POLLS = 256;
constexpr uint64_t WAIT_REST_NS = WAIT_LIMIT_NS - 2ull * WAIT_POLLS * WAIT_SLICE_NS;
static_assert(2ull * WAIT_POLLS * WAIT_SLICE_NS < WAIT_LIMIT_NS, "the looks before and after the count are part of the limit");
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (i % WAIT_POLLS == 0) {
      const uint64_t t = global_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > WAIT_REST_NS || i >= WAIT_LIMIT) return false;
    }
  }
}
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// True in exactly one lane of a converged warp.  Loops that only issue asynchronous work run
// on the whole warp with this predicate around the issuing instructions, so that addresses
// and descriptors stay warp-uniform values.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}
// Programmatic dependent launch: when the kernel was launched with the programmatic-serialization
// attribute, `grid_dep_wait` returns once the preceding kernel in the stream has completed (otherwise at
// once); everything that may depend on that kernel (activations, workspace, outputs) is touched after it,
// while the weight stream, which depends on nothing, starts before.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A status other than 0 for a host that waits on the call (`host`: pinned memory, or NULL).
__device__ __forceinline__ void show_status(uint32_t* host, uint32_t code) {
  if (host && code) *(volatile uint32_t*)host = code;
}

}  // namespace razer
