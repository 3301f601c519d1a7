// Bounded waits of the GEMM kernels' roles on their mbarriers (the PTX wrappers are in tc_ptx.cuh).  They return false (and
// record `site`) if the barrier did not flip within the time limit or another role of this CTA already gave up.
#pragma once

#include "tc_ptx.cuh"

namespace nvfp4 {
namespace {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s
__device__ unsigned int g_error_word = 0;                   // where the waits that ran out are recorded

// mbar_wait spins without pause: for the MMA issuer, whose latency is the kernel's critical path.
// mbar_wait_relaxed sleeps between polls: every other role waits most of the time, and a dozen
// warps polling shared memory back to back slow the issuer's own barrier reads several times over.
__device__ __forceinline__ bool mbar_wait_timeout(uint32_t site, volatile uint32_t* abort_flag, unsigned long long t0) {
  if (*abort_flag) return true;
  if (global_timer_ns() - t0 > kWaitLimitNs) {
    *abort_flag = 1u;
    atomicOr(&g_error_word, 0x100u | site);
    return true;
  }
  return false;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
  for (int i = 0; i < 4096; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (mbar_wait_timeout(site, abort_flag, t0)) return false;
  }
}
__device__ __forceinline__ bool mbar_wait_relaxed(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  while (true) {
    for (int i = 0; i < 256; ++i) {
      __nanosleep(32);
      if (mbar_try_wait(bar, parity)) return true;
    }
    if (mbar_wait_timeout(site, abort_flag, t0)) return false;
  }
}
// Wait of the MMA-issuing warp.  The poll is a relaxed one: with MMAs in flight an acquiring
// try_wait stalls its thread for ~170 cycles even when the phase is already complete, a relaxed one
// for ~40, and the issuer has only 512 cycles per stage.  Nothing the issuer does afterwards reads
// memory through the generic proxy: it issues tcgen05.mma, whose shared-memory operands were written
// by the bulk copies that completed the phase, and whose tensor-memory scales are ordered by
// tcgen05.fence::after_thread_sync.
__device__ __forceinline__ bool mbar_wait_issuer(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
  for (int i = 0; i < 4096; ++i)
    if (mbar_try_wait_relaxed(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait_relaxed(bar, parity)) return true;
    if (mbar_wait_timeout(site, abort_flag, t0)) return false;
  }
}
// A whole-warp wait ends alike for every lane: behind it stand instructions that the whole warp has to execute (tcgen05.ld, .st),
// and lanes that poll for themselves may see the barrier flip, or the time run out, at different polls.
//
// The scale movers' waits are polled as the issuer's by every lane: these warps issue tcgen05.st, and next to such operations an
// acquiring poll costs ~180 cycles even when the phase is complete (see mbar_wait_issuer), which with two waits per stage made the
// movers the slowest role.  What they read afterwards is shared memory written by the bulk copies that completed the phase, so
// the successful polls are followed by one acquire fence at CTA scope: relaxed observation + fence is the acquire pattern of the
// PTX memory model.  A stage's two waits share the vote and the fence: products of 3001 x 4096 x 11008 and 3001 x 11008 x 4096, one
// chained to the other, took 171.5 us with a fence for each wait and no vote, 171.7 with a vote for each too, and take 170.0 so.
__device__ __forceinline__ bool warp_acquire(bool ok) {
  ok = __all_sync(0xFFFFFFFFu, ok);
  asm volatile("fence.acq_rel.cta;" ::: "memory");
  return ok;
}
__device__ __forceinline__ bool mbar_wait_warp_spin(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
  return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag, site));
}
// Whole-warp wait: lane 0 polls, then every lane observes the completed phase once itself.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait_relaxed(bar, parity, abort_flag, site);
  ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
  if (ok) (void)mbar_try_wait(bar, parity);
  return ok;
}

}  // namespace
}  // namespace nvfp4
