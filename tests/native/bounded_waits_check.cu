// The whole-warp waits of paper_2505_19115_b200/csrc/bounded_waits.cuh end alike for every lane.  One warp waits on two barriers,
// one complete and one that nothing completes; every wait ends by itself.  Prints "ok" and exits 0 when every check holds.
#include <cstdio>

#include "bounded_waits.cuh"

using namespace nvfp4;

using Wait = bool (*)(uint32_t, uint32_t, volatile uint32_t*, uint32_t);

// odd: which barrier the odd lanes wait on; aborted: another role has given up already.
template <Wait WAIT>
__global__ void wait_kernel(int even, int odd, uint32_t aborted, uint32_t site, unsigned int* ended_true) {
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t abort_flag;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) mbar_init(smem_u32(&bars[i]), 1);
    mbar_arrive(smem_u32(&bars[0]));
    abort_flag = aborted;
  }
  __syncthreads();
  const bool ok = WAIT(smem_u32(&bars[(threadIdx.x & 1) ? odd : even]), 0, &abort_flag, site);
  const unsigned int votes = __ballot_sync(0xFFFFFFFFu, ok);
  if (threadIdx.x == 0) *ended_true = votes;
}

__device__ bool movers_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t site) {
  return warp_acquire(mbar_wait_issuer(bar, parity, abort_flag, site));
}

template <Wait WAIT>
bool ends_as(unsigned int want, unsigned int want_word, int even, int odd, uint32_t aborted, uint32_t site) {
  unsigned int *dev = nullptr, got = 0x5555u, word = 0, zero = 0;
  if (cudaMalloc(&dev, sizeof(got)) != cudaSuccess) return false;
  wait_kernel<WAIT><<<1, 32>>>(even, odd, aborted, site, dev);
  const bool ran = cudaDeviceSynchronize() == cudaSuccess && cudaMemcpy(&got, dev, sizeof(got), cudaMemcpyDeviceToHost) == cudaSuccess &&
                   cudaMemcpyFromSymbol(&word, g_error_word, sizeof(word)) == cudaSuccess &&
                   cudaMemcpyToSymbol(g_error_word, &zero, sizeof(zero)) == cudaSuccess;
  cudaFree(dev);
  if (ran && got == want && word == want_word) return true;
  std::printf("FAILED: barriers %d %d, aborted %u: lanes %08x (want %08x), word %x (want %x), ran %d\n", even, odd, aborted, got, want, word, want_word, (int)ran);
  return false;
}

template <Wait WAIT>
bool check(uint32_t site) {
  return ends_as<WAIT>(~0u, 0u, 0, 0, 0u, site) &&                 // complete
         ends_as<WAIT>(~0u, 0u, 0, 0, 1u, site) &&                 // complete, and another role has given up
         ends_as<WAIT>(0u, 0u, 1, 1, 1u, site) &&                  // another role has given up
         ends_as<WAIT>(0u, 0x100u | site, 1, 1, 0u, site);         // the time runs out
}

int main() {
  bool ok = check<mbar_wait_warp>(0x04) && check<mbar_wait_warp_spin>(0x14) && check<movers_wait>(0x16);
  // some lanes see the barrier flip, others give up: none goes on
  ok = ok && ends_as<mbar_wait_warp_spin>(0u, 0u, 0, 1, 1u, 0x14) && ends_as<mbar_wait_warp_spin>(0u, 0x114u, 1, 0, 0u, 0x14);
  ok = ok && ends_as<movers_wait>(0u, 0u, 0, 1, 1u, 0x16) && ends_as<movers_wait>(0u, 0x116u, 1, 0, 0u, 0x16);
  std::puts(ok ? "ok" : "failed");
  return ok ? 0 : 1;
}
