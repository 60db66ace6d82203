// psl_tail_wide.cu -- the short walks' step tail in blocks of eight warps, for batches too small to
// fill the SMs with one-warp blocks: each walk's phases, a chain of loads and reductions bound by their
// latency, are then spread over eight warps (one walk of L = 1023: the tail 40 -> 23 us of the step).
#include "psl_tail.cuh"

namespace psl {

constexpr int kTailWideThreads = 256;

static uint32_t g_tail_wide_per_sm = 1;

cudaError_t prepare_tail_wide_kernel() {
  int nb = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_step_tail<kTailWideThreads, kTailWideThreads, 2>,
                                                                kTailWideThreads, 0);
  g_tail_wide_per_sm = (uint32_t)(nb > 0 ? nb : 1);
  return e;
}

cudaError_t launch_step_tail_wide(const LaunchCtx &c) {
  k_step_tail<kTailWideThreads, kTailWideThreads, 2>
      <<<g_tail_wide_per_sm * c.sm_count, kTailWideThreads, 0, c.stream>>>(c.hdr, c.active, c.sched);
  return cudaGetLastError();
}

}  // namespace psl
