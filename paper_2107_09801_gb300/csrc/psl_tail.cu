// psl_tail.cu -- the short walks' step tail in blocks of one warp, for batches of many walks.
#include "psl_tail.cuh"

namespace psl {

// Blocks of one warp: each walk's chain of phases is bound by latency, so the more walks an
// SM holds at once the better.  Measured at L = 1023 x 4096: 256 threads, 3 blocks per SM
// 0.230 ms per step; 64 threads at 80 registers, 12 blocks 0.108 ms (then, after the shared
// header copy, 0.074 ms); 64 registers, 16 blocks 0.067 ms; one warp, 32 blocks 0.063 ms.
// (The register bound stays that of 64-thread blocks: bounding for 32-thread blocks makes
// the compiler spill a kilobyte.)
constexpr int kTailThreads = 32;

static uint32_t g_tail_per_sm = 4;

cudaError_t prepare_tail_kernel() {
  int nb = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_step_tail<kTailThreads, 64, 16>, kTailThreads, 0);
  g_tail_per_sm = (uint32_t)(nb > 0 ? nb : 1);
  return e == cudaSuccess ? prepare_tail_wide_kernel() : e;
}

cudaError_t launch_step_tail(const LaunchCtx &c) {
  if (c.tail_wide) return launch_step_tail_wide(c);
  k_step_tail<kTailThreads, 64, 16><<<g_tail_per_sm * c.sm_count, kTailThreads, 0, c.stream>>>(c.hdr, c.active, c.sched);
  return cudaGetLastError();
}

}  // namespace psl
