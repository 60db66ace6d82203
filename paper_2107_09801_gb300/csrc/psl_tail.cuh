// psl_tail.cuh -- the step after the neighbourhood score for batches of short walks
// (arXiv 2107.09801, Algorithm 1): one block per walk runs selection, exact re-check,
// decision and update back to back.  Compiled for blocks of one warp (psl_tail.cu) and of
// eight (psl_tail_wide.cu), in translation units of their own.
#pragma once
#include <cstdint>

#include "psl_device.cuh"
#include "psl_internal.h"
#include "psl_step.cuh"

namespace psl {

// NT: threads per block; BOUND, PER_SM: the register bound (see the instances).  Every phase below
// is written for any block size; the block-wide selection takes the place of one warp's.
template <int NT, int BOUND, int PER_SM>
__global__ void __launch_bounds__(BOUND, PER_SM) k_step_tail(WalkDev *hdr, const uint32_t *active, Schedule *sched) {
  // The walk's header lives in shared memory for the whole of its step: the phases below
  // read and write its fields one after another (one block owns the walk, nothing else runs
  // on it meanwhile), so a dependent chain of header accesses costs shared-memory latency
  // instead of L2 latency.  Copied in before, written back after.
  __shared__ WalkDev sW;
  static_assert(sizeof(WalkDev) % 8 == 0 && alignof(WalkDev) <= 8, "the header copies in 8-byte words");
  constexpr int kHdrWords = (int)(sizeof(WalkDev) / 8);
  // the neighbourhood kernel of this step has finished: rearm its work counter
  if (blockIdx.x == 0 && threadIdx.x == 0) sched->hot_next = 0;
  const bool exact = sched->alpha2 != 0;  // the closed form kept every neighbour's exact Delta F
  for (uint32_t a = blockIdx.x; a < sched->nactive; a += gridDim.x) {
    WalkDev &G = hdr[active[a]];
    __syncthreads();  // the previous walk's shared buffers and header copy are free
    if (G.status != kRunning) continue;  // one reading for the block: nothing below changes it before it is read
    for (int q = (int)threadIdx.x; q < kHdrWords; q += (int)blockDim.x)
      reinterpret_cast<uint2 *>(&sW)[q] = reinterpret_cast<const uint2 *>(&G)[q];
    __syncthreads();
    WalkDev &W = sW;
    if constexpr (NT == 32)
      select_warp(W);
    else
      select_one(W);
    __syncthreads();  // candidates, bound and window PSL are visible to the block
    const uint32_t nslots = min(W.ncand, (uint32_t)kQcap);
    for (uint32_t qslot = 0; qslot < nslots; qslot++) {
      __syncthreads();
      recheck_one<true, kRcBoth>(W, 0, qslot, exact);
    }
    __syncthreads();  // re-check partials are visible
    decide_one(W);
    __syncthreads();  // the decision (mode, k*, flips, next exponent) is visible
    if (W.mode == kModeMove)
      apply_move_dispatch(W, 0);
    else
      apply_one(W, 0);
    __syncthreads();
    for (int q = (int)threadIdx.x; q < kHdrWords; q += (int)blockDim.x)
      reinterpret_cast<uint2 *>(&G)[q] = reinterpret_cast<const uint2 *>(&sW)[q];
  }
}

}  // namespace psl
