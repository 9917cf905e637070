// Softmax regression 784 -> 10, batch 1: which kernel runs a launch of round-tasks.
//
// As long as the device runs a cluster for every round-task at once, the round's serial chain sets the time: eight or six CTAs per
// round-task, one of which does nothing but walk it (lr_relay_kernel.cu; up to 15 round-tasks, and up to 22 with rounds above 64 samples:
// 16 clients, three rounds of 32 / 64 / 128 / 400 samples each 54 / 63 / 66 / 142 us on six, 45 to 53 / 59 to 72 / 70 to 84 / 164 to 195 on four, by
// the step size); four or two that do everything alike (lr_chain_kernel.cu; up to 74).  With more round-tasks than that, a cluster would leave some of them waiting for SMs: one CTA each
// (lr_block_kernel.cu), and with more round-tasks than SMs its two-per-SM shape.  Rounds of 400
// samples: 33 clients 88 us on four CTAs, 98 on two; 74 clients 113 us on two, 161 on one.
#include <cuda_runtime.h>

#include "aet_kernels.h"
#include "lr_common.cuh"

namespace aet {
namespace {

using namespace lr;

// Exercises the give-up path of the bounded wait without any faulty hardware:
// an mbarrier that nothing ever arrives on is polled `max_polls` times, then the
// CTA flags `status` exactly as a round kernel does and returns normally.
__global__ void wait_probe_kernel(uint32_t* status, uint32_t max_polls) {
  __shared__ __align__(8) uint64_t never;
  if (threadIdx.x == 0) {
    mbar_init(&never, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const bool landed = mbar_wait_limit(&never, 0, max_polls);
  if (__syncthreads_or(!landed) && threadIdx.x == 0) atomicOr(status, 1u);
}

}  // namespace

cudaError_t launch_wait_probe(uint32_t* status, uint32_t max_polls, cudaStream_t s) {
  wait_probe_kernel<<<1, 32, 0, s>>>(status, max_polls);
  return cudaGetLastError();
}

LrChoice choose_lr_kernel(uint32_t n_tasks, uint32_t longest, bool by_value, const uint32_t (&at_once)[9]) {
  const bool eights = n_tasks <= at_once[8], fours = n_tasks <= at_once[4];
  const bool sixes = !eights && n_tasks <= at_once[6] && longest > 64;
  if (eights || sixes) return {LrKernel::kRelay, eights ? 8u : 6u};
  // descriptors in the launch: a kernel on clusters, whichever there is
  if (by_value || n_tasks <= at_once[2]) return {LrKernel::kChain, fours ? 4u : 2u};
  return {n_tasks <= at_once[1] ? LrKernel::kBlock : LrKernel::kCrowded, 1};
}

cudaError_t launch_lr_rounds(const RoundLaunch& p, cudaStream_t s) {
  if (p.n_tasks == 0) return cudaSuccess;
  uint32_t at_once[9];
  if (const cudaError_t e = clusters_at_once(at_once)) return e;
  const LrChoice c = choose_lr_kernel(p.wave_tasks ? p.wave_tasks : p.n_tasks, p.longest, p.by_value != 0, at_once);
  if (c.kernel == LrKernel::kRelay) return launch_lr_relay_rounds(p, c.cluster, s);
  if (c.kernel == LrKernel::kChain) return launch_lr_chain_rounds(p, c.cluster, s);
  return launch_lr_block_rounds(p, c.kernel == LrKernel::kCrowded, s);
}

}  // namespace aet
