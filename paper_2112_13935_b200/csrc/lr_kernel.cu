// Softmax regression 784 -> 10, batch 1: which kernel runs a launch of round-tasks.
//
// Up to about half an SM's share of the launch per round-task, the round's serial chain sets the time: a cluster of two or
// four CTAs per round-task (lr_chain_kernel.cu).  With more round-tasks than that, a cluster would leave some of them
// waiting for SMs: one CTA each (lr_block_kernel.cu), and with more round-tasks than SMs its two-per-SM shape.
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

cudaError_t launch_lr_rounds(const RoundLaunch& p, cudaStream_t s) {
  if (p.n_tasks == 0) return cudaSuccess;
  static int sm_count[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < 64;
  int sms = known ? sm_count[dev] : 0;
  if (!sms) {
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (known) sm_count[dev] = sms;
  }
  const bool crowded = p.n_tasks > (uint32_t)sms || p.crowded_hint;
  if (crowded) return launch_lr_block_rounds(p, true, s);
  // (clusters do not straddle GPCs: one SM in sixteen is not counted on)
  if (p.n_tasks * 2 > (uint32_t)(sms - sms / 16)) return launch_lr_block_rounds(p, false, s);
  return launch_lr_chain_rounds(p, (uint32_t)sms, s);
}

}  // namespace aet
