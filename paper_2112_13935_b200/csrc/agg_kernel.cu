// Server side: ordered aggregation of the triggered update sums.
//
// Algorithm 3, Receive: "w = w - eta_k * U; H_v = H_v + 1", applied in the
// order the simulated-time schedule fixes; wherever a later round starts from
// the model after update k the running value is also stored as that round's
// start snapshot (this replaces a separate broadcast copy into client slots).
//
// A CTA has a slice of 128 parameters and a range of consecutive updates: it
// fetches the slice of all its update sums at once (asynchronous copies into
// shared memory, one row per warp instruction), its four thread groups sum
// -eta_k U_k over a quarter of the range each, and with everything that comes
// before known every group walks its quarter in order, keeping the parameter
// in a register.  Long ranges are cut over a cluster of up to eight CTAs, which
// exchange their totals through distributed shared memory.  The result is the
// paper's sequential rule up to fp32 re-association across quarters, and
// identical from run to run.
// What bounds it: L2 (every update sum read once, every snapshot written once)
// and the latency of one such fetch.  Two passes of eight-deep walks over the
// range (group totals, then the walk) took 24 us cold for 700 updates of 7,850
// parameters; this takes 6.5 to 19 us for 680 to 1,000.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "aet_kernels.h"
#include "mma_common.cuh"

namespace aet {
namespace {

constexpr int kSlice = 128;                 // parameters per CTA
constexpr int kSub = 4, kAggThreads = kSlice * kSub;
constexpr int kMostRows = 384;              // updates per CTA: 192 KB of shared memory
constexpr int kMostGroups = 8;

struct AggSmem {   // behind it rows[n][kSlice]
  float sub[kSub][kSlice], total[kSlice];
  float eta[kMostRows];
  int32_t slot[kMostRows];
  uint32_t row[kMostRows];
};

// Launched with programmatic stream serialisation: the CTAs may become resident while the kernel ahead of them in the
// stream (the round kernel) is draining; before griddepcontrol.wait they read descriptors only, which the host wrote.
__global__ void __launch_bounds__(kAggThreads) apply_updates_kernel(ApplyLaunch p, uint32_t per) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  AggSmem& sm = *reinterpret_cast<AggSmem*>(smem_raw);
  float* rows = reinterpret_cast<float*>(smem_raw + sizeof(AggSmem));
  // The round kernel behind this one may start its set-up: it reads nothing this grid writes before its own wait.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, j = tid & (kSlice - 1), q = tid / kSlice;
  const uint32_t lo = min(p.hi, p.lo + blockIdx.y * per), n = min(p.hi, lo + per) - lo;
  const uint32_t col = blockIdx.x * kSlice, at = col + j;
  for (uint32_t k = tid; k < n; k += kAggThreads) {
    const ApplyDesc d = p.applies[lo + k];
    sm.eta[k] = d.eta; sm.slot[k] = d.snap_slot; sm.row[k] = d.u_row;
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float w = at < p.n_params ? p.w[at] : 0.f;
  if (col + 4 * lane < p.stride)   // (rows are padded to a multiple of 32 floats)
    for (uint32_t k = warp; k < n; k += kAggThreads / 32)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                   ::"r"((uint32_t)__cvta_generic_to_shared(rows + k * kSlice + 4 * lane)), "l"(p.U + (size_t)sm.row[k] * p.stride + col + 4 * lane) : "memory");
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const uint32_t quarter = (n + kSub - 1) / kSub, r0 = min(n, q * quarter), r1 = min(n, r0 + quarter);
  {
    float s = 0.f;
    for (uint32_t k = r0; k < r1; ++k) s = fmaf(-sm.eta[k], rows[k * kSlice + j], s);
    sm.sub[q][j] = s;
  }
  __syncthreads();
  if (gridDim.y > 1) {
    if (q == 0) sm.total[j] = (sm.sub[0][j] + sm.sub[1][j]) + (sm.sub[2][j] + sm.sub[3][j]);
    mma::cluster_sync();
    for (uint32_t r = 0; r < blockIdx.y; ++r) w += mma::ld_peer(mma::peer_addr((uint32_t)__cvta_generic_to_shared(&sm.total[j]), r));
  }
  for (int s = 0; s < q; ++s) w += sm.sub[s][j];
  if (at < p.n_params) {
    for (uint32_t k = r0; k < r1; ++k) {
      w = fmaf(-sm.eta[k], rows[k * kSlice + j], w);
      if (sm.slot[k] >= 0) p.snaps[(size_t)sm.slot[k] * p.stride + at] = w;
    }
    if (q == kSub - 1 && blockIdx.y + 1 == gridDim.y) {
      p.w[at] = w;
      // the server model after this range: a non-finite entry (a NaN or an overflow that came in
      // through a client's rows or step size) is reported, never trapped on
      if (p.status && !isfinite(w)) atomicOr(p.status, 2u);
    }
  }
  // history map and apply log: one thread per update of the range
  if (blockIdx.x == 0)
    for (uint32_t k = tid; k < n; k += kAggThreads) {
      const ApplyDesc d = p.applies[lo + k];
      ApplyRec r;
      r.client = d.client; r.round = d.round; r.seq = lo + k;
      r.h_after = atomicAdd(&p.H[d.client], 1u) + 1u;
      p.log[lo + k] = r;
    }
  if (gridDim.y > 1) mma::cluster_sync();   // nobody leaves while its total may still be read
}

__global__ void copy_and_zero_kernel(float4* dst, const float4* src, size_t n4, uint32_t* zero, size_t nz) {
  const size_t step = (size_t)gridDim.x * blockDim.x, i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (size_t i = i0; i < n4; i += step) dst[i] = src[i];
  for (size_t i = i0; i < nz; i += step) zero[i] = 0;
}

// What bounds it: the host link, 50 GB/s read from here against 55 by the copy engine; but nothing is paid per array, and with
// the next client's CTAs already waiting little between clients: 64 clients of 627 KB, create to event log, 1.93 -> 1.47 ms
// (1.57 without the early launch).  A bf16 client needs no fp32 copy on the device.
template <bool BF>
__global__ void __launch_bounds__(256) fetch_client_kernel(const float4* __restrict__ x, void* __restrict__ dx, size_t n4, const int32_t* __restrict__ y,
                                                            int32_t* __restrict__ dy, uint32_t n) {
  const size_t step = (size_t)gridDim.x * blockDim.x, i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next client's CTAs come up meanwhile ...
  asm volatile("griddepcontrol.wait;" ::: "memory");               // ... and wait here for everything before them
  for (size_t i = i0; i < n; i += step) dy[i] = y[i];
  for (size_t i = i0; i < n4; i += 4 * step) {
    float4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i + q * step < n4) v[q] = x[i + q * step];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (i + q * step >= n4) continue;
      if (BF) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v[q].x, v[q].y), b = __floats2bfloat162_rn(v[q].z, v[q].w);
        static_cast<uint2*>(dx)[i + q * step] = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      } else {
        static_cast<float4*>(dx)[i + q * step] = v[q];
      }
    }
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, size_t n) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t step = (size_t)gridDim.x * blockDim.x;
  for (; i < n; i += step) dst[i] = __float2bfloat16_rn(src[i]);
}

constexpr int kRingThreads = 128;
// Peer-to-peer ring: Receive at every node (Algorithm 3: w_c = w_c - eta_k * U) for the sums that
// reached it, preceded by the node's own sum of the round it has just finished.  One y-block per node
// whose model moves; a thread keeps its parameter in a register and walks the node's short list.
__global__ void __launch_bounds__(kRingThreads) ring_apply_kernel(RingApplyLaunch p) {
  // (launched as apply_updates_kernel is, and for the same reasons)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t j = blockIdx.x * kRingThreads + threadIdx.x;
  if (j >= p.n_params) return;
  const RingApplyDesc a = p.applies[p.lo + blockIdx.y];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float* wp = p.node_w + (size_t)a.node * p.stride + j;
  float w = *wp;
  for (uint32_t k = 0; k < a.op_cnt; ++k) {
    const RingOp op = p.ops[a.op_off + k];
    w = fmaf(-op.eta, p.U[(size_t)op.u_row * p.stride + j], w);
  }
  *wp = w;
  if (p.status && !isfinite(w)) atomicOr(p.status, 2u);
}

// Debug pass over a client's data set as it is loaded: a label outside [0, n_classes) sets bit 2
// of *status, a non-finite pixel bit 1.  Nothing is trapped on; the host turns the bits into
// AET_ERR_STATE / AET_ERR_NUMERIC at its next synchronising call.
__global__ void validate_data_kernel(const float* __restrict__ x, const int32_t* __restrict__ y, uint32_t n,
                                     uint32_t dim, uint32_t n_classes, uint32_t* status) {
  const size_t step = (size_t)gridDim.x * blockDim.x;
  uint32_t bad = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step)
    if ((uint32_t)y[i] >= n_classes) bad |= 4u;
  if (x)
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < (size_t)n * dim; i += step)
      if (!isfinite(x[i])) bad |= 2u;
  if (bad) atomicOr(status, bad);
}

}  // namespace

cudaError_t launch_validate_data(const float* x, const int32_t* y, uint32_t n, uint32_t dim, uint32_t n_classes,
                                 uint32_t* status, cudaStream_t s) {
  if (!n) return cudaSuccess;
  size_t blocks = ((size_t)n * dim + 255) / 256;
  if (blocks > 148 * 8) blocks = 148 * 8;
  validate_data_kernel<<<(unsigned)blocks, 256, 0, s>>>(x, y, n, dim, n_classes, status);
  return cudaGetLastError();
}

cudaError_t launch_ring_apply(const RingApplyLaunch& p, cudaStream_t s) {
  if (p.hi <= p.lo) return cudaSuccess;
  const uint32_t blocks = (p.n_params + kRingThreads - 1) / kRingThreads;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks, p.hi - p.lo, 1);
  cfg.blockDim = dim3(kRingThreads, 1, 1);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ring_apply_kernel, p);
}

cudaError_t launch_apply_updates(const ApplyLaunch& p0, cudaStream_t s) {
  static bool opted_in[64] = {};   // more than 48 KB of shared memory has to be asked for once per device
  int dev = 0;
  cudaError_t de = cudaGetDevice(&dev);
  if (de != cudaSuccess) return de;
  const bool known = dev >= 0 && dev < 64;
  if (!known || !opted_in[dev]) {
    de = cudaFuncSetAttribute(apply_updates_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(AggSmem) + kMostRows * kSlice * sizeof(float)));
    if (de != cudaSuccess) return de;
    if (known) opted_in[dev] = true;
  }
  ApplyLaunch p = p0;
  const uint32_t slices = (p.n_params + kSlice - 1) / kSlice;
  for (uint32_t lo = p0.lo; lo < p0.hi; lo += kMostRows * kMostGroups) {
    p.lo = lo;
    p.hi = min(p0.hi, lo + kMostRows * kMostGroups);
    const uint32_t n = p.hi - p.lo;
    // a CTA per 64 updates: a quarter of them is a walk as long as the exchange of totals takes
    uint32_t groups = 1;
    while (groups < (uint32_t)kMostGroups && n > 64 * groups) groups *= 2;
    const uint32_t per = (n + groups - 1) / groups;
    const size_t smem = sizeof(AggSmem) + (size_t)per * kSlice * sizeof(float);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = groups;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(slices, groups, 1);
    cfg.blockDim = dim3(kAggThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = groups > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, apply_updates_kernel, p, per);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_copy_and_zero(float* dst, const float* src, size_t n, uint32_t* zero, size_t nz, cudaStream_t s) {
  size_t blocks = (n / 4 + nz + 255) / 256;
  if (blocks > 148 * 4) blocks = 148 * 4;
  copy_and_zero_kernel<<<(unsigned)blocks, 256, 0, s>>>(reinterpret_cast<float4*>(dst), reinterpret_cast<const float4*>(src), n / 4, zero, nz);
  return cudaGetLastError();
}

cudaError_t launch_fetch_client(const float* x, void* dx, bool bf16, size_t n4, const int32_t* y, int32_t* dy, uint32_t n, cudaStream_t s) {
  size_t blocks = (n4 + 4 * 256 - 1) / (4 * 256);
  if (blocks > 148) blocks = 148;
  if (!blocks) blocks = 1;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks, 1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return bf16 ? cudaLaunchKernelEx(&cfg, fetch_client_kernel<true>, x4, dx, n4, y, dy, n) : cudaLaunchKernelEx(&cfg, fetch_client_kernel<false>, x4, dx, n4, y, dy, n);
}

cudaError_t launch_to_bf16(const float* src, void* dst, size_t n, cudaStream_t s) {
  if (!n) return cudaSuccess;
  size_t blocks = (n + 255) / 256;
  if (blocks > 148 * 16) blocks = 148 * 16;
  to_bf16_kernel<<<(unsigned)blocks, 256, 0, s>>>(src, reinterpret_cast<__nv_bfloat16*>(dst), n);
  return cudaGetLastError();
}

}  // namespace aet
