// Launch interfaces of the device kernels (plain structs, no library types).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "aet_schedule.h"

namespace aet {

// Device view of one client's local data set D_c.
struct ClientData {
  const void* x;     // [n, D] row-major; fp32, or bf16 when precision == 1
  const int32_t* y;  // [n]
  uint32_t n;
  uint32_t pad;
};

// What a local-SGD kernel leaves behind when a round's last sample is done:
// the device-side record of the event trigger (message (c, U_i, i)).
struct TriggerRec { uint32_t client, round, samples_done, flags; };
// What the aggregation kernel leaves behind per applied update.
struct ApplyRec { uint32_t client, round, h_after, seq; };

// Rows of the snapshot / update-sum / work arrays are `stride` floats apart
// (n_params rounded up to a multiple of 32, so every row is 128-byte aligned).
struct RoundLaunch {
  const TaskDesc* tasks;         // device
  const InflightRef* inflight;   // device
  const ClientData* clients;     // device, [n_clients]
  const uint64_t* sample_keys;   // device, [n_clients]
  const float* snaps;            // [n_snap, stride] models rounds start from
  float* U;                      // [n_u_rows, stride] update sums, row = TaskDesc::u_row
  float* w_end;                  // optional [n_events, stride] end-of-round models
  TriggerRec* trig;              // [n_events], row = seq
  uint32_t* status;              // optional: bit 0 set if a bounded device wait gave up,
                                 // bit 2 if a debug index check failed (see debug_checks)
  uint32_t debug_checks;         // non-zero: sample indices and row numbers are range-checked before use
  size_t stride;
  uint32_t task_begin, n_tasks;
  uint32_t longest;              // samples of the longest round-task of a launch of few (0: many, or not known)
  uint32_t n_u_rows, n_snap;     // extents of U and snaps (for the debug checks)
  uint32_t wave_tasks;           // non-zero: pick the kernel a launch of so many round-tasks would get, however few
                                 // this one holds (single-task parity runs of the regression)
  // One round-task with its descriptors in the launch itself (n_tasks 1, no sums in flight; lr_relay_kernel and lr_chain_kernel):
  // nothing has to be in device memory beforehand, and rows and labels are read behind the device-side wait too.
  uint32_t by_value;
  TaskDesc one_task;
  ClientData one_client;
  uint64_t one_key;
  uint32_t step_by_step;         // non-zero: the recurrence of a block is always walked step by step
  float l2;
  // Failure checks, lr_relay_kernel only (0 in every run): 1 + the CTA of the cluster whose copies are left out, or, if that is the
  // walker, whose couplings are; and how often every wait polls then.
  uint32_t lose, max_polls;
};

// How many clusters of 1 to 8 CTAs with an SM each the current device runs at once, 0 where it runs none (see device_info.cu).
cudaError_t clusters_at_once(uint32_t cluster, uint32_t* out);
cudaError_t clusters_at_once(uint32_t (&out)[9]);   // all of them, [CTAs], with one question to the runtime

// One CTA waits (at most max_polls polls) on a barrier nobody signals, then sets bit 0 of *status.
cudaError_t launch_wait_probe(uint32_t* status, uint32_t max_polls, cudaStream_t s);

// Softmax regression 784 -> 10, batch 1; the kernel is picked by how many round-tasks the launch holds.  Asynchronous on s; may start under the tail of the previous kernel in s
// (programmatic stream serialisation) and waits on the device before reading that kernel's output.
cudaError_t launch_lr_rounds(const RoundLaunch& p, cudaStream_t s);
// ... the choice: which kernel, on how many CTAs per round-task.  at_once[n]: clusters of n CTAs the device runs at once.
enum class LrKernel : uint32_t { kRelay, kChain, kBlock, kCrowded };
struct LrChoice { LrKernel kernel; uint32_t cluster; };
LrChoice choose_lr_kernel(uint32_t n_tasks, uint32_t longest, bool by_value, const uint32_t (&at_once)[9]);
// a cluster of eight or six CTAs per round-task (see lr_relay_kernel.cu), of four or two (lr_chain_kernel.cu)
cudaError_t launch_lr_relay_rounds(const RoundLaunch& p, uint32_t cluster, cudaStream_t s);
cudaError_t launch_lr_chain_rounds(const RoundLaunch& p, uint32_t cluster, cudaStream_t s);
// one CTA per round-task; crowded: two CTAs per SM (see lr_block_kernel.cu)
cudaError_t launch_lr_block_rounds(const RoundLaunch& p, bool crowded, cudaStream_t s);

struct MlpShape {
  uint32_t n_layers, dims[8], batch, precision;
  uint32_t cluster;              // CTAs per round-task
};
struct MlpLaunch {
  RoundLaunch r;
  MlpShape shape;
  float* work;                   // [n_clients, stride] client's current model
  float* act;                    // per-task activation scratch
  size_t act_stride;             // floats per task
};
cudaError_t launch_mlp_rounds(const MlpLaunch& p, cudaStream_t s);
size_t mlp_act_floats(const MlpShape& shape);
uint32_t mlp_pick_cluster(const MlpShape& shape, uint32_t n_clients);
const char* mlp_check_shape(const MlpShape& shape);  // null if the kernel can run it
// bf16 shapes whose update sum of W_0 is (W_start - W_end) / eta instead of a sum over the iterations: large first layers with
// whole 128-row chunks per CTA, where a second fp32 array of W_0's size would have to be streamed or kept on the chip beside it.
// The quotient is only as good as 2^-24 |w| / eta (1e-3 of U's rms at eta 5e-4 and one iteration, a sum 5e-8): no other shape
// is given to a kernel that derives.
bool mlp_derives_w0(const MlpShape& shape);
// bf16 D0-256-(128-)C models, batch 32 or 64: the first layer streams through a cluster (see mlp_wide_kernel.cu)
bool mlp_wide_eligible(const MlpShape& shape);
cudaError_t launch_mlp_wide_rounds(const MlpLaunch& p, cudaStream_t s);
// minibatches of up to 64 samples, first hidden layer of at most 128 units (bf16: 256): the first layer stays on the chip,
// spread over a cluster (see mlp_mma_kernel.cu)
bool mlp_mma_eligible(const MlpShape& shape);
cudaError_t launch_mlp_mma_rounds(const MlpLaunch& p, cudaStream_t s);
// bf16 models whose first layer fits the tensor-core kernel (tcgen05 + TMEM)
bool mlp_tc_eligible(const MlpShape& shape);
cudaError_t launch_mlp_tc_rounds(const MlpLaunch& p, cudaStream_t s);

// Small convolutional classifier (two 5x5 convolutions with average pooling, three dense layers):
// dims = {side, c_in, c1, c2, f1, f2, classes}; the whole model stays in shared memory for the round.
struct CnnShape { uint32_t dims[8], batch; };
struct CnnLaunch {
  RoundLaunch r;
  CnnShape shape;
  float* act;                    // per-task activation scratch
  size_t act_stride;             // floats per task
  uint32_t stage_rows = 0;       // set by the launcher: the CTA's minibatch rows fit in shared memory beside the model,
  uint32_t stage_acts = 0;       //   and so do its activations other than the first convolution's maps
};
uint32_t cnn_n_params(const CnnShape& s);
size_t cnn_act_floats(const CnnShape& s);
const char* cnn_check_shape(const CnnShape& s);   // null if the kernel can run it
cudaError_t launch_cnn_rounds(const CnnLaunch& p, cudaStream_t s);
// The LeNet shape, minibatches of up to 24 samples, on clusters of 8 or 4 CTAs (see cnn_mma_kernel.cu); 0: not eligible
cudaError_t cnn_mma_cluster(const CnnShape& s, uint32_t n_tasks, uint32_t* cluster);
cudaError_t launch_cnn_mma_rounds(const CnnLaunch& p, uint32_t cluster, cudaStream_t s);

// Ordered aggregation: for seq in [lo, hi): w -= eta_seq * U[seq]; keep a copy
// where a later round starts from it; bump H and log the apply.
struct ApplyLaunch {
  const ApplyDesc* applies;  // device, indexed by seq
  const float* U;
  float* snaps;
  float* w;                  // server model [stride], before and after the range
  uint32_t* H;               // [n_clients]
  ApplyRec* log;             // [n_events]
  uint32_t* status;          // optional: bit 1 set if the model after the range is not finite
  size_t stride;
  uint32_t n_params, lo, hi;
};
cudaError_t launch_apply_updates(const ApplyLaunch& p, cudaStream_t s);

// Peer-to-peer ring: the models of the nodes listed in applies[lo, hi) take their operations.
struct RingApplyLaunch {
  const RingApplyDesc* applies;  // device
  const RingOp* ops;             // device
  const float* U;                // [n_tasks, stride]
  float* node_w;                 // [n_nodes, stride]
  uint32_t* status;              // optional: bit 1 set if a model is not finite afterwards
  size_t stride;
  uint32_t n_params, lo, hi;
};
cudaError_t launch_ring_apply(const RingApplyLaunch& p, cudaStream_t s);

// Debug checks at load time: labels in range (else bit 2 of *status), pixels finite (else bit 1; x may be null).
cudaError_t launch_validate_data(const float* x, const int32_t* y, uint32_t n, uint32_t dim, uint32_t n_classes,
                                 uint32_t* status, cudaStream_t s);

#if defined(__CUDACC__)
// Debug check at the top of every round kernel (all threads of a CTA, and all CTAs of a cluster,
// take the same decision): are the rows and slots the task names inside the arrays?  If not,
// bit 2 of *status is set and the caller skips the task without touching memory.
__device__ __forceinline__ bool debug_task_ok(const RoundLaunch& p, const TaskDesc& t) {
  if (!p.debug_checks) return true;
  bool ok = t.u_row < p.n_u_rows && t.snap_slot < p.n_snap;
  for (uint32_t f = 0; ok && f < t.inflight_cnt; ++f) ok = p.inflight[t.inflight_off + f].row < p.n_u_rows;
  if (!ok && threadIdx.x == 0 && p.status) atomicOr(p.status, 4u);
  return ok;
}
// A round without a single iteration (a node the Setup split of Algorithm 2 gave nothing in this
// round): Algorithm 3 still sends (c, U_i, i) after the empty inner loop, with U_i = 0.  One CTA
// writes the zero update sum, the unchanged model where the caller wants it, and the trigger record.
__device__ __forceinline__ void publish_empty_round(const RoundLaunch& p, const TaskDesc& t, uint32_t n_params) {
  float* U = p.U + (size_t)t.u_row * p.stride;
  const float* snap = p.snaps + (size_t)t.snap_slot * p.stride;
  for (uint32_t i = threadIdx.x; i < n_params; i += blockDim.x) {
    U[i] = 0.f;
    if (p.w_end) {
      float w = snap[i];
      for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
        const InflightRef ref = p.inflight[t.inflight_off + f];
        w = fmaf(-ref.eta, p.U[(size_t)ref.row * p.stride + i], w);
      }
      p.w_end[(size_t)t.u_row * p.stride + i] = w;
    }
  }
  if (threadIdx.x == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = 0; rec.flags = 1;
    p.trig[t.seq] = rec;
  }
}
#endif

// dst[0, n) = src (n a multiple of 4), zero[0, nz) = 0 (nz words): what a run or a reset sets up, in one launch
cudaError_t launch_copy_and_zero(float* dst, const float* src, size_t n, uint32_t* zero, size_t nz, cudaStream_t s);

// A client's rows (4 n4 values from a 16-byte boundary on; bf16: rounded on the way) and labels out of page-locked host
// memory the device can address, in one launch.
cudaError_t launch_fetch_client(const float* x, void* dx, bool bf16, size_t n4, const int32_t* y, int32_t* dy, uint32_t n, cudaStream_t s);

// bf16 conversion of a client's rows at load time (precision 1).
cudaError_t launch_to_bf16(const float* src, void* dst, size_t n, cudaStream_t s);

}  // namespace aet
