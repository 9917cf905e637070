// Local-SGD round of one client for the bf16-operand MLPs D0 -> 256 -> (128 ->) C, C <= 16, minibatch 32 or 64: the first
// layer's fp32 master streams through every warp's registers once per SGD iteration.
//
// Algorithm 3, MainComputeNode, inner loop with xi a minibatch (mean gradient; w_c -= eta_i g; U_i += g).  Rounding points
// as everywhere in the bf16 path: inputs once at load, W_l on every read of the fp32 master, hidden activations after
// bias + ReLU, dZ_l before the two backward products; logits, softmax, bias gradients, master updates in fp32.
//
// A cluster of CL CTAs of 16 warps per round-task; a CTA has a range of the inputs, warp w the hidden units 16 w .. 16 w + 15.
// One pass over the CTA's inputs, 16 at a time, does the backward product of an iteration and the forward product of the
// next: the thread fetches its 8 entries of W_0 (four units ahead), forms their gradient dZ_0^T X (m16n8k16, the accumulator
// fragment is the thread's own entries), updates, writes them back and multiplies the new bf16 values - already the operand
// fragment - with the next minibatch.  No thread waits for another inside a pass but for the input columns: chunks of 32
// columns of both minibatches come through a ring of three (cp.async, counted by mbarriers).  The master lies in
// the client's work row in the order the threads read it, 512 contiguous bytes per warp instruction; the first units (and
// W_1's master) stay in tensor memory, used as 128 registers per thread.  The first pass of a round reads the start model,
// the last writes the update sums.
// Between passes: a warp's part of Z_0^T goes to the CTA that owns its hidden units (st.async), which adds the parts in
// rank order, applies bias and ReLU and sends bf16 A_0 to everybody; the narrow layers run in every CTA alike (same inputs,
// same order: the same bits).  Memory is reused without cluster barriers: parts are sent only after every peer's warps have
// said that they are done with what lies there.
//
// The update sum of W_0 is (W_start - W_end) / eta (w -= eta g and U += g in the same step; mlp_derives_w0 says for which
// shapes), W_1's likewise at minibatch 64; at 32 tensor memory holds it, and W_0 streams from its first unit on.  The class layer's and the
// biases' are accumulated.
//
// What bounds it: with enough clients the shared memory pipe, busy nine cycles of ten during a pass (every warp reads the fragments of
// both minibatches' columns: 32 wavefronts per unit; the stream itself takes 16), 1,150 cycles per unit; with few, the warp-level
// tensor rate (16 instructions of 8 cycles per 16 x 16 entries and scheduler) and the narrow layers.
// A pass is not bound by HBM any more: W_0 is read and written once per iteration, 6.3 MB per client at D0 = 3072, and since every pass
// goes the other way round than the one before it a quarter of that stays in L2 (DRAM traffic of two waves 938 -> 706 MB).
// Measured, 64 clients of 3072-256-128-10, 30 rounds: 103.3 -> 95.8 ms with units four ahead in shared memory for all cluster widths
// (before: two in registers, fed from two in shared memory, which a unit's wait emptied); tcgen05 products on bf16 tiles
// that every iteration rebuilt in shared memory from the same stream took 181 ms.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "aet_kernels.h"
#include "aet_rng.h"
#include "lr_common.cuh"
#include "mma_common.cuh"

namespace aet {
namespace {

using lr::kWaitLimit;
using lr::mbar_arrive;
using lr::mbar_expect_tx;
using lr::mbar_init;
using lr::mbar_wait;
using lr::smem_addr;
using mma::ldmatrix4;
using mma::ldmatrix4t;
using mma::mma_bf16;
using mma::pack_bf16;
typedef __nv_bfloat16 bf16;

constexpr int kWarps = 16, kThreads = kWarps * 32;
constexpr int kH0 = 256, kH1 = 128, kMaxC = 16;
constexpr int kP0 = kH0 + 8, kP1 = kH1 + 8, kPz = 24, kPx = 40;   // row pitches: the rows of a fragment load hit different banks
constexpr int kRing = 3, kChunk = 32;                              // chunks of input columns in shared memory, columns of a chunk
constexpr int kB1 = kH0, kB2 = kH0 + kH1, kNb = kH0 + kH1 + 16;    // places of the layers' biases

// ---- a thread's own words in tensor memory, eight at a time ------------------------------------------------------------
struct Own {
  uint32_t tmem;
  __device__ __forceinline__ void load(int group, float (&v)[8]) const {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(tmem + 8u * group) : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
  }
  __device__ __forceinline__ void store(int group, const float (&v)[8]) const {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(tmem + 8u * group), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
                   "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])) : "memory");
  }
  __device__ __forceinline__ void store_wait() const { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
};

template <int BT, bool MID>
struct Lay {   // shared memory, in bytes
  static constexpr int Bp = 8 * BT, K2 = MID ? kH1 : kH0, kPw2 = K2 + 8;
  static constexpr int w1 = 0, a0 = w1 + (MID ? kH1 * kP0 * 2 : 0);
  // dZ_0, dZ_1, A_1: dead during a pass, whose parts of Z_0 come in there: up to 7 / 8 of 16 tiles of 16 x Bp
  static constexpr int z0 = a0 + Bp * kP0 * 2, z1 = z0 + Bp * kP0 * 2, a1 = z1 + (MID ? Bp * kP1 * 2 : 0), dead_end = a1 + (MID ? Bp * kP1 * 2 : 0);
  static constexpr int in_end = z0 + 14 * BT * 512;
  static constexpr int kSlots = 4, stage_end = z0 + kSlots * kWarps * 1024;   // units of W_0 on their way in, from z0 on
  static constexpr int part = MID ? z1 : z0;   // the class layer's partial sums: before dZ of the layer below is written
  static constexpr int top = dead_end > in_end ? dead_end : in_end;
  static constexpr int w2 = top > stage_end ? top : stage_end, logit = w2 + 16 * kPw2 * 4, z2 = logit + Bp * 17 * 4;
  static constexpr int bias = z2 + Bp * kPz * 2, ub = bias + kNb * 4, gb = ub + kNb * 4, gb2 = gb + kNb * 4;
  static constexpr int kStage = 2 * Bp * kPx * 2;
  static constexpr bool kSum1 = MID && BT == 4;   // W_1's update sum is accumulated (tensor memory), W_2's lies here
  static constexpr int u2 = (gb2 + kNb * 4 + 15) / 16 * 16, ring = u2 + (kSum1 ? kH1 / 16 * 32 * 32 : 0), idx = ring + kRing * kStage, bars = idx + 4 * 64 * 4, total = bars + 128;
  // units of W_0 in tensor memory (a group each); then W_1's 8 groups; then W_2's update sum, or W_1's 8 groups
  static constexpr int kRes = kSum1 ? 0 : MID ? 6 : 14;
  static_assert(z0 % 16 == 0 && z1 % 16 == 0 && a1 % 16 == 0 && w2 % 16 == 0 && logit % 16 == 0 && z2 % 16 == 0 && bias % 16 == 0 && idx % 16 == 0 && bars % 8 == 0, "alignment");
  static_assert(total <= 227 * 1024, "fits an SM");
};

struct WideLaunch {
  RoundLaunch r;
  float* work;
  int D0, C, CL;
};

template <int BT, bool MID>
__global__ void __launch_bounds__(kThreads, 1) mlp_wide_kernel(const __grid_constant__ WideLaunch p) {
  typedef Lay<BT, MID> M;
  constexpr int Bp = M::Bp, K2 = M::K2, kPw2 = M::kPw2, KS = BT / 2, kRes = M::kRes, kU2 = kRes + (MID ? 8 : 0);
  extern __shared__ __align__(128) unsigned char smem[];
  const int CL = p.CL, C = p.C, D0 = p.D0;
  const TaskDesc t = p.r.tasks[p.r.task_begin + blockIdx.x / CL];
  if (!debug_task_ok(p.r, t)) return;   // the whole cluster alike
  const size_t ob0 = (size_t)D0 * kH0, oW1 = ob0 + kH0, ob1 = oW1 + (size_t)kH0 * kH1, oW2 = MID ? ob1 + kH1 : oW1, ob2 = oW2 + (size_t)K2 * C;
  const int rank = CL > 1 ? (int)mma::cluster_rank() : 0;
  if (t.steps == 0) {
    if (rank == 0) publish_empty_round(p.r, t, (uint32_t)(ob2 + C));
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tt = lane & 3;
  const float eta = t.eta, lambda = p.r.l2;
  bf16* const W1 = reinterpret_cast<bf16*>(smem + M::w1);      // [n][k]
  bf16* const A0 = reinterpret_cast<bf16*>(smem + M::a0);      // [sample][unit]
  bf16* const Z0 = reinterpret_cast<bf16*>(smem + M::z0);
  bf16* const Z1 = reinterpret_cast<bf16*>(smem + M::z1);
  bf16* const A1 = reinterpret_cast<bf16*>(smem + M::a1);
  bf16* const Z2 = reinterpret_cast<bf16*>(smem + M::z2);
  bf16* const AL = MID ? A1 : A0;                              // what the class layer reads
  float* const W2 = reinterpret_cast<float*>(smem + M::w2);    // fp32 master, [class][k]
  float* const inbox = reinterpret_cast<float*>(smem + M::z0);
  float* const part = reinterpret_cast<float*>(smem + M::part);
  float* const logit = reinterpret_cast<float*>(smem + M::logit);
  float* const bias = reinterpret_cast<float*>(smem + M::bias);
  float* const ubias = reinterpret_cast<float*>(smem + M::ub);
  float* const gbias = reinterpret_cast<float*>(smem + M::gb);
  float* const gbias2 = reinterpret_cast<float*>(smem + M::gb2);
  bf16* const ring = reinterpret_cast<bf16*>(smem + M::ring);
  int* const idx = reinterpret_cast<int*>(smem + M::idx);      // [2][64] row numbers, [2][64] labels
  uint64_t* const full = reinterpret_cast<uint64_t*>(smem + M::bars);
  uint64_t* const freed = full + kRing;
  uint64_t* const b_in = freed + kRing;     // parts of Z_0 of the own hidden units
  uint64_t* const b_a0 = b_in + 1;          // A_0 of the others
  uint64_t* const b_free = b_in + 2;        // the peers' inboxes may be written
  uint32_t* const tmem_at = reinterpret_cast<uint32_t*>(b_in + 3);

  const int nch = D0 / (kChunk * CL), nu = 2 * nch, u0 = rank * nu;   // this CTA's chunks and units of 16 inputs
  const int tpc = kWarps / CL, owner = warp / tpc;                    // hidden tiles per CTA; who owns this warp's

  for (int i = tid; i < M::total / 4; i += kThreads) reinterpret_cast<uint32_t*>(smem)[i] = 0;
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tmem_at)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const uint32_t in_bytes = (uint32_t)((CL - 1) * tpc * BT * 512), a0_bytes = (uint32_t)((kWarps - tpc) * Bp * 32);
  if (tid == 0) {
    for (int s = 0; s < kRing; ++s) { mbar_init(&full[s], kThreads); mbar_init(&freed[s], kWarps); }
    mbar_init(b_in, 1);
    mbar_init(b_a0, 1);
    mbar_init(b_free, CL > 1 ? (CL - 1) * kWarps : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (CL > 1) mma::cluster_sync(); else __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (tid == 0 && CL > 1) {
    mbar_expect_tx(b_in, in_bytes);
    mbar_expect_tx(b_a0, a0_bytes);
  }
  Own own;
  own.tmem = *tmem_at + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * 128u;

  // A thread whose wait has given up waits no more and runs through on whatever is there, but neither arms a barrier (a second arrival
  // on one that is short of bytes would be invalid) nor sends: whoever depends on it gives up in turn, the status word is set, and
  // every CTA of the cluster reaches the end.
  bool ok = true;
  auto wait = [&](uint64_t* bar, uint32_t parity) { if (ok) ok = mbar_wait(bar, parity); };
  auto wait_cluster = [&](uint64_t* bar, uint32_t parity) {
    const uint32_t at = smem_addr(bar);
    for (uint32_t i = 0; ok; ++i) {
      if (mma::try_wait_cluster(at, parity)) break;
      if (i >= kWaitLimit) ok = false;
    }
  };

  const ClientData cd = p.r.clients[t.client];
  const uint64_t key = p.r.sample_keys[t.client];
  const bf16* xrows = reinterpret_cast<const bf16*>(cd.x) + 16 * u0;
  auto draw_rows = [&](uint32_t it) {
    if (tid < Bp) {
      const uint32_t id = sample_index(draw(key, t.sample_ctr0 + (uint64_t)it * Bp + tid), cd.n);
      idx[(it & 1) * 64 + tid] = (int)id;
      // (covered by this thread's next arrival on a chunk's barrier)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(idx + 128 + (it & 1) * 64 + tid)), "l"(cd.y + id) : "memory");
    }
  };
  // Copies of chunk c: threads [0, 4 Bp) the columns of iteration itc's rows, the next 4 Bp those of iteration itc + 1.
  uint32_t qi = 0, qc = 0;   // chunks issued and consumed so far
  auto issue = [&](int c, int itc, bool cur, bool next) {
    const int s = qi % kRing;
    if (qi >= (uint32_t)kRing) wait(&freed[s], (qi / kRing - 1) & 1);
    ++qi;
    const int half = tid / (4 * Bp), r = (tid % (4 * Bp)) >> 2, piece = tid & 3;
    if (half == 0 ? cur : (half == 1 && next)) {
      const bf16* src = xrows + (size_t)idx[((itc + half) & 1) * 64 + r] * D0 + kChunk * c + 8 * piece;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(ring + ((s * 2 + half) * Bp + r) * kPx + 8 * piece)), "l"(src) : "memory");
    }
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(&full[s])) : "memory");
  };

  // ---- start model: snapshot minus own update sums still in flight ----
  const float* snap = p.r.snaps + (size_t)t.snap_slot * p.r.stride;
  auto start_value = [&](size_t at) {
    float v = snap[at];
#pragma unroll 1
    for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
      const InflightRef ref = p.r.inflight[t.inflight_off + f];
      v = fmaf(-ref.eta, p.r.U[(size_t)ref.row * p.r.stride + at], v);
    }
    return v;
  };
  // words 0 .. 7 of a thread's group: rows g (+ 8 with bit 1), columns 2 tt + bit 0 (+ 8 with bit 2), `pitch` apart
  auto start_words = [&](size_t at, int pitch, float (&v)[8]) {
    auto word = [&](const float* row, int i) { return row[at + (size_t)((i & 1) + ((i & 4) ? 8 : 0)) * pitch + ((i & 2) ? 8 : 0)]; };
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = word(snap, i);
#pragma unroll 1
    for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
      const InflightRef ref = p.r.inflight[t.inflight_off + f];
      const float* us = p.r.U + (size_t)ref.row * p.r.stride;
      float x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = word(us, i);
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = fmaf(-ref.eta, x[i], v[i]);
    }
  };
  const int i1 = warp & 7, h1 = warp >> 3;   // this warp's tiles of W_1: outputs 16 i1 .., inputs 128 h1 ..
  auto w1_at = [&](int q) { return oW1 + (size_t)(128 * h1 + 16 * q + 2 * tt) * kH1 + 16 * i1 + g; };
  auto put_w1 = [&](int q, const float (&w)[8]) {   // the bf16 operand of group q
    bf16* d = W1 + (16 * i1 + g) * kP0 + 128 * h1 + 16 * q + 2 * tt;
    *reinterpret_cast<uint32_t*>(d) = pack_bf16(w[0], w[1]);
    *reinterpret_cast<uint32_t*>(d + 8 * kP0) = pack_bf16(w[2], w[3]);
    *reinterpret_cast<uint32_t*>(d + 8) = pack_bf16(w[4], w[5]);
    *reinterpret_cast<uint32_t*>(d + 8 * kP0 + 8) = pack_bf16(w[6], w[7]);
  };
  constexpr bool kSum1 = M::kSum1;
  float* const us2 = reinterpret_cast<float*>(smem + M::u2) + tid * 8;   // kSum1: W_2's update sum, a thread's own words
  auto load_u2 = [&](float (&v)[8]) {
    if constexpr (!kSum1) {
      own.load(kU2, v);
    } else {
#pragma unroll
      for (int i = 0; i < 8; i += 4) {
        const float4 x = *reinterpret_cast<const float4*>(us2 + i);
        v[i] = x.x; v[i + 1] = x.y; v[i + 2] = x.z; v[i + 3] = x.w;
      }
    }
  };
  auto store_u2 = [&](const float (&v)[8]) {
    if constexpr (!kSum1) {
      own.store(kU2, v);
      own.store_wait();
    } else {
#pragma unroll
      for (int i = 0; i < 8; i += 4) *reinterpret_cast<float4*>(us2 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
  };
  {
    const float zero[8] = {};
    if (kSum1) {
#pragma unroll
      for (int q = 0; q < 8; ++q) own.store(kU2 + q, zero);
    } else {
      own.store(kU2, zero);
    }
    own.store_wait();
  }
  draw_rows(0);
  if (MID) {
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
      float w[8];
      start_words(w1_at(q), kH1, w);
      own.store(kRes + q, w);
      put_w1(q, w);
    }
    own.store_wait();
  }
#pragma unroll 1
  for (int e = tid; e < K2 * C; e += kThreads) W2[(e % C) * kPw2 + e / C] = start_value(oW2 + e);
#pragma unroll 1
  for (int e = tid; e < kH0; e += kThreads) bias[e] = start_value(ob0 + e);
#pragma unroll 1
  for (int e = tid; MID && e < kH1; e += kThreads) bias[kB1 + e] = start_value(ob1 + e);
  if (tid < C) bias[kB2 + tid] = start_value(ob2 + tid);
  __syncthreads();

  float* const master = p.work + (size_t)t.client * p.r.stride + ((size_t)u0 * kWarps + warp) * 256 + lane * 4;   // + u * 4096
  const size_t nat = (size_t)(16 * u0 + 2 * tt) * kH0 + 16 * warp + g;                                            // + u * 4096, natural order
  float* const Urow = p.r.U + (size_t)t.u_row * p.r.stride;
  float* const wrow = p.r.w_end ? p.r.w_end + (size_t)t.u_row * p.r.stride : nullptr;
  const float inv_eta = 1.f / eta;
  auto publish_words = [&](size_t at, int pitch, const float (&s)[8], const float (&w)[8]) {   // update sums, weights
    // a round whose copies or hand-overs gave up leaves NaN behind as well as the status bit
    const float bad = ok ? 0.f : __int_as_float(0x7FFFFFFF);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const size_t a = at + (size_t)((i & 1) + ((i & 4) ? 8 : 0)) * pitch + ((i & 2) ? 8 : 0);
      Urow[a] = s[i] + bad;
      if (wrow) wrow[a] = w[i] + bad;
    }
  };

  constexpr int kSlots = M::kSlots;
  float* const slot = reinterpret_cast<float*>(smem + M::z0) + warp * 256 + lane * 4;   // + 4096 per slot
  // One pass over the CTA's inputs.  GRAD: the gradient of iteration itc and the update (otherwise the start model comes
  // in); LOOK: the forward product of iteration itc + 1 and its hand-over (otherwise the update sums go out).
  auto pass = [&](auto grad_, auto look_, int itc) {
    constexpr bool GRAD = decltype(grad_)::value, LOOK = decltype(look_)::value;
    float acc[LOOK ? BT : 1][4] = {};
    uint32_t a[GRAD ? KS : 1][4];
    if (GRAD) {   // dZ_0^T of this warp's hidden units, all samples
#pragma unroll
      for (int k = 0; k < (GRAD ? KS : 0); ++k)
        ldmatrix4t(a[k], smem_addr(Z0 + (16 * k + (lane >> 4) * 8 + (lane & 7)) * kP0 + 16 * warp + ((lane >> 3) & 1) * 8));
    }
    // Units of the master on their way into shared memory, kSlots ahead: each lane copies and reads its own 32 bytes of a
    // unit, a group of copies per unit.
    // Every pass walks the inputs the other way round than the pass before it: what that one touched last is still in L2.
    const bool back = GRAD && !(itc & 1);
    const int lo = back ? 0 : kRes, hi = back ? nu - kRes : nu;   // places in that order whose units stream
    auto unit = [&](int i) { return back ? nu - 1 - i : i; };
    auto stage = [&](int i) {
      const float* s = master + (size_t)unit(i) * (kWarps * 256);
      const uint32_t d = smem_addr(slot + (i % kSlots) * 4096);
      if (i < hi) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(s) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 512), "l"(s + 128) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (GRAD) {   // (what the slots lie in)
      __syncthreads();   // every warp has its fragments of dZ_0 and is done with dZ_1 and A_1
#pragma unroll
      for (int i = 0; i < kSlots; ++i) stage(lo + i);
    }
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
      float sv[GRAD && LOOK ? 1 : 2][8];
      if (!(GRAD && LOOK)) {
#pragma unroll
        for (int j = 0; j < 2; ++j) start_words(nat + (size_t)unit(2 * c + j) * (16 * kH0), kH0, sv[GRAD && LOOK ? 0 : j]);
      }
      wait(&full[qc % kRing], (qc / kRing) & 1);
      const bf16* xc = ring + (qc % kRing) * 2 * Bp * kPx;
      const bf16* xn = xc + Bp * kPx;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i2 = 2 * c + j, u = unit(i2), col = 16 * (u & 1);
        float w[8];
        if (!GRAD) {
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = sv[GRAD && LOOK ? 0 : j][i];
        } else if (u < kRes) {
          own.load(u, w);
        } else {
          asm volatile("cp.async.wait_group %0;" ::"n"(kSlots - 1) : "memory");
          const float4* s = reinterpret_cast<const float4*>(slot + (i2 % kSlots) * 4096);
          const float4 v0 = s[0], v1 = s[32];
          w[0] = v0.x; w[1] = v0.y; w[2] = v0.z; w[3] = v0.w;
          w[4] = v1.x; w[5] = v1.y; w[6] = v1.z; w[7] = v1.w;
          stage(i2 + kSlots);
        }
        if (GRAD) {
          float gr[2][4] = {};
#pragma unroll
          for (int k = 0; k < KS; ++k) {
            uint32_t f[4];   // the columns of this unit as second operand, 16 samples
            ldmatrix4t(f, smem_addr(xc + (16 * k + (lane & 15)) * kPx + col + (lane >> 4) * 8));
            mma_bf16(gr[0], a[GRAD ? k : 0], f[0], f[1]);
            mma_bf16(gr[1], a[GRAD ? k : 0], f[2], f[3]);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = fmaf(-eta, fmaf(lambda, w[i], gr[i >> 2][i & 3]), w[i]);
        }
        if (LOOK) {
          if (u < kRes) {
            own.store(u, w);
          } else {
            float4* d = reinterpret_cast<float4*>(master + (size_t)u * (kWarps * 256));
            __stcg(d, make_float4(w[0], w[1], w[2], w[3]));
            __stcg(d + 32, make_float4(w[4], w[5], w[6], w[7]));
          }
          const uint32_t f[4] = {pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]), pack_bf16(w[4], w[5]), pack_bf16(w[6], w[7])};
#pragma unroll
          for (int b = 0; b < BT; b += 2) {
            uint32_t x[4];   // two groups of eight samples
            ldmatrix4(x, smem_addr(xn + (8 * b + (lane >> 4) * 8 + (lane & 7)) * kPx + col + ((lane >> 3) & 1) * 8));
            mma_bf16(acc[LOOK ? b : 0], f, x[0], x[1]);
            mma_bf16(acc[LOOK ? b + 1 : 0], f, x[2], x[3]);
          }
        } else {
          float (&s)[8] = sv[GRAD && LOOK ? 0 : j];
#pragma unroll
          for (int i = 0; i < 8; ++i) s[i] = (s[i] - w[i]) * inv_eta;
          publish_words(nat + (size_t)u * (16 * kH0), kH0, s, w);
        }
      }
      ++qc;
      __syncwarp();
      if (lane == 0) mbar_arrive(&freed[(qc - 1) % kRing]);
      // at the end of a chunk the slot of the one before is free without a wait: every warp is about as far
      if (c + 2 < nch) issue(back ? nch - 3 - c : c + 2, itc, GRAD, LOOK);
    }
    if (!LOOK) return;
    own.store_wait();
    if (CL > 1) {   // this warp needs nothing any more of what the peers' parts will overwrite
      __syncwarp();
      if (lane < CL && lane != rank) mma::arrive_peer(mma::peer_addr(smem_addr(b_free), lane));
    }
    const uint32_t par = (uint32_t)(itc + 1) & 1;
    if (owner != rank) {
      wait_cluster(b_free, par);
      const int s = rank < owner ? rank : rank - 1;
      const uint32_t at = mma::peer_addr(smem_addr(inbox + (s * tpc + warp % tpc) * BT * 128 + 4 * lane), owner), bar = mma::peer_addr(smem_addr(b_in), owner);
#pragma unroll
      for (int b = 0; b < (LOOK ? BT : 0); ++b)
        if (ok) mma::send_peer(at + 512u * b, make_float4(acc[b][0], acc[b][1], acc[b][2], acc[b][3]), bar);
      return;
    }
    if (CL > 1) {
      wait_cluster(b_in, par);
      if (ok && lane == 0 && warp % tpc == 0) mbar_expect_tx(b_in, in_bytes);
    }
#pragma unroll 1
    for (int s = 0; s < CL - 1; ++s) {
      const float4* in = reinterpret_cast<const float4*>(inbox + (s * tpc + warp % tpc) * BT * 128 + 4 * lane);
#pragma unroll
      for (int b = 0; b < (LOOK ? BT : 0); ++b) {
        const float4 v = in[32 * b];
        acc[b][0] += v.x; acc[b][1] += v.y; acc[b][2] += v.z; acc[b][3] += v.w;
      }
    }
    const float bias0 = bias[16 * warp + g], bias8 = bias[16 * warp + g + 8];
#pragma unroll
    for (int b = 0; b < (LOOK ? BT : 0); ++b)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        A0[(8 * b + 2 * tt + (i & 1)) * kP0 + 16 * warp + g + ((i & 2) ? 8 : 0)] = __float2bfloat16_rn(fmaxf(acc[b][i] + ((i & 2) ? bias8 : bias0), 0.f));
    __syncwarp();
#pragma unroll 1
    for (int q = lane; q < 2 * Bp && CL > 1; q += 32) {
      const bf16* s = A0 + (q >> 1) * kP0 + 16 * warp + 8 * (q & 1);
      const float4 v = *reinterpret_cast<const float4*>(s);
      for (int r = 0; r < CL; ++r)
        if (ok && r != rank) mma::send_peer(mma::peer_addr(smem_addr(s), r), v, mma::peer_addr(smem_addr(b_a0), r));
    }
  };
  typedef std::true_type Yes;
  typedef std::false_type No;

  issue(0, -1, false, true);
  issue(1, -1, false, true);
  pass(No(), Yes(), -1);

#pragma unroll 1
  for (uint32_t it = 0; it < t.steps; ++it) {
    const bool more = it + 1 < t.steps;
    if (more) draw_rows(it + 1);
    if (CL > 1) {
      wait_cluster(b_a0, it & 1);
      if (ok && tid == 0 && more) mbar_expect_tx(b_a0, a0_bytes);
    }
    __syncthreads();   // A_0 is complete, the parts of Z_0 have been read
    const bool back = !(it & 1);
    issue(back ? nch - 1 : 0, (int)it, true, more);
    issue(back ? nch - 2 : 1, (int)it, true, more);

    if (MID) {   // A_1 = relu(A_0 W_1 + b_1): a warp has 16 outputs and half of the samples
      float acc[BT / 2][4] = {};
      const int i = warp & 7, s0 = (warp >> 3) * (Bp / 2);
#pragma unroll 4
      for (int k = 0; k < kH0; k += 16) {
        uint32_t f[4];
        ldmatrix4(f, smem_addr(W1 + (16 * i + ((lane >> 3) & 1) * 8 + (lane & 7)) * kP0 + k + (lane >> 4) * 8));
#pragma unroll
        for (int b = 0; b < BT / 2; b += 2) {
          uint32_t x[4];
          ldmatrix4(x, smem_addr(A0 + (s0 + 8 * b + (lane >> 4) * 8 + (lane & 7)) * kP0 + k + ((lane >> 3) & 1) * 8));
          mma_bf16(acc[b], f, x[0], x[1]);
          mma_bf16(acc[b + 1], f, x[2], x[3]);
        }
      }
      const float c0 = bias[kB1 + 16 * i + g], c8 = bias[kB1 + 16 * i + g + 8];
#pragma unroll
      for (int b = 0; b < BT / 2; ++b)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          A1[(s0 + 8 * b + 2 * tt + (q & 1)) * kP1 + 16 * i + g + ((q & 2) ? 8 : 0)] = __float2bfloat16_rn(fmaxf(acc[b][q] + ((q & 2) ? c8 : c0), 0.f));
      __syncthreads();
    }
    {   // logits: eight samples and a part of the inputs per warp
      constexpr int kParts = kWarps / BT, kLen = K2 / kParts;
      const int b = warp % BT, k0 = (warp / BT) * kLen;
      float acc[4] = {};
#pragma unroll
      for (int k = 0; k < kLen; k += 16) {
        uint32_t f[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float* w = W2 + g * kPw2 + k0 + k + 8 * h + 2 * tt;
          const float2 v0 = *reinterpret_cast<const float2*>(w), v8 = *reinterpret_cast<const float2*>(w + 8 * kPw2);
          f[2 * h] = pack_bf16(v0.x, v0.y); f[2 * h + 1] = pack_bf16(v8.x, v8.y);
        }
        constexpr int kPl = MID ? kP1 : kP0;
        const bf16* x = AL + (8 * b + g) * kPl + k0 + k + 2 * tt;
        mma_bf16(acc, f, *reinterpret_cast<const uint32_t*>(x), *reinterpret_cast<const uint32_t*>(x + 8));
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) part[warp * 128 + q * 32 + lane] = acc[q];
      __syncthreads();
#pragma unroll 1
      for (int e = tid; e < BT * 128; e += kThreads) {
        const int bb = e >> 7, q = (e >> 5) & 3, n = g + ((q & 2) ? 8 : 0);
        float v = bias[kB2 + n];
#pragma unroll
        for (int r = 0; r < kParts; ++r) v += part[r * BT * 128 + e];
        logit[(8 * bb + 2 * tt + (q & 1)) * 17 + n] = v;
      }
      __syncthreads();
    }
    if (tid < 4 * Bp) {   // dZ_2 = (p - onehot) / B; four lanes per sample
      const int s = tid >> 2, q = tid & 3;
      float* z = logit + s * 17;
      float v[4], mx = -3e38f, sum = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        v[i] = q + 4 * i < C ? z[q + 4 * i] : -3e38f;
        mx = fmaxf(mx, v[i]);
      }
      mx = fmaxf(mx, lr::shx(mx, 1));
      mx = fmaxf(mx, lr::shx(mx, 2));
#pragma unroll
      for (int i = 0; i < 4; ++i) { v[i] = lr::ex2((v[i] - mx) * lr::kLog2e); sum += v[i]; }
      sum += lr::shx(sum, 1);
      sum += lr::shx(sum, 2);
      const float inv = lr::rcp(sum);
      const int y = idx[128 + (it & 1) * 64 + s];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = q + 4 * i;
        const float d = c < C ? (v[i] * inv - (c == y ? 1.f : 0.f)) * (1.f / (float)Bp) : 0.f;
        Z2[s * kPz + c] = __float2bfloat16_rn(d);
        z[c] = d;   // unrounded, for the bias gradient
      }
    }
    __syncthreads();
    {   // dZ of the layer below = relu' (W_2 dZ_2): a warp has 16 inputs of the class layer
      constexpr int kPl = MID ? kP1 : kP0, kN = MID ? BT / 2 : BT;
      const int i = MID ? warp & 7 : warp, s0 = MID ? (warp >> 3) * (Bp / 2) : 0;
      bf16* const Z = MID ? Z1 : Z0;
      uint32_t f[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float* w = W2 + (8 * h + 2 * tt) * kPw2 + 16 * i + g;
        f[2 * h] = pack_bf16(w[0], w[kPw2]); f[2 * h + 1] = pack_bf16(w[8], w[kPw2 + 8]);
      }
      float g0 = 0.f, g8 = 0.f;
#pragma unroll
      for (int b = 0; b < kN; ++b) {
        float acc[4] = {};
        const bf16* x = Z2 + (s0 + 8 * b + g) * kPz + 2 * tt;
        mma_bf16(acc, f, *reinterpret_cast<const uint32_t*>(x), *reinterpret_cast<const uint32_t*>(x + 8));
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int s = s0 + 8 * b + 2 * tt + (q & 1), n = 16 * i + g + ((q & 2) ? 8 : 0);
          const float v = __bfloat162float(AL[s * kPl + n]) > 0.f ? acc[q] : 0.f;
          Z[s * kPl + n] = __float2bfloat16_rn(v);
          if (q & 2) g8 += v; else g0 += v;
        }
      }
      g0 += lr::shx(g0, 1); g8 += lr::shx(g8, 1);
      g0 += lr::shx(g0, 2); g8 += lr::shx(g8, 2);
      if (tt == 0) {
        float* d = (MID && s0 ? gbias2 : gbias) + (MID ? kB1 : 0) + 16 * i + g;
        d[0] = g0; d[8] = g8;
      }
    }
    if (tid >= kThreads - kMaxC) {   // the class layer's bias gradient
      const int c = tid - (kThreads - kMaxC);
      float v = 0.f;
#pragma unroll 8
      for (int s = 0; s < Bp; ++s) v += logit[s * 17 + c];
      gbias[kB2 + c] = v;
    }
    __syncthreads();
    if (warp < K2 / 16) {   // dW_2: 16 inputs per warp
      constexpr int kPl = MID ? kP1 : kP0;
      float acc[2][4] = {};
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t f[4], x[4];
        ldmatrix4t(f, smem_addr(Z2 + (16 * k + (lane >> 4) * 8 + (lane & 7)) * kPz + ((lane >> 3) & 1) * 8));
        ldmatrix4t(x, smem_addr(AL + (16 * k + (lane & 15)) * kPl + 16 * warp + (lane >> 4) * 8));
        mma_bf16(acc[0], f, x[0], x[1]);
        mma_bf16(acc[1], f, x[2], x[3]);
      }
      float us[8];
      load_u2(us);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float2* w = reinterpret_cast<float2*>(W2 + (g + 8 * q) * kPw2 + 16 * warp + 8 * h + 2 * tt);
          float2 v = *w;
          const float g0 = fmaf(lambda, v.x, acc[h][2 * q]), g1 = fmaf(lambda, v.y, acc[h][2 * q + 1]);
          v.x = fmaf(-eta, g0, v.x);
          v.y = fmaf(-eta, g1, v.y);
          *w = v;
          us[4 * h + 2 * q] += g0; us[4 * h + 2 * q + 1] += g1;
        }
      store_u2(us);
    }
    if (MID) {
      {   // dZ_0 = relu' (W_1 dZ_1): a warp has 16 hidden units of layer 0, all samples
        float acc[BT][4] = {};
#pragma unroll 2
        for (int k = 0; k < kH1; k += 16) {
          uint32_t f[4];
          ldmatrix4t(f, smem_addr(W1 + (k + (lane >> 4) * 8 + (lane & 7)) * kP0 + 16 * warp + ((lane >> 3) & 1) * 8));
#pragma unroll
          for (int b = 0; b < BT; b += 2) {
            uint32_t x[4];
            ldmatrix4(x, smem_addr(Z1 + (8 * b + (lane >> 4) * 8 + (lane & 7)) * kP1 + k + ((lane >> 3) & 1) * 8));
            mma_bf16(acc[b], f, x[0], x[1]);
            mma_bf16(acc[b + 1], f, x[2], x[3]);
          }
        }
        float g0 = 0.f, g8 = 0.f;
#pragma unroll
        for (int b = 0; b < BT; ++b)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int at = (8 * b + 2 * tt + (q & 1)) * kP0 + 16 * warp + g + ((q & 2) ? 8 : 0);
            const float v = __bfloat162float(A0[at]) > 0.f ? acc[b][q] : 0.f;
            Z0[at] = __float2bfloat16_rn(v);
            if (q & 2) g8 += v; else g0 += v;
          }
        g0 += lr::shx(g0, 1); g8 += lr::shx(g8, 1);
        g0 += lr::shx(g0, 2); g8 += lr::shx(g8, 2);
        if (tt == 0) { gbias[16 * warp + g] = g0; gbias[16 * warp + g + 8] = g8; }
      }
      __syncthreads();   // nobody reads the old W_1 any more
      uint32_t f[KS][4];
#pragma unroll
      for (int k = 0; k < KS; ++k)
        ldmatrix4t(f[k], smem_addr(Z1 + (16 * k + (lane >> 4) * 8 + (lane & 7)) * kP1 + 16 * i1 + ((lane >> 3) & 1) * 8));
#pragma unroll 1
      for (int q = 0; q < 8; ++q) {   // dW_1 and update: 16 inputs at a time
        float acc[2][4] = {}, w[8];
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          uint32_t x[4];
          ldmatrix4t(x, smem_addr(A0 + (16 * k + (lane & 15)) * kP0 + 128 * h1 + 16 * q + (lane >> 4) * 8));
          mma_bf16(acc[0], f[k], x[0], x[1]);
          mma_bf16(acc[1], f[k], x[2], x[3]);
        }
        own.load(kRes + q, w);
        if (kSum1) {
          float us[8];
          own.load(kU2 + q, us);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float gr = fmaf(lambda, w[i], acc[i >> 2][i & 3]);
            w[i] = fmaf(-eta, gr, w[i]);
            us[i] += gr;
          }
          own.store(kU2 + q, us);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = fmaf(-eta, fmaf(lambda, w[i], acc[i >> 2][i & 3]), w[i]);
        }
        own.store(kRes + q, w);
        put_w1(q, w);
      }
      own.store_wait();
    } else {
      __syncthreads();
    }
    if (tid < kNb) {
      const float gr = gbias[tid] + gbias2[tid];
      bias[tid] = fmaf(-eta, gr, bias[tid]);
      ubias[tid] += gr;
    }
    if (more) pass(Yes(), Yes(), (int)it);
    else pass(Yes(), No(), (int)it);
  }

  // ---- event trigger: h reached s_{i,c}; the last pass has published W_0's update sum, here go the others ----
  __syncthreads();
  if (MID) {
#pragma unroll 1
    for (int q = rank; q < 8; q += CL) {
      float s[8], w[8];
      own.load(kRes + q, w);
      if (kSum1) {
        own.load(kU2 + q, s);
      } else {
        start_words(w1_at(q), kH1, s);
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i] = (s[i] - w[i]) * inv_eta;
      }
      publish_words(w1_at(q), kH1, s, w);
    }
  }
  if (rank == 0) {
    const float bad = ok ? 0.f : __int_as_float(0x7FFFFFFF);
    if (warp < K2 / 16) {
      float us[8];
      load_u2(us);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = 16 * warp + 2 * tt + (i & 1) + ((i & 4) ? 8 : 0), c = g + ((i & 2) ? 8 : 0);
        if (c < C) {
          Urow[oW2 + (size_t)k * C + c] = us[i] + bad;
          if (wrow) wrow[oW2 + (size_t)k * C + c] = W2[c * kPw2 + k] + bad;
        }
      }
    }
    if (tid < kNb && (MID || tid < kB1 || tid >= kB2) && tid < kB2 + C) {
      const size_t at = tid < kB1 ? ob0 + tid : (tid < kB2 ? ob1 + tid - kB1 : ob2 + tid - kB2);
      Urow[at] = ubias[tid] + bad;
      if (wrow) wrow[at] = bias[tid] + bad;
    }
  }
  if (!ok && p.r.status && lane == 0) atomicOr(p.r.status, 1u);
  if (tid == 0 && rank == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = t.steps * (uint32_t)Bp; rec.flags = 1;
    p.r.trig[t.seq] = rec;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (CL > 1) mma::cluster_sync(); else __syncthreads();   // no CTA leaves while a peer may still send to it
  if (!ok) lr::linger();
  __syncwarp();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_at) : "memory");
}

template <int BT, bool MID>
cudaError_t launch(const WideLaunch& p, cudaStream_t s) {
  constexpr size_t smem = Lay<BT, MID>::total;
  cudaError_t e = cudaFuncSetAttribute(mlp_wide_kernel<BT, MID>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.r.n_tasks * p.CL, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.CL;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.CL > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, mlp_wide_kernel<BT, MID>, p);
}

// A CTA needs four chunks of 32 inputs: fewer than the ring's three, and a warp could run a whole pass ahead of another.
bool splits(uint32_t d0, uint32_t cl) { return d0 % (kChunk * cl) == 0 && d0 / (kChunk * cl) >= 4; }

}  // namespace

bool mlp_wide_eligible(const MlpShape& s) {
  const bool mid = s.n_layers == 3 && s.dims[2] == (uint32_t)kH1;
  return s.precision == 1 && s.dims[1] == (uint32_t)kH0 && (mid || s.n_layers == 2) && s.dims[s.n_layers] <= (uint32_t)kMaxC &&
         (s.batch == 32 || s.batch == 64) && splits(s.dims[0], 1) && mlp_derives_w0(s);
}

cudaError_t launch_mlp_wide_rounds(const MlpLaunch& p, cudaStream_t s) {
  WideLaunch q;
  q.r = p.r;
  q.work = p.work;
  q.D0 = (int)p.shape.dims[0];
  q.C = (int)p.shape.dims[p.shape.n_layers];
  // As many CTAs per round-task as the device runs at once (20 iterations of 3072-256-128-10: 16 clients 1.03 ms on four CTAs
  // each, 1.33 in two waves of eight; 35 clients 1.83 on two, 2.11 in two waves of four)
  for (q.CL = 8; q.CL > 1; q.CL >>= 1) {
    uint32_t fit = 0;
    if (const cudaError_t e = clusters_at_once((uint32_t)q.CL, &fit)) return e;
    if (splits(p.shape.dims[0], q.CL) && p.r.n_tasks <= fit) break;
  }
  if (p.shape.n_layers == 3) return p.shape.batch == 64 ? launch<8, true>(q, s) : launch<4, true>(q, s);
  return p.shape.batch == 64 ? launch<8, false>(q, s) : launch<4, false>(q, s);
}

}  // namespace aet
