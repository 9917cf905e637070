// Local-SGD round of one client for softmax regression 784 -> 10, batch 1, for launches of few round-tasks: a round is a chain of
// dependent steps, and one CTA of a cluster has nothing to do but to walk it.
//
// Algorithm 3, MainComputeNode, inner loop (g = grad f(w_c, xi) + lambda W; w_c -= eta g; U_i += g; h++).  With
// q = 1 - eta lambda, W_k, b_k the model at the start of block k of sixteen samples and delta_s = softmax(z_s) - onehot(y_s),
// step t of block k + 1 sees
//     z_t = q^(t+16) W_k x_t + b_k + sum_{s in block k} C[t][s] delta_s + sum_{s<t} L[t][s] delta_s,
//     L[t][s] = -eta (q^(t-1-s) x_s.x_t + 1),   C[t][s] = -eta (q^(t+15-s) x_s.x_t + 1):
// everything but the two small sums is known a block ahead.  A cluster per round-task:
//   model CTAs   (3 or 4, each a range of the inputs)  as soon as delta_k is there: U^T += delta^T X of block k, then the logits of
//                block k + 2 with the model that gives;
//   Gram CTAs    (2 or 3, each a range of the inputs)  products of a block's rows with one another and with those of the block before;
//   the walker   warp R walks the samples one by one, substituting: an exponential per class, their sum, delta, and with it the
//                corrections of the next sixteen samples and more, one coupling per sample; warps beside it add up couplings and
//                logits as they come in, and send each block's deltas, split for the tensor cores, to the model CTAs.
// Between CTAs everything goes by st.async, counted by mbarriers; the cluster never meets between start and trigger.
//
// The step, 116 cycles: exponential 17, through shared memory to all lanes 29 (a sum over ten lanes by shuffles takes 60 and more, by
// the integer reduction 44), sum 16, reciprocal 23, two FMAs 8; the rest is what the walker's other accesses to shared memory hold up.
// So R has a CTA to itself: beside product warps it took 140 to 150.  Its loop is as short as it can be: one value waits per step, the
// fifteen others are corrected while the next exponentials go round.  Substitution is exact; sweeps over the sixteen samples until they
// no longer move (lr_chain_kernel.cu) took 400 cycles each, 4.4 to 6 of them a block.
//
// fp32 products on the tensor cores: the update and its deltas as three bf16 parts each, logits and Gram matrices as two tf32 (see
// lr_chain_kernel.cu, where the fragments are the same).  With lambda the kernel carries D = sum_s q^(n-1-s) delta_s x_s;
// U = D + W_start (1 - q^n) / eta.
//
// What bounds it: in rounds of hundreds of samples the way from a block's deltas to the logits of the block after next (update, product, sums,
// two hand-overs), 2,340 cycles a block of sixteen, of which R walks 1,970 and waits 370; in short rounds the way from one wave to the
// next (from R's last step to the next wave's first 9 us: end of the round 2, server's kernel 5, start model and first logits 2).  The
// next kernel may come up four blocks before a round's end, so that its rows and Gram matrices are ready when the model is (from then to
// the first step 3.0 -> 1.5 us; 16 clients 1.28 -> 1.20 ms, ring 6.22 -> 6.12).
// Measured against four CTAs that did everything alike: 5 clients for 110 rounds on the ring 8.27 -> 6.17 ms, 16 skewed clients
// 1.39 -> 1.22 ms, 4 clients with l2 92 -> 83 us, one round of 50 samples 13.4 -> 11.3 us.
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include "aet_kernels.h"
#include "aet_rng.h"
#include "lr_common.cuh"
#include "mma_common.cuh"

namespace aet {
namespace {

using namespace lr;
using mma::Parts;
using mma::parts;
using mma::parts_t;
using mma::Split;
using mma::split_r;
using mma::split_t;

constexpr int kB = 16;                       // samples per block
constexpr int kSteps8 = kD / 8;              // 98 k-steps of 8 inputs
constexpr int kZ = kC * kB;                  // logits of a block, [class][sample]
constexpr int kGp = 20;                      // row pitch of a 16 x 16 matrix: fragments and 16-byte rows hit different banks
constexpr int kCoup = 2 * kB * kGp;          // couplings within a block, then those to the block before
constexpr int kOffC = kB * kGp;
constexpr int kQuadZ = kZ / 4;               // the logits as 16-byte pieces
// bytes a Gram CTA sends about a block: the own couplings' pairs that reach below the diagonal, and the others'
constexpr uint32_t kSendG0 = 8 * 64, kSendG = kSendG0 + 8 * 128;
constexpr uint32_t kSendD = 3 * kC * 8 * 4;  // ... and the walker about a block's deltas: three planes of [class][pair of samples]
constexpr int kNg = 11;                      // Gram warps of a CTA
constexpr int kNgEven = kNg / 2;             // the first of them add up the parts of even blocks, the others those of odd ones
constexpr int kGramParts = 3;                // blocks of Gram parts not yet added up (two are too few: see where they are)
constexpr int kNs = 4;                       // blocks of rows
constexpr int kInZ = 4, kInG = 4, kCoups = 3;   // rings: logits, couplings as they come in; couplings summed
constexpr uint32_t kEarly = 4;               // blocks before a round's end at which the next kernel may come up
constexpr int kWarps = 12, kThreads = kWarps * 32;
// Corrections move a logit by at most 31 max |L|; below this they cannot leave the range of the exponential.
constexpr float kTame = 1.9f;

constexpr int pitch_of(int cols) { return cols % 16 == 8 ? cols : cols + 8; }   // 8 or 24 mod 32 floats: the fragment loads of eight rows hit 32 banks

// MC CTAs with the model, NM warps with KM k-steps each; then GC with the Gram matrices, KG k-steps a warp; then the walker.
template <int MC, int NM, int KM, int GC, int KG>
struct Shape {
  static constexpr int kMc = MC, kGc = GC, kCl = MC + GC + 1, kNm = NM, kKm = KM, kKg = KG;
  static constexpr int kColsM = 8 * NM * KM, kColsG = 8 * kNg * KG, kPitchM = pitch_of(kColsM), kPitchG = pitch_of(kColsG);
  static_assert(NM * KM >= (kSteps8 + MC - 1) / MC && kNg * KG >= (kSteps8 + GC - 1) / GC, "every k-step has a warp");
  static_assert(NM >= 2 && NM < kWarps && kNg < kWarps, "a thread per 16-byte piece of the logits; a warp for the copies");
  struct Model {
    float rows[kNs][kB][kPitchM];
    float zpart[2][NM][kZ];         // per warp: products not yet summed over the warps
    uint32_t dpart[2][3][kB][8];    // deltas in three bf16 parts by parity of the block: [class][pair of samples], as first operand
  };
  struct Gram {
    float rows[kNs][kB][kPitchG];
    float part[kGramParts][kNg][kCoup];
  };
  struct Walk {
    float zin[kInZ][MC][kZ], gin[kInG][GC][kCoup];   // per CTA, as they come in
    float coup[kCoups][kCoup];      // summed over the CTAs, a row per sample: what it adds to the sixteen
    float zsum[2][kC * kGp];        // [class][sample], less the sample's largest
    float ebuf[2][kB][kB], zbuf[kB];   // exponentials by parity of the block: [sample][class]; logits (corrections too large)
    uint32_t dstage[3][kC][8];
    float ub[2][kB];                // update sums of the biases
    float amax[kCoups];             // largest coupling
    uint32_t hot[8][kB];            // [block][class] which samples have the label
  };
  struct __align__(128) Smem {
    union { Model m; Gram g; Walk w; };
    float qp[32];                   // powers of q
    double qd[kB + 1];
    uint64_t full[kNs], freed[kNs];                   // rows
    uint64_t delta[2];                                // (model) the deltas of a block
    uint64_t gfree[kInG];                             // (Gram) the walker has taken what lies there
    uint64_t bz[kInZ], bg[kInG], rz[2], rg[4], done[2], bsum[2];   // (walker) parts in; logits, couplings ready; steps, biases done
  };
  static_assert(sizeof(Smem) <= 227 * 1024, "fits an SM");
};

__device__ __forceinline__ float sum_of(float4 a, float4 b, float2 c) { return ((a.x + a.y) + (a.z + a.w)) + (((b.x + b.y) + (b.z + b.w)) + (c.x + c.y)); }
__device__ __forceinline__ void send_pair(uint32_t addr, float a, float b, uint32_t bar) {   // 8 bytes to a peer
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(a), "f"(b), "r"(bar) : "memory");
}
__device__ __forceinline__ void send_quad(uint32_t addr, uint4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar) : "memory");
}

// The walker's accesses to shared memory, in the order they are written in: what the next sample waits for goes first.
__device__ __forceinline__ void store_if(uint32_t at, float v, bool p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t@q st.shared.f32 [%0], %1;\n\t}" ::"r"(at), "f"(v), "r"((int)p) : "memory");
}
__device__ __forceinline__ float4 load4(uint32_t at) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ float2 load2(uint32_t at) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ float load1(uint32_t at) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
  return v;
}

// LOSE: as if copies never came, with waits that end soon (RoundLaunch::lose; never part of a run).
template <class S, bool LOSE>
__global__ void __launch_bounds__(kThreads, 1) lr_relay_kernel(RoundLaunch p) {
  constexpr int CL = S::kCl, MC = S::kMc, NM = S::kNm, KM = S::kKm, NG = kNg, KG = S::kKg, NS = kNs, GC = S::kGc;
  constexpr int PM = S::kPitchM, PG = S::kPitchG;
  constexpr uint32_t kWalker = MC + GC;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  typename S::Smem& sm = *reinterpret_cast<typename S::Smem*>(smem_raw);

  const TaskDesc t = p.by_value ? p.one_task : p.tasks[p.task_begin + blockIdx.x / CL];
  if (!debug_task_ok(p, t)) return;
  const uint32_t rank = mma::cluster_rank();
  if (t.n_samples == 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (rank == 0) publish_empty_round(p, t, kParams);
    return;
  }
  const bool models = rank < MC, walks = rank == kWalker;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t n = t.n_samples, nblk = (n + kB - 1) / kB;
  const float eta = t.eta, neta = -t.eta;
  const bool decay = p.l2 != 0.f;
  // this CTA's k-steps [ks0, ks0 + cnt)
  const int share = models ? MC : GC, part = models ? (int)rank : (int)rank - MC;
  const int ks0 = part * (kSteps8 / share) + min(part, kSteps8 % share);
  const int cnt = kSteps8 / share + (part < kSteps8 % share ? 1 : 0);
  const int pitch = models ? PM : PG;
  float* const rows = models ? &sm.m.rows[0][0][0] : &sm.g.rows[0][0][0];

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) { mbar_init(&sm.full[s], 1); mbar_init(&sm.freed[s], models ? NM : NG); }
    for (int s = 0; s < kInZ; ++s) mbar_init(&sm.bz[s], 1);
    for (int s = 0; s < kInG; ++s) { mbar_init(&sm.bg[s], 1); mbar_init(&sm.gfree[s], 1); }
    for (int s = 0; s < 4; ++s) mbar_init(&sm.rg[s], 1);
    for (int s = 0; s < 2; ++s) { mbar_init(&sm.rz[s], 1); mbar_init(&sm.done[s], 1); mbar_init(&sm.bsum[s], 1); mbar_init(&sm.delta[s], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (models)
      for (uint32_t s = 0; s < min(2u, nblk); ++s) mbar_expect_tx(&sm.delta[s], kSendD);
  }
  if (warp == kWarps - 1) {
    double q = 1.0 - (double)eta * (double)p.l2, v = 1.0;
    for (int i = lane; i; i >>= 1) {
      if (i & 1) v *= q;
      q *= q;
    }
    sm.qp[lane] = (float)v;
    if (lane <= kB) sm.qd[lane] = v;
  }
  if (walks) {
    for (int i = threadIdx.x; i < 2 * kB * kB; i += kThreads) (&sm.w.ebuf[0][0][0])[i] = 0.f;   // (columns without a class stay zero)
  } else {
    if (models)
      for (int i = threadIdx.x; i < 2 * 3 * kB * 8; i += kThreads) (&sm.m.dpart[0][0][0][0])[i] = 0u;   // (rows without a class stay zero)
    for (int i = threadIdx.x; i < NS * kB; i += kThreads)   // columns no copy writes: inputs that add nothing
      for (int c = 8 * cnt; c < (models ? S::kColsM : S::kColsG); ++c) rows[i * pitch + c] = 0.f;
  }
  mma::cluster_sync();   // a peer's barriers exist before anything is sent to it

  // A thread whose wait has given up waits no more and runs through on whatever is there, but makes no other operation on a barrier
  // and sends nothing: a second arrival on a barrier that is short of bytes would be invalid, and so would bytes without end on one
  // that nobody arms.  Whoever depends on it gives up in turn, the model warps among them, which sets the status word and, for
  // callers without one, leaves NaN in the update sum; every CTA of the cluster reaches the end.  (NaN among what such a thread
  // makes, where another one would pass it on as a result.)
  bool ok = true;
  const float kNone = __int_as_float(0x7FFFFFFF);
  const uint32_t limit = LOSE ? p.max_polls : kWaitLimit;
  const bool lost = LOSE && p.lose == rank + 1;
  auto wait = [&](uint64_t* bar, uint32_t parity) { if (ok) ok = mbar_wait_limit(bar, parity, limit); };
  auto wait_peer = [&](uint64_t* bar, uint32_t parity) {   // for what peers sent, or have taken
    const uint32_t at = smem_addr(bar);
    for (uint32_t i = 0; ok && !mma::try_wait_cluster(at, parity); ++i) ok = i < limit;
  };
  const float scale = neta * kLog2e;
  // The kernel behind this one may come up while the last blocks are walked: what it does before its own wait, it does with what the
  // host wrote (and the kernel behind it, in turn: a round's rows, their Gram matrices).
  auto launch_next = []() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); };
  const uint32_t early = nblk > kEarly ? nblk - kEarly : 0;

  if (walks && warp == 0) {
    // ================= R: the recurrence, step by step; lane = (half, class) =================
    // One half of the lanes has the logits of the block's samples, the other what the block adds to the next block's; the
    // halves change places from block to block.
    const int c = lane & 15, half = lane >> 4;
    float z[kB];
#pragma unroll
    for (int s = 0; s < kB; ++s) z[s] = 0.f;
    for (uint32_t k = 0; k < nblk; ++k) {
      const int b = k & 1;
      const uint32_t nv = min((uint32_t)kB, n - k * kB);
      const bool mine = half == b, tells = mine && c < kC;   // (the lanes without a class keep zeros)
      if (k == early) launch_next();
      if (k == 0) wait(&sm.rg[0], 0);
      const bool next = k + 1 < nblk;
      if (next) wait(&sm.rg[(k + 1) & 3], ((k + 1) >> 2) & 1);
      const float* col = mine || !next ? sm.w.coup[k % kCoups] : sm.w.coup[(k + 1) % kCoups] + kOffC;   // row s: what sample s adds to the sixteen
      float f[kB];
      wait(&sm.rz[b], (k >> 1) & 1);
      const uint32_t hot = sm.w.hot[k & 7][c];
      {
        const float4* zr = reinterpret_cast<const float4*>(&sm.w.zsum[b][(c < kC ? c : 0) * kGp]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 v = zr[i];
          z[4 * i] = mine ? z[4 * i] + v.x : 0.f;
          z[4 * i + 1] = mine ? z[4 * i + 1] + v.y : 0.f;
          z[4 * i + 2] = mine ? z[4 * i + 2] + v.z : 0.f;
          z[4 * i + 3] = mine ? z[4 * i + 3] + v.w : 0.f;
        }
      }
      // A step uses up z[0] and moves the others down by one, round the end: after sixteen every sample is in its place again.
      // Only the next sample's logit is formed at once; the others follow while the next exponentials go round the lanes.  (A loop,
      // not sixteen copies of it: those do not fit the instruction cache, 270 cycles a step.)
      float zc = ok ? z[0] : kNone, d = 0.f;   // (one sample's exponentials pass it on to all that follow)
      auto others = [&]() {
        const float end = z[0];
#pragma unroll
        for (int i = 1; i + 1 < kB; ++i) z[i] = fmaf(f[i], d, z[i + 1]);
        z[kB - 1] = fmaf(f[kB - 1], d, end);
        z[0] = zc;
      };
      {   // as if a step that adds nothing had just been made
        const float last = z[kB - 1];
#pragma unroll
        for (int i = kB - 1; i > 0; --i) z[i] = z[i - 1];
        z[0] = last;
#pragma unroll
        for (int i = 0; i < kB; ++i) f[i] = 0.f;
      }
      auto steps = [&](auto wild_) {
        uint32_t eb = smem_addr(&sm.w.ebuf[b][0][0]), row = smem_addr(col);
        auto exponential = [&]() {
          if (decltype(wild_)::value) {
            if (tells) sm.w.zbuf[c] = zc;
            __syncwarp();
            float m = sm.w.zbuf[0];
#pragma unroll
            for (int i = 1; i < kC; ++i) m = fmaxf(m, sm.w.zbuf[i]);
            if (mine) zc -= m;
            __syncwarp();
          }
          return ex2(zc);
        };
        float mye = exponential();
#pragma unroll 1
        for (uint32_t s = 0; s < nv; ++s, eb += 4 * kB, row += 4 * kGp) {
          store_if(eb + 4 * c, mye, tells);
          __syncwarp();
          const float4 e0 = load4(eb), e1 = load4(eb + 16);
          const float2 e2 = load2(eb + 32);
          const float e = load1(eb + 4 * c);
          others();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = load4(row + 16 * i);
            f[4 * i] = v.x; f[4 * i + 1] = v.y; f[4 * i + 2] = v.z; f[4 * i + 3] = v.w;
          }
          const float oh = (hot >> s) & 1u ? 1.f : 0.f;
          const float inv = rcp(sum_of(e0, e1, e2));
          zc = fmaf(f[0] * e, inv, fmaf(-f[0], oh, z[1]));   // the product with e beside the sum
          mye = exponential();
          d = fmaf(e, inv, -oh);
        }
      };
      // (the shift of the softmax must follow corrections that are large)
      if (sm.w.amax[k % kCoups] < kTame) steps(std::false_type());
      else steps(std::true_type());
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.done[b]);
      others();
    }
  } else if (walks && warp == 1) {
    // ================= the block's deltas, from R's exponentials, to the CTAs with the model; lane = (class half, sample) =================
    const int s = lane & 15, h = lane >> 4;
    float ub[kCh] = {};
    for (uint32_t k = 0; k < nblk; ++k) {
      const int b = k & 1;
      const bool live = k * kB + s < n, upper = s & 4;
      const float f = !decay ? 1.f : live ? sm.qp[min((uint32_t)kB, n - k * kB) - 1 - s] : 0.f;
      wait(&sm.done[b], (k >> 1) & 1);
      const float* eb = sm.w.ebuf[b][s];
      const float4 e0 = *reinterpret_cast<const float4*>(eb), e1 = *reinterpret_cast<const float4*>(eb + 4);
      const float2 e2 = *reinterpret_cast<const float2*>(eb + 8);
      uint32_t hot[kCh];
#pragma unroll
      for (int i = 0; i < kCh; ++i) hot[i] = sm.w.hot[k & 7][h * kCh + i];
      const float inv = rcp(sum_of(e0, e1, e2));   // as R has it
      const float e[kCh] = {h ? e1.y : e0.x, h ? e1.z : e0.y, h ? e1.w : e0.z, h ? e2.x : e0.w, h ? e2.y : e1.x};
      float d[kCh];
      Parts q[kCh];
#pragma unroll
      for (int i = 0; i < kCh; ++i) {
        d[i] = live ? fmaf(e[i], inv, (hot[i] >> s) & 1u ? -1.f : 0.f) : 0.f;
        const float w = d[i] * f, o = shx(w, 4);   // samples s and s + 4 share a word
        q[i] = parts(upper ? o : w, upper ? w : o);
      }
#pragma unroll
      for (int i = 0; i < kCh; ++i) {
        uint32_t* to = &sm.w.dstage[0][h * kCh + i][2 * (s & 3) + (s >> 3)];
        to[upper ? kC * 8 : 0] = upper ? q[i].b : q[i].a;
        if (upper == (i > 2)) to[2 * kC * 8] = q[i].c;
      }
      __syncwarp();
#pragma unroll
      for (int j = lane; j < 3 * kC * 2 && ok; j += 32) {   // (every lane sends some)
        const uint4 v = *reinterpret_cast<const uint4*>(&sm.w.dstage[0][0][4 * j]);
        const uint32_t to = smem_addr(&sm.m.dpart[b][j / (2 * kC)][0][4 * (j % (2 * kC))]), bar = smem_addr(&sm.delta[b]);
#pragma unroll
        for (uint32_t r = 0; r < MC; ++r) send_quad(mma::peer_addr(to, r), v, mma::peer_addr(bar, r));
      }
#pragma unroll
      for (int i = 0; i < kCh; ++i) {   // the biases' update sums
#pragma unroll
        for (int x = 1; x < kB; x *= 2) d[i] += shx(d[i], x);
        ub[i] += d[i];
      }
      if (s == 0) {
#pragma unroll
        for (int i = 0; i < kCh; ++i) sm.w.ub[b][h * kCh + i] = ub[i];
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.bsum[b]);
    }
  } else if (walks && warp == 2) {
    // ================= couplings, summed in rank order, and labels: a block ahead of R =================
    if (p.by_value) asm volatile("griddepcontrol.wait;" ::: "memory");   // (labels: see the producer)
    const ClientData cd = p.by_value ? p.one_client : p.clients[t.client];
    const uint64_t key = p.by_value ? p.one_key : p.sample_keys[t.client];
    auto label = [&](uint32_t k) {
      const uint32_t at = k * kB + lane;
      return lane < kB && at < n ? __ldg(cd.y + sample_index(draw(key, t.sample_ctr0 + at), cd.n)) : -1;
    };
    if (lane == 0) mbar_expect_tx(&sm.bg[0], GC * kSendG0);
    int y = label(0);
    for (uint32_t k = 0; k < (lost ? 0 : nblk); ++k) {
      uint32_t hot = 0;
#pragma unroll
      for (int i = 0; i < kC; ++i) {
        const uint32_t m = __ballot_sync(0xffffffffu, y == i);
        if (lane == i) hot = m;
      }
      if (lane < kB) sm.w.hot[k & 7][lane] = hot;
      if (k + 1 < nblk) y = label(k + 1);
      const int ig = k % kInG, s = lane & 15;
      wait_peer(&sm.bg[ig], (k / kInG) & 1);
      if (k >= kCoups) wait(&sm.done[(k - kCoups) & 1], ((k - kCoups) >> 1) & 1);   // R is done with block k - 3, whose place this is
      ok = __all_sync(0xffffffffu, ok);
      float* out = sm.w.coup[k % kCoups];
      const float* in = &sm.w.gin[ig][0][0];
      float v[8], c[8], big = 0.f;   // (all loads before the first store: the compiler cannot tell them apart)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int tr = 2 * i + (lane >> 4), at = tr * kGp + s;
        v[i] = in[at]; c[i] = in[kOffC + at];
#pragma unroll
        for (int r = 1; r < GC; ++r) { v[i] += in[r * kCoup + at]; c[i] += in[r * kCoup + kOffC + at]; }
        if (s >= tr) v[i] = 0.f;
        if (!k) c[i] = 0.f;
        big = fmaxf(big, fmaxf(fabsf(v[i]), fabsf(c[i])));
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int tr = 2 * i + (lane >> 4), to = s * kGp + ((tr - s - 1) & 15);   // in the order in which R's registers have the samples then
        out[to] = v[i];
        out[kOffC + to] = c[i];
      }
      big = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(big)));
      if (lane == 0) {
        sm.w.amax[k % kCoups] = big;
        if (ok && k + 1 < nblk) mbar_expect_tx(&sm.bg[(k + 1) % kInG], GC * kSendG);
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.rg[k & 3]);
      if (ok && lane < GC && k + kInG < nblk)   // the CTAs that sent them may send block k + 4
        mma::arrive_peer(mma::peer_addr(smem_addr(&sm.gfree[ig]), MC + lane));
    }
  } else if (walks && warp == 3) {
    // ================= logits: the CTAs' parts in rank order, and the biases =================
    const int h = lane >> 4, s = lane & 15;
    float b0[kCh];   // this half's classes at the start of the round
    {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      const size_t at = kD * kC + h * kCh;
#pragma unroll
      for (int i = 0; i < kCh; ++i) b0[i] = p.snaps[(size_t)t.snap_slot * p.stride + at + i];
#pragma unroll 1
      for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
        const InflightRef ref = p.inflight[t.inflight_off + f];
#pragma unroll
        for (int i = 0; i < kCh; ++i) b0[i] = fmaf(-ref.eta, p.U[(size_t)ref.row * p.stride + at + i], b0[i]);
      }
    }
    if (lane == 0) mbar_expect_tx(&sm.bz[0], MC * kZ * 4);
    for (uint32_t k = 0; k < nblk; ++k) {
      const int iz = k % kInZ, b = k & 1;
      float bk[kCh];
#pragma unroll
      for (int i = 0; i < kCh; ++i) bk[i] = kLog2e * b0[i];
      if (k >= 2) {   // (R, too, is done with block k - 2)
        wait(&sm.bsum[b], ((k >> 1) - 1) & 1);
#pragma unroll
        for (int i = 0; i < kCh; ++i) bk[i] = kLog2e * fmaf(neta, sm.w.ub[b][h * kCh + i], b0[i]);
      }
      wait_peer(&sm.bz[iz], (k / kInZ) & 1);
      const float* in = &sm.w.zin[iz][0][h * kCh * kB + s];
      float v[kCh];   // five classes of a sample
#pragma unroll
      for (int i = 0; i < kCh; ++i) {
        v[i] = in[i * kB];
#pragma unroll
        for (int r = 1; r < MC; ++r) v[i] += in[r * kZ + i * kB];
        v[i] += bk[i];
      }
      float m = fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])), v[4]);
      m = fmaxf(m, shx(m, 16));
#pragma unroll
      for (int i = 0; i < kCh; ++i) sm.w.zsum[b][(h * kCh + i) * kGp + s] = v[i] - m;
      if (!ok) sm.w.zsum[b][h * kCh * kGp + s] = kNone;
      if (ok && lane == 0 && k + 1 < nblk) mbar_expect_tx(&sm.bz[(k + 1) % kInZ], MC * kZ * 4);
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.rz[b]);
    }
    // the biases' part of what a round leaves behind
    const int last = (nblk - 1) & 1;
    wait(&sm.bsum[last], ((nblk - 1) >> 1) & 1);
    const float bad = ok ? 0.f : kNone;
#pragma unroll 1
    for (int pass = 0; pass < (p.w_end ? 2 : 1); ++pass) {
      float* row = (pass == 0 ? p.U : p.w_end) + (size_t)t.u_row * p.stride;
      if (s == 0) {
#pragma unroll
        for (int i = 0; i < kCh; ++i) {
          const float u = sm.w.ub[last][h * kCh + i];
          row[kD * kC + h * kCh + i] = (pass == 0 ? u : fmaf(neta, u, b0[i])) + bad;
        }
      }
      if (p.stride && lane < kStageFloats - kParams) row[kParams + lane] = 0.f;   // the row's padding
    }
  } else if (!walks && warp == kWarps - 1) {
    // ================= producer: rows =================
    // Inside a handle rows and labels are older than the set-up launch of the run, which lets nothing start early; without
    // one they are the caller's, whose kernel ahead in the stream may still be writing them.
    if (p.by_value) asm volatile("griddepcontrol.wait;" ::: "memory");
    const ClientData cd = p.by_value ? p.one_client : p.clients[t.client];
    const uint64_t key = p.by_value ? p.one_key : p.sample_keys[t.client];
    const float* xrows = reinterpret_cast<const float*>(cd.x) + 8 * ks0;
    const uint32_t bytes = 32u * cnt;
    for (uint32_t kb = 0; kb < (lost ? 0 : nblk); ++kb) {
      const int sb = kb % NS;
      if (kb >= (uint32_t)NS) wait(&sm.freed[sb], (kb / NS - 1) & 1);   // block kb - NS has left its slot
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint32_t nvb = min((uint32_t)kB, n - kb * kB);
      float* const slot = rows + sb * kB * pitch;
      for (uint32_t r = nvb; r < (uint32_t)kB; ++r)   // short last block: rows that add nothing anywhere
        for (int i = lane; i < 8 * cnt; i += 32) slot[r * pitch + i] = 0.f;
      if (lane == 0) mbar_expect_only(&sm.full[sb], nvb * bytes);
      __syncwarp();
      if ((uint32_t)lane < nvb) {
        const uint32_t idx = sample_index(draw(key, t.sample_ctr0 + (uint64_t)kb * kB + lane), cd.n);
        bulk_load(slot + lane * pitch, xrows + (size_t)idx * kD, bytes, &sm.full[sb]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.full[sb]);
    }
  } else if (!models && !walks && warp < NG) {
    // ================= Gram warps; lane = 4 g + tt =================
    const int g = lane >> 2, tt = lane & 3;
    float* const gpart = &sm.g.part[0][0][0];
    const uint32_t grank = rank - MC;
    launch_next();
    Split pv[KG][4];   // the rows of the block before, split
    int slot = 0;      // kb mod kGramParts
    for (uint32_t kb = 0; kb < nblk; ++kb) {
      wait(&sm.full[kb % NS], (kb / NS) & 1);
      const float* xr = rows + ((kb % NS) * kB + g) * PG + 8 * warp + 2 * tt;
      float gh[2][4] = {}, gs[2][4] = {}, hh[2][4] = {}, cx[2][4] = {};
#pragma unroll
      for (int j = 0; j < KG; ++j) {
        const float2 x0 = *reinterpret_cast<const float2*>(xr + 8 * NG * j);
        const float2 x1 = *reinterpret_cast<const float2*>(xr + 8 * PG + 8 * NG * j);
        const Split a = split_t(x0.x), b = split_t(x0.y), c = split_t(x1.x), d = split_t(x1.y);
        mma::tf32(gh[0], a.hi, c.hi, b.hi, d.hi, a.hi, b.hi);
        mma::tf32(gh[1], a.hi, c.hi, b.hi, d.hi, c.hi, d.hi);
        mma::tf32(gs[0], a.hi, c.hi, b.hi, d.hi, a.lo, b.lo);
        mma::tf32(gs[1], a.hi, c.hi, b.hi, d.hi, c.lo, d.lo);
        if (kb) {
          Split e, f, u, v;
          e = pv[j][0]; f = pv[j][1]; u = pv[j][2]; v = pv[j][3];
          mma::tf32(hh[0], a.hi, c.hi, b.hi, d.hi, e.hi, f.hi);
          mma::tf32(hh[1], a.hi, c.hi, b.hi, d.hi, u.hi, v.hi);
          mma::tf32(cx[0], a.lo, c.lo, b.lo, d.lo, e.hi, f.hi);
          mma::tf32(cx[1], a.lo, c.lo, b.lo, d.lo, u.hi, v.hi);
          mma::tf32(cx[0], a.hi, c.hi, b.hi, d.hi, e.lo, f.lo);
          mma::tf32(cx[1], a.hi, c.hi, b.hi, d.hi, u.lo, v.lo);
        }
        { pv[j][0] = a; pv[j][1] = b; pv[j][2] = c; pv[j][3] = d; }
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.freed[kb % NS]);
      float* const block = gpart + slot * NG * kCoup;
      slot = slot + 1 < kGramParts ? slot + 1 : 0;
      float* part = block + warp * kCoup;
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2) {
          // below the diagonal hi.hi + hi.lo, above it hi.lo: x_r . x_c = part[r][c] + part[c][r] for r > c
          const int r = g + 8 * r2, s = 8 * m + 2 * tt;
          *reinterpret_cast<float2*>(part + r * kGp + s) =
              make_float2(gs[m][2 * r2] + (r > s ? gh[m][2 * r2] : 0.f), gs[m][2 * r2 + 1] + (r > s + 1 ? gh[m][2 * r2 + 1] : 0.f));
          *reinterpret_cast<float2*>(part + kOffC + r * kGp + s) =
              make_float2(hh[m][2 * r2] + cx[m][2 * r2], hh[m][2 * r2 + 1] + cx[m][2 * r2 + 1]);
        }
      if (!ok)
        for (int i = 0; i < kCoup; ++i) part[i] = kNone;
      // Half of the warps add up a block's parts while the others are at the next block's products: they only say that theirs are
      // there.  A barrier per parity.  A warp that writes block kb has waited at kb - 1 or at kb - 2, whichever its half adds up, and every
      // warp arrives there behind its sums of block kb - 3: those have been read.  The sums of kb - 2 may not have been: warps of one half
      // do not wait for one another between two of their blocks.  Hence three buffers, not two.
      const int first = kb & 1 ? kNgEven : 0, sums = kb & 1 ? NG - kNgEven : kNgEven;
      if (warp < first || warp >= first + sums) {
        asm volatile("bar.arrive %0, %1;" ::"r"(2 + (kb & 1)), "n"(NG * 32) : "memory");
        continue;
      }
      asm volatile("bar.sync %0, %1;" ::"r"(2 + (kb & 1)), "n"(NG * 32) : "memory");
      // sums over the warps, in warp order, with the factors of the couplings; sent to the walker
      const int ig = kb % kInG;
      const float one = grank == 0 ? scale : 0.f;   // the bias input's part of a coupling
      // two entries per thread: 64 pairs that reach below the diagonal, 128 of the matrix to the block before
      if (kb >= kInG) wait_peer(&sm.gfree[ig], (kb / kInG - 1) & 1);   // the walker has taken block kb - 4
      for (int e = (warp - first) * 32 + lane; e < (kb ? 192 : 64) && ok; e += sums * 32) {
        const bool own = e < 64;
        int tr, s0;
        if (own) {   // rows 2q + 1 and 2q + 2 have q + 1 pairs each, q = 0 .. 6; row 15 eight
          const int q = e < 2 ? 0 : e < 6 ? 1 : e < 12 ? 2 : e < 20 ? 3 : e < 30 ? 4 : e < 42 ? 5 : e < 56 ? 6 : 7, r = e - q * (q + 1);
          tr = 2 * q + 1 + (r > q ? 1 : 0);
          s0 = 2 * (r > q ? r - q - 1 : r);
        } else {
          tr = (e - 64) >> 3; s0 = 2 * (e & 7);
        }
        const float* from = block + (own ? 0 : kOffC) + tr * kGp + s0;
        float v0 = 0.f, v1 = 0.f;
#pragma unroll
        for (int w = 0; w < NG; ++w) {
          const float2 x = *reinterpret_cast<const float2*>(from + w * kCoup);
          v0 += x.x; v1 += x.y;
        }
        if (own) {
          const float* up = block + s0 * kGp + tr;
#pragma unroll
          for (int w = 0; w < NG; ++w) { v0 += up[w * kCoup]; v1 += up[w * kCoup + kGp]; }
        }
        float f0 = scale, f1 = scale;
        if (decay) {
          f0 *= sm.qp[own ? tr - 1 - s0 : tr + kB - 1 - s0];
          f1 *= sm.qp[own ? max(tr - 2 - s0, 0) : tr + kB - 2 - s0];
        }
        v0 = fmaf(v0, f0, one);
        v1 = own && s0 + 1 >= tr ? 0.f : fmaf(v1, f1, one);
        send_pair(mma::peer_addr(smem_addr(&sm.w.gin[ig][grank][(own ? 0 : kOffC) + tr * kGp + s0]), kWalker), v0, v1,
                  mma::peer_addr(smem_addr(&sm.bg[ig]), kWalker));
      }
    }
  } else if (models && warp < NM) {
    // ================= model warps; lane = 4 g + tt =================
    const int g = lane >> 2, tt = lane & 3;
    const bool two = g < kC - 8;               // this lane holds a class of the second eight
    float U[KM][4], ws[KM][4];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    {
      auto load = [&](const float* src, float (&v)[KM][4]) {
#pragma unroll
        for (int j = 0; j < KM; ++j) {
          const int i = warp + j * NM;
          const bool in = i < cnt;
          const int at = (8 * (ks0 + i) + 2 * tt) * kC + g;
          v[j][0] = in ? src[at] : 0.f;
          v[j][1] = in ? src[at + kC] : 0.f;
          v[j][2] = in && two ? src[at + 8] : 0.f;
          v[j][3] = in && two ? src[at + kC + 8] : 0.f;
        }
      };
      load(p.snaps + (size_t)t.snap_slot * p.stride, ws);
#pragma unroll 1
      for (uint32_t f = 0; f < t.inflight_cnt; ++f) {   // own update sums still on their way to the server
        const InflightRef ref = p.inflight[t.inflight_off + f];
        load(p.U + (size_t)ref.row * p.stride, U);
#pragma unroll
        for (int j = 0; j < KM; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) ws[j][c] = fmaf(-ref.eta, U[j][c], ws[j][c]);
      }
#pragma unroll
      for (int j = 0; j < KM; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) U[j][c] = 0.f;
    }
    float qw = 1.f;      // q^(samples in U): W = qw W_start - eta U
    double qwd = 1.0;

    // block kb's logits follow the update by block kb - 2: everything R needs is one block ahead of it
    for (uint32_t kb = 0; kb < nblk + 2; ++kb) {
      if (kb == early) launch_next();
      const bool update = kb >= 2, look = kb < nblk;
      const uint32_t k = update ? kb - 2 : 0, nv = min((uint32_t)kB, n - k * kB);
      // the rows of block k as the update's second operand ([sample][pixel], pixel g of the warp's k-steps), and those of block kb
      const float* xb = rows + ((k % NS) * kB + tt) * PM + 8 * warp + g;
      const float* xr = rows + ((kb % NS) * kB + g) * PM + 8 * warp + 2 * tt;
      auto rows_of = [&](int j, Parts (&x)[2]) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const float* at = xb + 8 * m * PM + 8 * NM * j;
          x[m] = parts_t(at[0], at[4 * PM]);
        }
      };
      auto inputs_of = [&](int j, Split (&x)[4]) {
        const float2 x0 = *reinterpret_cast<const float2*>(xr + 8 * NM * j), x1 = *reinterpret_cast<const float2*>(xr + 8 * PM + 8 * NM * j);
        x[0] = split_r(x0.x); x[1] = split_r(x0.y); x[2] = split_r(x1.x); x[3] = split_r(x1.y);
      };
      Parts xu[KM][2];
      Split xi[KM][4];
      if (update) {
#pragma unroll
        for (int j = 0; j < KM; ++j) rows_of(j, xu[j]);
      }
      if (look) {
        wait(&sm.full[kb % NS], (kb / NS) & 1);
#pragma unroll
        for (int j = 0; j < KM; ++j) inputs_of(j, xi[j]);
      }
      if (update) {
        // ---- U^T = q^nv U^T + sum_s q^(nv-1-s) delta_s x_s; the k index of the product is read as samples t, t + 4, t + 8, t + 12 ----
        wait_peer(&sm.delta[k & 1], (k >> 1) & 1);
        if (ok && threadIdx.x == 0 && kb < nblk) mbar_expect_tx(&sm.delta[k & 1], kSendD);   // for block k + 2
        uint32_t aa[4], ab[4], ac[4];
        {
          const uint32_t* at = &sm.m.dpart[k & 1][0][g][2 * tt];
          auto part_of = [&](int q, uint32_t (&a)[4]) {
            const uint2 x = *reinterpret_cast<const uint2*>(at + q * kB * 8), y = *reinterpret_cast<const uint2*>(at + q * kB * 8 + 64);
            a[0] = x.x; a[1] = y.x; a[2] = x.y; a[3] = y.y;
          };
          part_of(0, aa); part_of(1, ab); part_of(2, ac);
        }
        if (decay) {   // U decays with the block, and with it the share of the start model
          const float qn = sm.qp[nv];
#pragma unroll
          for (int j = 0; j < KM; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) U[j][c] *= qn;
          qwd *= sm.qd[nv];
          qw = (float)qwd;
        }
        // k-steps side by side, and small terms in two accumulators: the products of one depend on one another
        float d[KM][4] = {}, e[KM][4] = {}, f[KM][4] = {};
#pragma unroll
        for (int term = 0; term < 6; ++term)
#pragma unroll
          for (int j = 0; j < KM; ++j) {
            const Parts &x0 = xu[j][0], &x1 = xu[j][1];
            if (term == 0) mma::mma_bf16(e[j], ac, x0.a, x1.a);
            if (term == 1) mma::mma_bf16(f[j], aa, x0.c, x1.c);
            if (term == 2) mma::mma_bf16(d[j], aa, x0.a, x1.a);
            if (term == 3) mma::mma_bf16(f[j], ab, x0.b, x1.b);
            if (term == 4) mma::mma_bf16(e[j], ab, x0.a, x1.a);
            if (term == 5) mma::mma_bf16(f[j], aa, x0.b, x1.b);
          }
#pragma unroll
        for (int j = 0; j < KM; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) U[j][c] += d[j][c] + (e[j][c] + f[j][c]);
      }
      if (look) {
        // ---- logits of block kb with the model W = qw W_start - eta U ----
        float zm[2][4] = {}, zx[2][4] = {}, zy[2][4] = {};
#pragma unroll
        for (int j = 0; j < KM; ++j) {
          const Split (&x)[4] = xi[j];
          const Split w0 = split_r(fmaf(neta, U[j][0], qw * ws[j][0])), w2 = split_r(fmaf(neta, U[j][1], qw * ws[j][1]));
          const Split w1 = split_r(fmaf(neta, U[j][2], qw * ws[j][2])), w3 = split_r(fmaf(neta, U[j][3], qw * ws[j][3]));
          mma::tf32(zm[0], w0.hi, w1.hi, w2.hi, w3.hi, x[0].hi, x[1].hi);
          mma::tf32(zm[1], w0.hi, w1.hi, w2.hi, w3.hi, x[2].hi, x[3].hi);
          mma::tf32(zx[0], w0.lo, w1.lo, w2.lo, w3.lo, x[0].hi, x[1].hi);
          mma::tf32(zx[1], w0.lo, w1.lo, w2.lo, w3.lo, x[2].hi, x[3].hi);
          mma::tf32(zy[0], w0.hi, w1.hi, w2.hi, w3.hi, x[0].lo, x[1].lo);
          mma::tf32(zy[1], w0.hi, w1.hi, w2.hi, w3.hi, x[2].lo, x[3].lo);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) { zx[0][c] += zy[0][c]; zx[1][c] += zy[1][c]; }
        float* const zpart = &sm.m.zpart[kb & 1][0][0];
        float* const mypart = zpart + warp * kZ;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int s = 8 * m + 2 * tt;
          float f0 = kLog2e, f1 = kLog2e;
          if (decay) { f0 *= sm.qp[s + (kb ? kB : 0)]; f1 *= sm.qp[s + 1 + (kb ? kB : 0)]; }
          *reinterpret_cast<float2*>(mypart + g * kB + s) = make_float2((zm[m][0] + zx[m][0]) * f0, (zm[m][1] + zx[m][1]) * f1);
          if (two)
            *reinterpret_cast<float2*>(mypart + (8 + g) * kB + s) = make_float2((zm[m][2] + zx[m][2]) * f0, (zm[m][3] + zx[m][3]) * f1);
        }
        if (!ok) mypart[0] = kNone;   // (the first sample is one of the round's in every block)
        asm volatile("bar.sync 1, %0;" ::"n"(NM * 32) : "memory");
        // sums over the warps, in warp order; sent to the walker
        if (warp < 2) {
          const int iz = kb % kInZ, e = warp * 32 + lane;
          if (e < kQuadZ && ok) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < NM; ++w) {
              const float4 x = *reinterpret_cast<const float4*>(zpart + w * kZ + 4 * e);
              v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            mma::send_peer(mma::peer_addr(smem_addr(&sm.w.zin[iz][rank][4 * e]), kWalker), v, mma::peer_addr(smem_addr(&sm.bz[iz]), kWalker));
          }
        }
      }
      if (update) {
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&sm.freed[k % NS]);
      }
    }

    // ---- event trigger: h reached s_{i,c}; publish U_i (and the end model) ----
    {
      const float bad = ok ? 0.f : kNone;
      const float c1 = (decay ? (float)((1.0 - qwd) / (double)eta) : 0.f) + bad;
      qw += bad;
#pragma unroll 1
      for (int pass = 0; pass < (p.w_end ? 2 : 1); ++pass) {
        float* row = (pass == 0 ? p.U : p.w_end) + (size_t)t.u_row * p.stride;
        const float fw = pass == 0 ? c1 : qw, fu = pass == 0 ? 1.f : neta;
        __syncwarp();   // the second pass starts with the buffer the first one ended with, where KM is odd
#pragma unroll
        for (int j = 0; j < KM; ++j) {   // a k-step's 80 parameters through the warp's own buffer: whole lines out
          float* st = sm.m.zpart[j & 1][warp];
          const int i = warp + j * NM, at = 2 * tt * kC + g;
          st[at] = fmaf(fu, U[j][0], fw * ws[j][0]);
          st[at + kC] = fmaf(fu, U[j][1], fw * ws[j][1]);
          if (two) {
            st[at + 8] = fmaf(fu, U[j][2], fw * ws[j][2]);
            st[at + kC + 8] = fmaf(fu, U[j][3], fw * ws[j][3]);
          }
          __syncwarp();
          if (i < cnt && lane < 20)
            *reinterpret_cast<float4*>(row + 80 * (ks0 + i) + 4 * lane) = *reinterpret_cast<const float4*>(st + 4 * lane);
        }
      }
    }
  }
  if (!ok && p.status && lane == 0) atomicOr(p.status, 1u);
  mma::cluster_sync();   // no CTA leaves while a peer may still send to it
  if (!ok) linger();
  if (!ok && !walks && warp == kWarps - 1)   // copies still in flight target this CTA's shared memory: a bounded chance to land
    for (int s = 0; s < NS; ++s) {
      mbar_wait_limit(&sm.full[s], 0, min(limit, 1u << 16));
      mbar_wait_limit(&sm.full[s], 1, min(limit, 1u << 16));
    }
  if (threadIdx.x == 0 && rank == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = n; rec.flags = 1;
    p.trig[t.seq] = rec;
  }
}

typedef Shape<3, 11, 3, 2, 5> Six;
typedef Shape<4, 9, 3, 3, 3> Eight;

template <class S, bool LOSE>
cudaError_t launch(const RoundLaunch& p, cudaStream_t s) {
  static std::atomic<uint64_t> opted_in{0};   // a bit per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
  if (!(opted_in.load(std::memory_order_relaxed) & bit)) {
    e = cudaFuncSetAttribute(lr_relay_kernel<S, LOSE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(typename S::Smem));
    if (e != cudaSuccess) return e;
    opted_in.fetch_or(bit, std::memory_order_relaxed);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.n_tasks * S::kCl, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = sizeof(typename S::Smem);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = S::kCl;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, lr_relay_kernel<S, LOSE>, p);
}

}  // namespace

cudaError_t launch_lr_relay_rounds(const RoundLaunch& p, uint32_t cluster, cudaStream_t s) {
  if (p.lose) return cluster == 8 ? launch<Eight, true>(p, s) : launch<Six, true>(p, s);
  return cluster == 8 ? launch<Eight, false>(p, s) : launch<Six, false>(p, s);
}

}  // namespace aet
