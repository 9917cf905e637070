// Local-SGD round of one client for softmax regression 784 -> 10, batch 1, for launches of 16 to 74 round-tasks that lr_relay_kernel.cu
// does not take: what counts is the length of a round's chain of dependent steps.
//
// Algorithm 3, MainComputeNode, inner loop (g = grad f(w_c, xi) + lambda W; w_c -= eta g; U_i += g; h++) sixteen
// steps at a time.  With q = 1 - eta lambda, W_k, b_k the model at the start of block k and
// delta_s = softmax(z_s) - onehot(y_s), step t of block k sees
//     z_t = q^t W_k x_t + b_k + sum_{s<t} L[t][s] delta_s,              L[t][s] = -eta (q^(t-1-s) x_s.x_t + 1),
// and because W_{k+1} = q^16 W_k - eta sum_s q^(15-s) delta_s x_s, step t of block k + 1 sees
//     z_t = q^(t+16) W_k x_t + b_k + sum_{s in block k} C[t][s] delta_s + sum_{s<t} L[t][s] delta_s,
//                                                                         C[t][s] = -eta (q^(t+15-s) x_s.x_t + 1):
// everything but the two small sums is known one block ahead.  So the chain of a round is the recurrence alone, and
// the rest of the work - two products with the 784 inputs and two 16 x 16 Gram matrices per block - runs beside it:
//   R warp       walks the blocks: z from the prepared logits and the previous block's deltas, then sweeps
//                z <- z0 + L delta(z) over the sixteen samples at once until they no longer move (below), delta out;
//   model warps  as soon as delta_k is out: U^T += delta^T X of block k (tensor cores), then the logits of block k + 2
//                with the model that gives;
//   Gram warps   the products of the rows of a block with one another and with those of the block before;
//   producer     row copies and labels, as soon as a block has left its slot;
//   sum warp     adds the CTAs' parts of the couplings.
// Partial sums over warps and CTAs are added in a fixed order.
// Few round-tasks leave SMs idle, so a round-task takes a cluster of 4 or 2 CTAs, each with its range of the
// inputs (98 k-steps of 8); the recurrence is repeated in every CTA (same inputs, same order: the same bits).
//
// Logits and Gram matrices are m16n8k8 tf32 products on split operands, the update m16n8k16 bf16 products on operands in three
// parts (mma_common.cuh): what it loses stays in U, and with tf32 a round of 50 samples was 1.5e-7 off fp64 instead of 0.6e-7
// (fp32 FMAs 0.7e-7), for 1 to 3 % of the time of few long chains.  The logits' heads are rounded, not cut: a round of 5 samples
// 5.1e-8 -> 4.0e-8 (FMAs 4.0e-8 to 4.3e-8), for another percent.  U^T[class][pixel] accumulates in the fragment
// (class g, pixels 2t, 2t + 1), which is the A fragment of the logits product Z^T = W^T X^T when the k index of a step
// is read as pixel (2t | 2t + 1): W = q^n W_start - eta U is formed in place.  A block's sum starts from zero and is
// added to U by an fp32 add, so that the tensor cores' own rounding never accumulates over a round.
//
// With lambda the kernel carries D = sum_s q^(n-1-s) delta_s x_s; U = D + W_start (1 - q^n) / eta (the sum of
// delta_s x_s + lambda W_s; both factors from double precision).
//
// Stopping the sweeps.  The solution satisfies z = z0 + L delta(z), L strictly lower triangular, softmax 1/2-Lipschitz in
// the maximum norm.  A sweep that moves z by at most d leaves it within (1 + a)^15 (r / 2) d of the solution,
// a = max |L| / 2, r = max_t sum_s |L[t][s]| (the inverse of a unit triangular matrix with entries below a).  Sweep i
// makes the first i samples exact, so at most fifteen are needed whatever the coupling.
//
// What bounds it: the latency of the recurrence, about 400 cycles a sweep, and the products' (the two in turn on one SM).  Measured
// against eight steps at a time on one CTA: rounds of 400 samples, 33 clients 88 instead of 161 us.
#include <cuda_runtime.h>

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
constexpr int kCoup = 2 * kB * kGp;          // own couplings [t][s], then those to the block before
constexpr int kOffC = kB * kGp;
constexpr int kQuadZ = kZ / 4;               // the logits as 16-byte pieces; a matrix has 64
// bytes a CTA sends about a block: the own couplings' pieces that reach below the diagonal, and the others'
constexpr uint32_t kSendG0 = 16 * 36, kSendG = kSendG0 + 16 * 64;
constexpr int kDbuf = 2 * kB * kCh;
constexpr float kTol = 2e-7f * kLog2e;       // logits are kept in units of log2

// CL CTAs per round-task; per CTA NM model warps with KM k-steps each, NG Gram warps with KG each, NS blocks of rows.
// QUIET: the recurrence has a scheduler to itself and the two light warps.
template <int CL, int NM, int KM, int NG, int KG, int NS, bool QUIET>
struct Shape {
  static constexpr int kCl = CL, kNm = NM, kKm = KM, kNg = NG, kKg = KG, kNs = NS;
  static constexpr bool kQuiet = QUIET;
  static constexpr int kMost = (kSteps8 + CL - 1) / CL;            // k-steps of the widest CTA
  static constexpr int kCols = 8 * (NM * KM > NG * KG ? NM * KM : NG * KG);
  // row pitch = 8 or 24 mod 32 floats: the fragment loads of eight rows then hit 32 different banks
  static constexpr int kPitch = kCols % 16 == 8 ? kCols : kCols + 8;
  // Rings of what CTAs send one another.  A CTA that has the deltas of block k knows that its peers have taken what
  // belongs to block k - 2; it may itself be sending logits of block k + 2 and couplings of block k + NS.
  static constexpr int kInZ = 4, kInG = NS + 2;
  static constexpr int kWarps = QUIET ? (NM + NG + 2) / 3 * 4 : NM + NG + 3;
  static constexpr int kThreads = kWarps * 32;
  static constexpr bool kCarry = KG <= 7;   // Gram warps keep the split rows of the block before in registers
  static_assert(!QUIET || (NM + NG > 6 && NM + NG <= 12), "three schedulers for the products, the fourth for the rest");
  static_assert(NM >= 2 && NG >= 4, "one 16-byte piece per thread");
  static_assert(NM * KM >= kMost && NG * KG >= kMost, "every k-step has a warp");
  struct __align__(128) Smem {
    float rows[NS][kB][kPitch];
    float zpart[2][NM][kZ];         // per warp: products not yet summed over the warps
    float gpart[2][NG][kCoup];
    float zin[kInZ][CL][kZ];        // per CTA of the cluster
    float gin[kInG][CL][kCoup];
    float coup[2][kCoup];   // summed over the cluster
    float zsum[2][kZ];
    float dbuf[2][2][kB * kCh];     // deltas by parity of the block and class half: [sample][five classes]
    uint32_t amax[2];               // largest coupling, as bits
    float qp[32];                   // powers of q
    int ys[8][kB];
    uint64_t full[NS], freed[NS];
    uint64_t bz[kInZ], bg[kInG], ready[2], delta[2];
  };
};

__device__ __forceinline__ uint32_t warp_max(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
enum Role { kModel, kGram, kRec, kProd, kSum, kIdle };

template <class S>
__global__ void __launch_bounds__(S::kThreads, 1) lr_chain_kernel(RoundLaunch p) {
  constexpr int CL = S::kCl, NM = S::kNm, KM = S::kKm, NG = S::kNg, KG = S::kKg, NS = S::kNs;
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
  const int lane = threadIdx.x & 31;
  int role, warp;   // what this warp does, and its number among those that do the same
  {
    const int w = threadIdx.x >> 5;
    int id;         // products first, then the others
    if (S::kQuiet) id = (w & 3) == 3 ? NM + NG + (w >> 2) : (w >> 2) * 3 + (w & 3) < NM + NG ? (w >> 2) * 3 + (w & 3) : NM + NG + 3;
    else id = w;
    if (id < NM) { role = kModel; warp = id; }
    else if (id < NM + NG) { role = kGram; warp = id - NM; }
    else { role = min(kRec + (id - NM - NG), (int)kIdle); warp = 0; }
  }
  const uint32_t n = t.n_samples, nblk = (n + kB - 1) / kB;
  const float eta = t.eta, neta = -t.eta;
  const bool decay = p.l2 != 0.f;
  // this CTA's k-steps [ks0, ks0 + cnt)
  const int ks0 = (int)rank * (kSteps8 / CL) + min((int)rank, kSteps8 % CL);
  const int cnt = kSteps8 / CL + ((int)rank < kSteps8 % CL ? 1 : 0);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) { mbar_init(&sm.full[s], 1); mbar_init(&sm.freed[s], NM + NG); }
    for (int s = 0; s < S::kInZ; ++s) mbar_init(&sm.bz[s], 1);
    for (int s = 0; s < S::kInG; ++s) mbar_init(&sm.bg[s], 1);
    for (int s = 0; s < 2; ++s) { mbar_init(&sm.ready[s], 1); mbar_init(&sm.delta[s], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    double q = 1.0 - (double)eta * (double)p.l2, v = 1.0;
    for (int i = 0; i < 32; ++i) { sm.qp[i] = (float)v; v *= q; }
  }
  for (int i = threadIdx.x; i < 2 * kDbuf; i += S::kThreads) (&sm.dbuf[0][0][0])[i] = 0.f;
  for (int i = threadIdx.x; i < NS * kB; i += S::kThreads)   // columns no copy writes: inputs that add nothing
    for (int c = 8 * cnt; c < S::kCols; ++c) sm.rows[i / kB][i % kB][c] = 0.f;
  mma::cluster_sync();   // a peer's barriers exist before anything is sent to it

  // A thread whose wait has given up waits no more and runs through on whatever is there, but neither arms a barrier (a second arrival
  // on one that is short of bytes would be invalid) nor sends: whoever depends on it gives up in turn, the status word is set, and
  // every CTA of the cluster reaches the end.
  bool ok = true;
  auto wait = [&](uint64_t* bar, uint32_t parity) { if (ok) ok = mbar_wait(bar, parity); };
  auto wait_cluster = [&](uint64_t* bar, uint32_t parity) {   // for what peers sent
    const uint32_t at = smem_addr(bar);
    for (uint32_t i = 0; ok; ++i) {
      if (mma::try_wait_cluster(at, parity)) break;
      if (i >= kWaitLimit) ok = false;
    }
  };
  const float scale = neta * kLog2e;

  if (role == kRec) {
    // ================= R: the recurrence; lane = (sample, class half) =================
    const int s_mine = lane & 15, h = lane >> 4;
    const float* dall0 = &sm.dbuf[0][h][0];
    for (uint32_t k = 0; k < nblk; ++k) {
      const int b = k & 1;
      const uint32_t nv = min((uint32_t)kB, n - k * kB);
      wait(&sm.ready[b], (k >> 1) & 1);
      const float* in = sm.coup[b];
      const float* zi = sm.zsum[b];
      float z0[kCh], L[kB];
#pragma unroll
      for (int c = 0; c < kCh; ++c) z0[c] = zi[(h * kCh + c) * kB + s_mine];
      const float4* lr4 = reinterpret_cast<const float4*>(in + s_mine * kGp);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = lr4[i];
        L[4 * i] = v.x; L[4 * i + 1] = v.y; L[4 * i + 2] = v.z; L[4 * i + 3] = v.w;
      }
      const float amax = __uint_as_float(sm.amax[b]);
      const int y = sm.ys[k & 7][s_mine];
      // acc[c] += sum over s < cnt of f[s] delta[s][c]; deltas lie [sample][class] in a class half, five apart
      auto add_deltas = [&](const float* d, const float (&f)[kB], float (&acc)[kCh]) {
        float v[4 * ((kB * kCh + 3) / 4)];
#pragma unroll
        for (int i = 0; i < kB * kCh / 4; ++i) {
          const float4 x = reinterpret_cast<const float4*>(d)[i];
          v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
        }
#pragma unroll
        for (int s = 0; s < kB; ++s)
#pragma unroll
          for (int c = 0; c < kCh; ++c) acc[c] = fmaf(f[s], v[s * kCh + c], acc[c]);
      };
      if (k) {   // what the deltas of the block before add
        float cf[kB];
        const float4* cr = reinterpret_cast<const float4*>(in + kOffC + s_mine * kGp);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 v = cr[i];
          cf[4 * i] = v.x; cf[4 * i + 1] = v.y; cf[4 * i + 2] = v.z; cf[4 * i + 3] = v.w;
        }
        add_deltas(dall0 + (b ^ 1) * kDbuf, cf, z0);
      }
      // amax is in units of log2 as the logits are; (1 + a)^15 <= exp(15 a)
      const float gain = 7.5f / kLog2e * amax * ex2(fminf(7.5f * amax, 60.f));
      const bool wild = amax > 4.f;   // the shift of the softmax must follow the corrections
      float oh[kCh];
#pragma unroll
      for (int c = 0; c < kCh; ++c) oh[c] = h * kCh + c == y ? -1.f : 0.f;
      auto top = [&](const float (&z)[kCh]) {
        float m = fmaxf(fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])), z[4]);
        return fmaxf(m, shx(m, 16));
      };
      {
        const float m = top(z0);
#pragma unroll
        for (int c = 0; c < kCh; ++c) z0[c] -= m;
      }
      float z[kCh], d[kCh];
#pragma unroll
      for (int c = 0; c < kCh; ++c) z[c] = z0[c];
      const float* dall = dall0 + b * kDbuf;
      float* dmine = const_cast<float*>(dall) + s_mine * kCh;
      const bool live = (uint32_t)s_mine < nv;
      const float need = live ? kTol : 3e38f;
      uint32_t left = nv - 1;   // sweeps that can still be needed
      while (true) {
        float e[kCh];
        if (wild) {
          const float m = top(z);
#pragma unroll
          for (int c = 0; c < kCh; ++c) e[c] = ex2(z[c] - m);
        } else {
#pragma unroll
          for (int c = 0; c < kCh; ++c) e[c] = ex2(z[c]);
        }
        float sum = ((e[0] + e[1]) + (e[2] + e[3])) + e[4];
        sum += shx(sum, 16);
        const float inv = rcp(sum);
#pragma unroll
        for (int c = 0; c < kCh; ++c) d[c] = fmaf(e[c], inv, oh[c]);
        if (!left) break;
        --left;
#pragma unroll
        for (int c = 0; c < kCh; ++c) dmine[c] = d[c];
        __syncwarp();
        float zn[kCh];
#pragma unroll
        for (int c = 0; c < kCh; ++c) zn[c] = z0[c];
        add_deltas(dall, L, zn);   // (L is zero from the diagonal on)
        const float change = fmaxf(fmaxf(fmaxf(fabsf(zn[0] - z[0]), fabsf(zn[1] - z[1])), fmaxf(fabsf(zn[2] - z[2]), fabsf(zn[3] - z[3]))),
                                   fabsf(zn[4] - z[4]));
#pragma unroll
        for (int c = 0; c < kCh; ++c) z[c] = zn[c];
        if (!__any_sync(0xffffffffu, !(change * gain <= need)) && !p.step_by_step) left = 0;
        __syncwarp();
      }
#pragma unroll
      for (int c = 0; c < kCh; ++c) dmine[c] = live ? d[c] : 0.f;
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.delta[b]);
    }
  } else if (role == kProd) {
    // ================= producer: rows and labels =================
    // Inside a handle rows and labels are older than the set-up launch of the run, which lets nothing start early; without
    // one they are the caller's, whose kernel ahead in the stream may still be writing them.
    if (p.by_value) asm volatile("griddepcontrol.wait;" ::: "memory");
    const ClientData cd = p.by_value ? p.one_client : p.clients[t.client];
    const uint64_t key = p.by_value ? p.one_key : p.sample_keys[t.client];
    const float* xrows = reinterpret_cast<const float*>(cd.x) + 8 * ks0;
    const uint32_t bytes = 32u * cnt;
    for (uint32_t kb = 0; kb < nblk; ++kb) {
      const int sb = kb % NS;
      if (kb >= (uint32_t)NS) wait(&sm.freed[sb], (kb / NS - 1) & 1);   // block kb - NS has left its slot
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint32_t nvb = min((uint32_t)kB, n - kb * kB);
      for (uint32_t r = nvb; r < (uint32_t)kB; ++r)   // short last block: rows that add nothing anywhere
        for (int i = lane; i < 8 * cnt; i += 32) sm.rows[sb][r][i] = 0.f;
      if (lane == 0) mbar_expect_only(&sm.full[sb], nvb * bytes);
      __syncwarp();
      if ((uint32_t)lane < nvb) {
        const uint32_t idx = sample_index(draw(key, t.sample_ctr0 + (uint64_t)kb * kB + lane), cd.n);
        bulk_load(sm.rows[sb][lane], xrows + (size_t)idx * kD, bytes, &sm.full[sb]);
        sm.ys[kb & 7][lane] = __ldg(cd.y + idx);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.full[sb]);
    }
  } else if (role == kSum) {
    // ================= the CTAs' parts, summed in rank order =================
    if (lane == 0) {
      mbar_expect_tx(&sm.bg[0], CL * kSendG0);
      mbar_expect_tx(&sm.bz[0], CL * kZ * 4);
    }
    for (uint32_t k = 0; k < nblk; ++k) {
      const int ig = k % S::kInG, b = k & 1;
      const int iz = k % S::kInZ;
      wait_cluster(&sm.bg[ig], (k / S::kInG) & 1);
      if (k >= 2) wait(&sm.delta[b], ((k >> 1) - 1) & 1);   // R has taken block k - 2
      float* out = sm.coup[b];
      float big = 0.f;
      const int s = lane & 15;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int tr = 2 * i + (lane >> 4), at = tr * kGp + s;
        float v = sm.gin[ig][0][at], c = sm.gin[ig][0][kOffC + at];
#pragma unroll
        for (int r = 1; r < CL; ++r) { v += sm.gin[ig][r][at]; c += sm.gin[ig][r][kOffC + at]; }
        if (s >= tr) v = 0.f;
        out[at] = v;
        big = fmaxf(big, fabsf(v));
        if (k) out[kOffC + at] = c;
      }
      const uint32_t m = warp_max(__float_as_uint(big));
      if (lane == 0) sm.amax[b] = m;
      wait_cluster(&sm.bz[iz], (k / S::kInZ) & 1);
#pragma unroll
      for (int i = 0; i < kZ / 32; ++i) {
        float v = sm.zin[iz][0][lane + 32 * i];
#pragma unroll
        for (int r = 1; r < CL; ++r) v += sm.zin[iz][r][lane + 32 * i];
        sm.zsum[b][lane + 32 * i] = v;
      }
      if (ok && lane == 0 && k + 1 < nblk) {
        mbar_expect_tx(&sm.bg[(k + 1) % S::kInG], CL * kSendG);
        mbar_expect_tx(&sm.bz[(k + 1) % S::kInZ], CL * kZ * 4);
      }
      __syncwarp();
      if (ok && lane == 0) mbar_arrive(&sm.ready[b]);
    }
  } else if (role == kGram) {
    // ================= Gram warps; lane = 4 g + tt =================
    const int g = lane >> 2, tt = lane & 3;
    Split pv[S::kCarry ? KG : 1][4];   // the rows of the block before, split
    for (uint32_t kb = 0; kb < nblk; ++kb) {
      wait(&sm.full[kb % NS], (kb / NS) & 1);
      const float* xr = &sm.rows[kb % NS][g][8 * warp + 2 * tt];
      const float* pr = &sm.rows[(kb + NS - 1) % NS][g][8 * warp + 2 * tt];
      float gh[2][4] = {}, gs[2][4] = {}, hh[2][4] = {}, cx[2][4] = {};
#pragma unroll
      for (int j = 0; j < KG; ++j) {
        const float2 x0 = *reinterpret_cast<const float2*>(xr + 8 * NG * j);
        const float2 x1 = *reinterpret_cast<const float2*>(xr + 8 * S::kPitch + 8 * NG * j);
        const Split a = split_t(x0.x), b = split_t(x0.y), c = split_t(x1.x), d = split_t(x1.y);
        mma::tf32(gh[0], a.hi, c.hi, b.hi, d.hi, a.hi, b.hi);
        mma::tf32(gh[1], a.hi, c.hi, b.hi, d.hi, c.hi, d.hi);
        mma::tf32(gs[0], a.hi, c.hi, b.hi, d.hi, a.lo, b.lo);
        mma::tf32(gs[1], a.hi, c.hi, b.hi, d.hi, c.lo, d.lo);
        if (kb) {
          Split e, f, u, v;
          if (S::kCarry) {
            e = pv[j][0]; f = pv[j][1]; u = pv[j][2]; v = pv[j][3];
          } else {
            const float2 y0 = *reinterpret_cast<const float2*>(pr + 8 * NG * j);
            const float2 y1 = *reinterpret_cast<const float2*>(pr + 8 * S::kPitch + 8 * NG * j);
            e = split_t(y0.x); f = split_t(y0.y); u = split_t(y1.x); v = split_t(y1.y);
          }
          mma::tf32(hh[0], a.hi, c.hi, b.hi, d.hi, e.hi, f.hi);
          mma::tf32(hh[1], a.hi, c.hi, b.hi, d.hi, u.hi, v.hi);
          mma::tf32(cx[0], a.lo, c.lo, b.lo, d.lo, e.hi, f.hi);
          mma::tf32(cx[1], a.lo, c.lo, b.lo, d.lo, u.hi, v.hi);
          mma::tf32(cx[0], a.hi, c.hi, b.hi, d.hi, e.lo, f.lo);
          mma::tf32(cx[1], a.hi, c.hi, b.hi, d.hi, u.lo, v.lo);
        }
        if (S::kCarry) { pv[j][0] = a; pv[j][1] = b; pv[j][2] = c; pv[j][3] = d; }
      }
      // with the split rows in registers a block's slot is done with here, else one block later
      __syncwarp();
      if (ok && lane == 0 && (S::kCarry || kb)) mbar_arrive(&sm.freed[(S::kCarry ? kb : kb - 1) % NS]);
      float* part = sm.gpart[kb & 1][warp];
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
      asm volatile("bar.sync 2, %0;" ::"n"(NG * 32) : "memory");
      // sums over the warps, in warp order, with the factors of the couplings, four entries per thread; sent to every
      // CTA of the cluster
      const int ig = kb % S::kInG;
      const float one = rank == 0 ? scale : 0.f;   // the bias input's part of a coupling
      const int e = warp * 32 + lane;
      const bool own = e < 64;
      const int tr = (e & 63) >> 2, s0 = 4 * (e & 3);
      if (own ? s0 < tr : kb > 0 && e < 128) {
        const int at = (own ? 0 : kOffC) + tr * kGp + s0;
        float v[4] = {};
#pragma unroll
        for (int w = 0; w < NG; ++w) {
          const float4 x = *reinterpret_cast<const float4*>(&sm.gpart[kb & 1][w][at]);
          v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
        }
        if (own) {
#pragma unroll
          for (int w = 0; w < NG; ++w)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] += sm.gpart[kb & 1][w][(s0 + i) * kGp + tr];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float f = scale;
          if (decay) f *= sm.qp[own ? max(tr - 1 - s0 - i, 0) : tr + kB - 1 - s0 - i];
          v[i] = fmaf(v[i], f, one);
          if (own && s0 + i >= tr) v[i] = 0.f;
        }
        const float4 out = make_float4(v[0], v[1], v[2], v[3]);
        const uint32_t to = smem_addr(&sm.gin[ig][rank][at]), bar = smem_addr(&sm.bg[ig]);
#pragma unroll
        for (uint32_t r = 0; r < CL; ++r)
          if (ok) mma::send_peer(mma::peer_addr(to, r), out, mma::peer_addr(bar, r));
      }
    }
  } else if (role == kModel) {
    // ================= model warps; lane = 4 g + tt =================
    const int g = lane >> 2, tt = lane & 3;
    const bool two = g < kC - 8;               // this lane holds a class of the second eight
    const bool biases = warp == 0 && rank == 0;   // the bias is added by one warp of one CTA
    float U[KM][4], ws[KM][4];
    float b0 = 0.f, b1 = 0.f, ub0 = 0.f, ub1 = 0.f;   // start values and update sums of the biases of classes g, g + 8
    asm volatile("griddepcontrol.wait;" ::: "memory");
    {
      auto load = [&](const float* src, float (&v)[KM][4], float& v0, float& v1) {
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
        v0 = biases ? src[kD * kC + g] : 0.f;
        v1 = biases && two ? src[kD * kC + 8 + g] : 0.f;
      };
      load(p.snaps + (size_t)t.snap_slot * p.stride, ws, b0, b1);
#pragma unroll 1
      for (uint32_t f = 0; f < t.inflight_cnt; ++f) {   // own update sums still on their way to the server
        const InflightRef ref = p.inflight[t.inflight_off + f];
        float v0, v1;
        load(p.U + (size_t)ref.row * p.stride, U, v0, v1);
#pragma unroll
        for (int j = 0; j < KM; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) ws[j][c] = fmaf(-ref.eta, U[j][c], ws[j][c]);
        b0 = fmaf(-ref.eta, v0, b0);
        b1 = fmaf(-ref.eta, v1, b1);
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
      const bool update = kb >= 2, look = kb < nblk;
      const uint32_t k = update ? kb - 2 : 0, nv = min((uint32_t)kB, n - k * kB);
      // the rows of block k as the update's second operand ([sample][pixel], pixel g of the warp's k-steps), and those of block kb
      const float* xb = &sm.rows[k % NS][tt][8 * warp + g];
      const float* xr = &sm.rows[kb % NS][g][8 * warp + 2 * tt];
      if (look) wait(&sm.full[kb % NS], (kb / NS) & 1);
      if (update) {
        // ---- U^T = q^nv U^T + sum_s q^(nv-1-s) delta_s x_s; the k index of the product is read as samples t, t + 4, t + 8, t + 12 ----
        wait(&sm.delta[k & 1], (k >> 1) & 1);
        Parts a[2][2];   // [eight samples][classes g, g + 8]
        {
          const float* d0 = &sm.dbuf[k & 1][g / kCh][g % kCh];
          const float* d1 = &sm.dbuf[k & 1][1][two ? g + 3 : 0];   // classes 8, 9
          float s0 = 0.f, s1 = 0.f;
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            float v0[2], v1[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int s = 8 * m + tt + 4 * i;
              v0[i] = d0[s * kCh]; v1[i] = two ? d1[s * kCh] : 0.f;
              if (biases) { s0 += v0[i]; s1 += v1[i]; }
              if (decay) {
                const float f = (uint32_t)s < nv ? sm.qp[nv - 1 - s] : 0.f;
                v0[i] *= f; v1[i] *= f;
              }
            }
            a[m][0] = parts(v0[0], v0[1]);
            a[m][1] = parts(v1[0], v1[1]);
          }
          if (biases) {
            s0 += shx(s0, 1); s1 += shx(s1, 1);
            ub0 += s0 + shx(s0, 2); ub1 += s1 + shx(s1, 2);
          }
        }
        if (decay) {   // U decays with the block, and with it the share of the start model
          const float qn = sm.qp[nv];
#pragma unroll
          for (int j = 0; j < KM; ++j)
#pragma unroll
            for (int c = 0; c < 4; ++c) U[j][c] *= qn;
          const double qd = 1.0 - (double)eta * (double)p.l2;
#pragma unroll 1
          for (uint32_t i = 0; i < nv; ++i) qwd *= qd;
          qw = (float)qwd;
        }
        const uint32_t aa[4] = {a[0][0].a, a[0][1].a, a[1][0].a, a[1][1].a}, ab[4] = {a[0][0].b, a[0][1].b, a[1][0].b, a[1][1].b};
        const uint32_t ac[4] = {a[0][0].c, a[0][1].c, a[1][0].c, a[1][1].c};
        // k-steps side by side, as many as there are registers for: the products of one depend on one another.  (Rows fetched and
        // split before the wait for the deltas: 5 clients on the ring 8.84 instead of 8.19 ms.)
        constexpr int kSide = S::kThreads <= 384 ? KM : 2;
#pragma unroll
        for (int j0 = 0; j0 < KM; j0 += kSide) {
          float d[kSide][4] = {}, e[kSide][4] = {};
          Parts x[kSide][2];
#pragma unroll
          for (int jj = 0; jj < kSide; ++jj)
#pragma unroll
            for (int m = 0; m < 2; ++m)
              if (j0 + jj < KM) {
                const float* at = xb + 8 * m * S::kPitch + 8 * NM * (j0 + jj);
                x[jj][m] = parts_t(at[0], at[4 * S::kPitch]);
              }
#pragma unroll
          for (int term = 0; term < 6; ++term)
#pragma unroll
            for (int jj = 0; jj < kSide; ++jj) {
              if (j0 + jj >= KM) continue;
              const Parts &x0 = x[jj][0], &x1 = x[jj][1];
              if (term == 0) mma::mma_bf16(e[jj], ac, x0.a, x1.a);
              if (term == 1) mma::mma_bf16(d[jj], aa, x0.a, x1.a);
              if (term == 2) mma::mma_bf16(e[jj], aa, x0.c, x1.c);
              if (term == 3) mma::mma_bf16(e[jj], ab, x0.b, x1.b);
              if (term == 4) mma::mma_bf16(e[jj], ab, x0.a, x1.a);
              if (term == 5) mma::mma_bf16(e[jj], aa, x0.b, x1.b);
            }
#pragma unroll
          for (int jj = 0; jj < kSide; ++jj)
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (j0 + jj < KM) U[j0 + jj][c] += d[jj][c] + e[jj][c];
        }
      }
      if (look) {
        // ---- logits of block kb with the model W = qw W_start - eta U ----
        float zm[2][4] = {}, zx[2][4] = {};
#pragma unroll
        for (int j = 0; j < KM; ++j) {
          const float2 x0 = *reinterpret_cast<const float2*>(xr + 8 * NM * j), x1 = *reinterpret_cast<const float2*>(xr + 8 * S::kPitch + 8 * NM * j);
          const Split a = split_r(x0.x), b = split_r(x0.y), c = split_r(x1.x), d = split_r(x1.y);
          const Split w0 = split_r(fmaf(neta, U[j][0], qw * ws[j][0])), w2 = split_r(fmaf(neta, U[j][1], qw * ws[j][1]));
          const Split w1 = split_r(fmaf(neta, U[j][2], qw * ws[j][2])), w3 = split_r(fmaf(neta, U[j][3], qw * ws[j][3]));
          mma::tf32(zm[0], w0.hi, w1.hi, w2.hi, w3.hi, a.hi, b.hi);
          mma::tf32(zm[1], w0.hi, w1.hi, w2.hi, w3.hi, c.hi, d.hi);
          mma::tf32(zx[0], w0.lo, w1.lo, w2.lo, w3.lo, a.hi, b.hi);
          mma::tf32(zx[1], w0.lo, w1.lo, w2.lo, w3.lo, c.hi, d.hi);
          mma::tf32(zx[0], w0.hi, w1.hi, w2.hi, w3.hi, a.lo, b.lo);
          mma::tf32(zx[1], w0.hi, w1.hi, w2.hi, w3.hi, c.lo, d.lo);
        }
        float* part = sm.zpart[kb & 1][warp];
        const float c0 = kLog2e * fmaf(neta, ub0, b0), c1 = kLog2e * fmaf(neta, ub1, b1);
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int s = 8 * m + 2 * tt;
          float f0 = kLog2e, f1 = kLog2e;
          if (decay) { f0 *= sm.qp[s + (kb ? kB : 0)]; f1 *= sm.qp[s + 1 + (kb ? kB : 0)]; }
          *reinterpret_cast<float2*>(part + g * kB + s) = make_float2(fmaf(zm[m][0] + zx[m][0], f0, c0), fmaf(zm[m][1] + zx[m][1], f1, c0));
          if (two)
            *reinterpret_cast<float2*>(part + (8 + g) * kB + s) = make_float2(fmaf(zm[m][2] + zx[m][2], f0, c1), fmaf(zm[m][3] + zx[m][3], f1, c1));
        }
        asm volatile("bar.sync 1, %0;" ::"n"(NM * 32) : "memory");
        // sums over the warps, in warp order; sent to every CTA of the cluster
        if (warp < 2) {
          const int iz = kb % S::kInZ, e = warp * 32 + lane;
          if (e < kQuadZ) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < NM; ++w) {
              const float4 x = *reinterpret_cast<const float4*>(&sm.zpart[kb & 1][w][4 * e]);
              v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
            }
            const uint32_t to = smem_addr(&sm.zin[iz][rank][4 * e]), bar = smem_addr(&sm.bz[iz]);
#pragma unroll
            for (uint32_t r = 0; r < CL; ++r)
              if (ok) mma::send_peer(mma::peer_addr(to, r), v, mma::peer_addr(bar, r));
          }
        }
      }
      if (update) {
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(&sm.freed[k % NS]);
      }
    }

    // ---- event trigger: h reached s_{i,c}; publish U_i (and the end model) ----
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    {
      // a round whose copies never came leaves NaN behind, for callers that have no status word to look at
      const float bad = ok ? 0.f : __int_as_float(0x7FFFFFFF);
      const float c1 = (decay ? (float)((1.0 - qwd) / (double)eta) : 0.f) + bad;
      qw += bad;
#pragma unroll 1
      for (int pass = 0; pass < (p.w_end ? 2 : 1); ++pass) {
        float* row = (pass == 0 ? p.U : p.w_end) + (size_t)t.u_row * p.stride;
        const float fw = pass == 0 ? c1 : qw, fu = pass == 0 ? 1.f : neta;
        __syncwarp();   // the second pass starts with the buffer the first one ended with, where KM is odd
#pragma unroll
        for (int j = 0; j < KM; ++j) {   // a k-step's 80 parameters through the warp's own buffer: whole lines out
          float* st = sm.zpart[j & 1][warp];
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
        if (biases) {
          if (tt == 0) row[kD * kC + g] = fmaf(fu, ub0, pass == 0 ? 0.f : b0);
          if (tt == 0 && two) row[kD * kC + 8 + g] = fmaf(fu, ub1, pass == 0 ? 0.f : b1);
          if (p.stride && lane < kStageFloats - kParams) row[kParams + lane] = 0.f;   // the row's padding
        }
      }
    }
  }
  if (!ok && p.status && lane == 0) atomicOr(p.status, 1u);
  mma::cluster_sync();   // no CTA leaves while a peer may still send to it
  if (!ok) linger();
  if (!ok && role == kProd)   // copies still in flight target this CTA's shared memory: a bounded chance to land
    for (int s = 0; s < NS; ++s) {
      mbar_wait_limit(&sm.full[s], 0, 1u << 16);
      mbar_wait_limit(&sm.full[s], 1, 1u << 16);
    }
  if (threadIdx.x == 0 && rank == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = n; rec.flags = 1;
    p.trig[t.seq] = rec;
  }
}

typedef Shape<2, 7, 7, 6, 9, 4, false> Two;
typedef Shape<4, 5, 5, 4, 7, 4, true> Four;

template <class S>
cudaError_t launch(const RoundLaunch& p, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.n_tasks * S::kCl, 1, 1);
  cfg.blockDim = dim3(S::kThreads, 1, 1);
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
  return cudaLaunchKernelEx(&cfg, lr_chain_kernel<S>, p);
}

}  // namespace

cudaError_t launch_lr_chain_rounds(const RoundLaunch& p, uint32_t cluster, cudaStream_t s) {
  static bool opted_in[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < 64;
  if (!known || !opted_in[dev]) {
    e = cudaFuncSetAttribute(lr_chain_kernel<Two>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Two::Smem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(lr_chain_kernel<Four>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Four::Smem));
    if (e != cudaSuccess) return e;
    if (known) opted_in[dev] = true;
  }
  return cluster == 4 ? launch<Four>(p, s) : launch<Two>(p, s);
}

}  // namespace aet
