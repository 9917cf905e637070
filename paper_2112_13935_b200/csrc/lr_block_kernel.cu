// Local-SGD round of one client for softmax regression 784 -> 10, batch 1, for launches that fill the SMs: one CTA per
// round-task.
//
// Algorithm 3, MainComputeNode, inner loop (g = grad f(w_c, xi) + lambda W; w_c -= eta g; U_i += g; h++) eight steps at
// a time.  With q = 1 - eta lambda, W, b the model at the start of a block and delta_s = softmax(z_s) - onehot(y_s), its
// step t sees
//     z_t = q^t W x_t + b + sum_{s<t} L[t][s] delta_s,      L[t][s] = -eta (q^(t-1-s) x_s.x_t + 1).
// MMA warps, each with its k-steps of 8 inputs (98 in all), per block:
//   Z^T = W^T X^T, partial sums to shared memory;            R warp: z, then sweeps z <- z0 + L delta(z) over the eight
//   the next block's Gram matrix, under R;                   samples at once until they no longer move; delta out;
//   U^T = q^8 U^T + sum_s q^(7-s) delta_s x_s^T.             biases; row copies two blocks ahead.
// Products are m16n8k8 tf32 with split operands (mma_common.cuh).  What the update loses stays in U: with one CTA per SM, or with lambda, it
// takes operands in three bf16 parts instead, two pairs of parts per instruction (a round of 50 samples 1.5e-7 -> 0.6e-7 off
// fp64, fp32 FMAs 0.7e-7); crowded without lambda both tf32 heads are rounded (0.9e-7; the kernel before 1.1e-7 to 20e-7 by the length
// of the round; three bf16 parts 0.6e-7, but 1.19 instead of 1.08 ms for 1,024 clients).  With the ten classes on the M side eight samples
// fill an n-tile of the logits and a k-step of the update exactly, and the accumulator fragment of U^T is the operand
// fragment of the next logits product when the k index of a step is read as pixel (2t | 2t + 1): U never leaves
// registers, W = q^n W_start - eta U is formed in place, W_start waits in shared memory in fragment order.  A block's
// contribution starts from zero and is added to U by fp32 adds: the tensor cores' rounding never accumulates over a round.
// With lambda, U holds D = sum_s q^(n-1-s) delta_s x_s and the update sum is D + W_start (1 - q^n) / eta.
//
// The sweeps: L is strictly lower triangular and softmax 1/2-Lipschitz in the maximum norm, so a sweep that moves z by at
// most d leaves it within (1 + a)^7 (r / 2) d of the solution, a = max |L| / 2, r = max_t sum_s |L[t][s]|; seven sweeps are
// always enough.
//
// What bounds it: latency.  Crowded launches run two CTAs per SM (7 MMA warps of 14 k-steps and R, 128 registers), one's R under
// the other's products, and rounds of one to ten blocks: start model, first rows and trigger are a third to a half of a launch; the
// tensor pipe is active 20 to 23 % of it, issue slots 30 %, DRAM at 33 % of the copy rate.  With one CTA per SM (14 MMA warps of 7
// k-steps) it is the chain products -> R -> products.  Measured: ten rounds of 1,024 clients, aggregation included, 1.58 -> 1.09
// ms (before: U in tensor memory, operands of the 128-row tcgen05 products staged and split through shared memory for ten rows that matter).
#include <cuda_runtime.h>

#include "aet_kernels.h"
#include "aet_rng.h"
#include "lr_common.cuh"
#include "mma_common.cuh"

namespace aet {
namespace {

using namespace lr;
using mma::Parts;
using mma::parts_t;
using mma::Split;
using mma::split;
using mma::split_r;
using mma::split_t;

constexpr int kBk = 8;                       // samples per block
constexpr int kSteps8 = kD / 8;              // 98 k-steps of 8 inputs
constexpr int kRing = 3;                     // blocks of rows in shared memory
constexpr int kPitch = kD + 8;               // 24 mod 32 floats: fragment loads hit different banks
constexpr float kTol = 2e-7f * kLog2e;       // logits are kept in units of log2

template <int NW, int KS, bool DECAY>
struct Shape {
  static constexpr int kNw = NW, kKs = KS;
  static constexpr bool kDecay = DECAY;
  static constexpr int kThreads = (NW + 1) * 32;
  static constexpr int kCtas = NW <= 7 ? 2 : 1;
  static constexpr bool kParts = kCtas == 1 || DECAY;   // the update's operands in three bf16 parts; otherwise in two tf32 parts
  static_assert(NW * KS == kSteps8, "every warp has the same number of k-steps");
  struct __align__(128) Smem {
    float rows[kRing][kBk][kPitch];
    float2 ws01[kSteps8][32];       // start model in fragment order: class g, pixels 2t and 2t + 1 of a k-step
    float2 ws23[2][kSteps8][4];     // ... classes 8 and 9
    float zpart[NW][16 * kBk];      // per warp: rows 0-9 logits [class][sample], rows 10-15 x_(row - 10) . x_sample
    float pair[NW];                 // per warp: x_6 . x_7
    float4 zsum[32];                // the same summed over the warps
    float4 dfrag[2][32];            // delta as first operand of the update, in fragment order: heads and remainders, or (kParts) as it is
    float dbuf[kBk][16];            // deltas between sweeps: [sample][4 q + i] = class q + 4 i
    float qp[16];                   // powers of q
    int ys[4][kBk];
    uint64_t full[kRing];
  };
  static_assert(sizeof(Smem) <= (size_t)(233472 / kCtas - 1024), "CTAs per SM");
};

template <class S>
__global__ void __launch_bounds__(S::kThreads, S::kCtas) lr_block_kernel(RoundLaunch p) {
  constexpr int NW = S::kNw, KS = S::kKs;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  typename S::Smem& sm = *reinterpret_cast<typename S::Smem*>(smem_raw);

  const TaskDesc t = p.tasks[p.task_begin + blockIdx.x];
  if (!debug_task_ok(p, t)) return;
  if (t.n_samples == 0) {   // this grid may run under the tail of the aggregation before it: wait before writing
    asm volatile("griddepcontrol.wait;" ::: "memory");
    publish_empty_round(p, t, kParams);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t n = t.n_samples, nblk = (n + kBk - 1) / kBk;
  const float eta = t.eta, neta = -t.eta;
  constexpr bool decay = S::kDecay;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRing; ++s) mbar_init(&sm.full[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    double q = 1.0 - (double)eta * (double)p.l2, v = 1.0;
    for (int i = 0; i < 16; ++i) { sm.qp[i] = (float)v; v *= q; }
  }
  if (threadIdx.x < 64) sm.dfrag[threadIdx.x >> 5][threadIdx.x & 31] = make_float4(0.f, 0.f, 0.f, 0.f);   // rows 10-15 stay zero
  __syncthreads();

  // After a wait has given up nothing waits any more: the round runs through on whatever is there and the status word
  // is set.
  bool ok = true;
  auto wait = [&](uint64_t* bar, uint32_t parity) { if (ok) ok = mbar_wait(bar, parity); };

  if (warp == NW) {
    // ================= R: recurrence, biases, row copies; lane = (sample, class group) =================
    const ClientData cd = p.clients[t.client];
    const uint64_t key = p.sample_keys[t.client];
    const float* xrows = reinterpret_cast<const float*>(cd.x);
    auto produce = [&](uint32_t kb) {
      const int sb = kb % kRing;
      // (long since here, if ever: the products of block kb - kRing are done; a barrier short of its bytes is not armed again)
      if (kb >= (uint32_t)kRing && !mbar_try_wait(&sm.full[sb], (kb / kRing - 1) & 1)) ok = false;
      if (!__all_sync(0xffffffffu, ok)) return;
      const uint32_t nvb = min((uint32_t)kBk, n - kb * kBk);
      for (uint32_t r = nvb; r < (uint32_t)kBk; ++r)   // short last block: rows that add nothing anywhere
        for (int i = lane; i < kD / 4; i += 32) reinterpret_cast<float4*>(sm.rows[sb][r])[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (lane == 0) mbar_expect_only(&sm.full[sb], nvb * kRowBytes);
      __syncwarp();
      if ((uint32_t)lane < nvb) {
        const uint32_t idx = sample_index(draw(key, t.sample_ctr0 + (uint64_t)kb * kBk + lane), cd.n);
        bulk_load_row(sm.rows[sb][lane], xrows + (size_t)idx * kD, &sm.full[sb]);
        sm.ys[kb & 3][lane] = __ldg(cd.y + idx);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.full[sb]);
    };
    produce(0);
    if (nblk > 1) produce(1);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const float scale = neta * kLog2e;
    constexpr int kOwn = 3;            // classes q, q + 4 and (q < 2) q + 8 of sample j
    const int j = lane >> 2, q = lane & 3;
    float b0[kOwn] = {}, ub[kOwn] = {};
    {
      const float* src = p.snaps + (size_t)t.snap_slot * p.stride + kD * kC;
#pragma unroll
      for (int i = 0; i < kOwn; ++i) b0[i] = q + 4 * i < kC ? src[q + 4 * i] : 0.f;
      for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
        const InflightRef ref = p.inflight[t.inflight_off + f];
        const float* us = p.U + (size_t)ref.row * p.stride + kD * kC;
#pragma unroll
        for (int i = 0; i < kOwn; ++i) b0[i] = fmaf(-ref.eta, q + 4 * i < kC ? us[q + 4 * i] : 0.f, b0[i]);
      }
    }
    for (uint32_t k = 0; k < nblk; ++k) {
      const uint32_t nv = min((uint32_t)kBk, n - k * kBk);
      const bool live = (uint32_t)j < nv;
      asm volatile("bar.sync 2, %0;" ::"n"((NW + 1) * 32) : "memory");   // logits and couplings of the block are in
      {
        float4 v = reinterpret_cast<const float4*>(sm.zpart[0])[lane];
#pragma unroll
        for (int w = 1; w < NW; ++w) {
          const float4 x = reinterpret_cast<const float4*>(sm.zpart[w])[lane];
          v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
        }
        sm.zsum[lane] = v;
        __syncwarp();
      }
      const float* zs = reinterpret_cast<const float*>(sm.zsum);
      float z0[kOwn], L[kBk - 1];
#pragma unroll
      for (int i = 0; i < kOwn; ++i) {
        const int c = q + 4 * i;
        float v = zs[(c < kC ? c : 0) * kBk + j];
        if (decay) v *= sm.qp[j];
        z0[i] = c < kC ? (v + fmaf(neta, ub[i], b0[i])) * kLog2e : -1e30f;   // no such class: contributes nothing
      }
      float amax = 0.f;   // largest coupling, in units of log2 as the logits are
#pragma unroll
      for (int s = 0; s < kBk - 1; ++s) {
        float v = 0.f;
        if (s < kBk - 2) {
          v = zs[(kC + s) * kBk + j];
        } else {
#pragma unroll
          for (int w = 0; w < NW; ++w) v += sm.pair[w];
        }
        v = fmaf(v, decay ? scale * sm.qp[max(j - 1 - s, 0)] : scale, scale);   // + 1: the bias input
        L[s] = s < j ? v : 0.f;
        if (live) amax = fmaxf(amax, fabsf(L[s]));
      }
      amax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(amax)));
      const float gain = 3.5f / kLog2e * amax * ex2(fminf(3.5f * amax, 60.f));   // (1 + a)^7 <= exp(7 a)
      const bool wild = amax > 8.f;   // the shift of the softmax must follow the corrections
      const int y = sm.ys[k & 3][j];
      float oh[kOwn];
#pragma unroll
      for (int i = 0; i < kOwn; ++i) oh[i] = q + 4 * i == y ? -1.f : 0.f;
      auto top = [&](const float (&z)[kOwn]) {
        float m = fmaxf(fmaxf(z[0], z[1]), z[2]);
        m = fmaxf(m, shx(m, 1));
        return fmaxf(m, shx(m, 2));
      };
      {
        const float m = top(z0);
#pragma unroll
        for (int i = 0; i < kOwn; ++i) z0[i] -= m;
      }
      float z[kOwn], d[kOwn];
#pragma unroll
      for (int i = 0; i < kOwn; ++i) z[i] = z0[i];
      uint32_t left = nv - 1;   // sweeps that can still be needed
      while (true) {
        float m = 0.f;
        if (wild) m = top(z);
        float e[kOwn];
#pragma unroll
        for (int i = 0; i < kOwn; ++i) e[i] = ex2(z[i] - m);
        float sum = (e[0] + e[1]) + e[2];
        sum += shx(sum, 1);
        sum += shx(sum, 2);
        const float inv = rcp(sum);
#pragma unroll
        for (int i = 0; i < kOwn; ++i) d[i] = fmaf(e[i], inv, oh[i]);
        if (!left) break;
        --left;
        *reinterpret_cast<float4*>(&sm.dbuf[j][4 * q]) = make_float4(d[0], d[1], d[2], 0.f);
        __syncwarp();
        float zn[kOwn];
#pragma unroll
        for (int i = 0; i < kOwn; ++i) zn[i] = z0[i];
#pragma unroll
        for (int s = 0; s < kBk - 1; ++s) {
          const float4 dv = *reinterpret_cast<const float4*>(&sm.dbuf[s][4 * q]);
          zn[0] = fmaf(L[s], dv.x, zn[0]); zn[1] = fmaf(L[s], dv.y, zn[1]); zn[2] = fmaf(L[s], dv.z, zn[2]);
        }
        float change = 0.f;
#pragma unroll
        for (int i = 0; i < kOwn; ++i) { change = fmaxf(change, fabsf(zn[i] - z[i])); z[i] = zn[i]; }
        if (!__any_sync(0xffffffffu, live && !(change * gain <= kTol)) && !p.step_by_step) left = 0;
        __syncwarp();
      }
      // delta as the update's first operand: (row class, column sample); lane 4 g + tt of a fragment holds rows g, g + 8,
      // and columns tt and tt + 4 (as its pair)
      float sum[kOwn];
#pragma unroll
      for (int i = 0; i < kOwn; ++i) {
        const int c = q + 4 * i;
        sum[i] = live && c < kC ? d[i] : 0.f;
        if (c < kC) {
          const float v = decay && live ? sum[i] * sm.qp[nv - 1 - j] : sum[i];
          const int at = 4 * (c & 7) + (j & 3), comp = (c >> 3) + 2 * (j >> 2);
          if (S::kParts) {
            reinterpret_cast<float*>(&sm.dfrag[0][at])[comp] = v;
          } else {
            const Split sp = split(v);
            reinterpret_cast<uint32_t*>(&sm.dfrag[0][at])[comp] = sp.hi;
            reinterpret_cast<uint32_t*>(&sm.dfrag[1][at])[comp] = sp.lo;
          }
        }
      }
      __syncwarp();
      asm volatile("bar.arrive 3, %0;" ::"n"((NW + 1) * 32) : "memory");
#pragma unroll
      for (int i = 0; i < kOwn; ++i) {
        sum[i] += shx(sum[i], 4);
        sum[i] += shx(sum[i], 8);
        ub[i] += sum[i] + shx(sum[i], 16);
      }
      if (k + 2 < nblk && ok) produce(k + 2);   // block k - 1 left its slot before this block's logits came in
    }
    if (ok && lane < 4) {
      float* U = p.U + (size_t)t.u_row * p.stride + kD * kC;
#pragma unroll
      for (int i = 0; i < kOwn; ++i)
        if (q + 4 * i < kC) {
          U[q + 4 * i] = ub[i];
          if (p.w_end) p.w_end[(size_t)t.u_row * p.stride + kD * kC + q + 4 * i] = fmaf(neta, ub[i], b0[i]);
        }
    }
    if (ok && lane < kStageFloats - kParams) p.U[(size_t)t.u_row * p.stride + kParams + lane] = 0.f;   // the row's padding
  } else {
    // ================= MMA warps; lane = 4 g + tt =================
    const int g = lane >> 2, tt = lane & 3;
    const bool two = g < kC - 8;   // this lane holds a class of the second eight
    const int k0 = warp * KS;
    float U[KS][4];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    {
      auto load = [&](const float* src, float (&v)[KS][4]) {
        const float* at = src + (8 * k0 + 2 * tt) * kC + g;
#pragma unroll
        for (int j = 0; j < KS; ++j) {
          v[j][0] = at[80 * j];
          v[j][1] = at[80 * j + kC];
          v[j][2] = two ? at[80 * j + 8] : 0.f;
          v[j][3] = two ? at[80 * j + kC + 8] : 0.f;
        }
      };
      load(p.snaps + (size_t)t.snap_slot * p.stride, U);
#pragma unroll 1
      for (uint32_t f = 0; f < t.inflight_cnt; ++f) {   // own update sums still on their way to the server
        const InflightRef ref = p.inflight[t.inflight_off + f];
        float v[KS][4];
        load(p.U + (size_t)ref.row * p.stride, v);
#pragma unroll
        for (int j = 0; j < KS; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) U[j][c] = fmaf(-ref.eta, v[j][c], U[j][c]);
      }
#pragma unroll
      for (int j = 0; j < KS; ++j) {
        sm.ws01[k0 + j][lane] = make_float2(U[j][0], U[j][1]);
        if (two) sm.ws23[g][k0 + j][tt] = make_float2(U[j][2], U[j][3]);
#pragma unroll
        for (int c = 0; c < 4; ++c) U[j][c] = 0.f;
      }
    }
    // only this warp reads what it wrote
    const float2* w01 = &sm.ws01[k0][lane];
    float qw = 1.f;      // q^(samples in U): W = qw W_start - eta U
    double qwd = 1.0;

    for (uint32_t k = 0; k < nblk; ++k) {
      const uint32_t nv = min((uint32_t)kBk, n - k * kBk);
      wait(&sm.full[k % kRing], (k / kRing) & 1);
      {
        // ---- Z^T = W^T X^T; rows 10-15 of the first operand, which no class needs, are the block's rows 0-5: their
        // products with all eight rows are the Gram matrix but for x_6 . x_7.  (U is zero there: W = the row.) ----
        const float* xr = &sm.rows[k % kRing][g][8 * k0 + 2 * tt];
        const float* second = two ? reinterpret_cast<const float*>(&sm.ws23[g][k0][tt]) : &sm.rows[k % kRing][g - 2][8 * k0 + 2 * tt];
        const float qs = two ? qw : 1.f;
        auto sp = [](float v) { return S::kCtas == 1 ? split_r(v) : split_t(v); };   // (5 samples 4.8e-8 -> 4.1e-8 off fp64)
        float zm[4] = {}, zx[4] = {};
#pragma unroll
        for (int j = 0; j < KS; ++j) {
          const float2 x = *reinterpret_cast<const float2*>(xr + 8 * j);
          const float2 wa = w01[32 * j];
          const float2 wb = *reinterpret_cast<const float2*>(second + 8 * j);
          const Split a = sp(x.x), b = sp(x.y);
          const Split v0 = sp(fmaf(neta, U[j][0], decay ? qw * wa.x : wa.x)), v2 = sp(fmaf(neta, U[j][1], decay ? qw * wa.y : wa.y));
          const Split v1 = sp(fmaf(neta, U[j][2], decay ? qs * wb.x : wb.x)), v3 = sp(fmaf(neta, U[j][3], decay ? qs * wb.y : wb.y));
          mma::tf32(zm, v0.hi, v1.hi, v2.hi, v3.hi, a.hi, b.hi);
          mma::tf32(zx, v0.lo, v1.lo, v2.lo, v3.lo, a.hi, b.hi);
          mma::tf32(zx, v0.hi, v1.hi, v2.hi, v3.hi, a.lo, b.lo);
        }
        float* part = sm.zpart[warp];
        *reinterpret_cast<float2*>(part + g * kBk + 2 * tt) = make_float2(zm[0] + zx[0], zm[1] + zx[1]);
        *reinterpret_cast<float2*>(part + (8 + g) * kBk + 2 * tt) = make_float2(zm[2] + zx[2], zm[3] + zx[3]);
        if (nv == kBk) {   // x_6 . x_7 over this warp's inputs
          const float* r6 = &sm.rows[k % kRing][kBk - 2][8 * k0];
          float v = 0.f;
#pragma unroll
          for (int i = 0; i < (8 * KS + 31) / 32; ++i) {
            const int c = lane + 32 * i;
            if (c < 8 * KS) v = fmaf(r6[c], r6[kPitch + c], v);
          }
#pragma unroll
          for (int m = 16; m; m >>= 1) v += shx(v, m);
          if (lane == 0) sm.pair[warp] = v;
        }
      }
      asm volatile("bar.arrive 2, %0;" ::"n"((NW + 1) * 32) : "memory");
      // the block's inputs as the second operand: [sample][pixel], pixel g of the warp's k-steps
      const float* xb = &sm.rows[k % kRing][tt][8 * k0 + g];
      if (decay) {   // U decays with the block, and with it the share of the start model
        const float qn = sm.qp[nv];
#pragma unroll
        for (int j = 0; j < KS; ++j)
#pragma unroll
          for (int c = 0; c < 4; ++c) U[j][c] *= qn;
        const double qd = 1.0 - (double)eta * (double)p.l2;
#pragma unroll 1
        for (uint32_t i = 0; i < nv; ++i) qwd *= qd;
        qw = (float)qwd;
      }
      asm volatile("bar.sync 3, %0;" ::"n"((NW + 1) * 32) : "memory");
      {
        // ---- U^T += sum_s q^(nv-1-s) delta_s x_s^T ----
        if (S::kParts) {
          const float4 dv = sm.dfrag[0][lane];
          const Parts p0 = mma::parts(dv.x, dv.z), p1 = mma::parts(dv.y, dv.w);   // classes g, g + 8
          const uint32_t ba[4] = {p0.b, p1.b, p0.a, p1.a};
#pragma unroll
          for (int j = 0; j < KS; ++j) {
            const Parts x = parts_t(xb[8 * j], xb[4 * kPitch + 8 * j]);
            // k index of 16: the eight samples with one pair of parts, then with another; the leading parts by themselves (beside
            // the small ones their sum would be cut further up)
            float d[4] = {}, e[4] = {};
            mma::mma_bf16_k8(e, p0.c, p1.c, x.a);
            mma::mma_bf16_k8(d, p0.a, p1.a, x.a);
            mma::mma_bf16(e, ba, x.b, x.c);
            mma::mma_bf16(e, ba, x.a, x.b);
#pragma unroll
            for (int c = 0; c < 4; ++c) U[j][c] += d[c] + e[c];
          }
        } else {
          float4 h4 = sm.dfrag[0][lane], l4 = sm.dfrag[1][lane];
          const uint32_t h0 = __float_as_uint(h4.x), h1 = __float_as_uint(h4.y), h2 = __float_as_uint(h4.z), h3 = __float_as_uint(h4.w);
          const uint32_t l0 = __float_as_uint(l4.x), l1 = __float_as_uint(l4.y), l2 = __float_as_uint(l4.z), l3 = __float_as_uint(l4.w);
#pragma unroll
          for (int j = 0; j < KS; ++j) {
            const Split v0 = split_r(xb[8 * j]), v1 = split_r(xb[4 * kPitch + 8 * j]);
            float d[4] = {};
            mma::tf32(d, l0, l1, l2, l3, v0.hi, v1.hi);
            mma::tf32(d, h0, h1, h2, h3, v0.lo, v1.lo);
            mma::tf32(d, h0, h1, h2, h3, v0.hi, v1.hi);
#pragma unroll
            for (int c = 0; c < 4; ++c) U[j][c] += d[c];
          }
        }
      }
    }

    // ---- event trigger: h reached s_{i,c}; publish U_i (and the end model) ----
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (ok) {
      const float c1 = decay ? (float)((1.0 - qwd) / (double)eta) : 0.f;
#pragma unroll 1
      for (int pass = 0; pass < (p.w_end ? 2 : 1); ++pass) {
        float* row = (pass == 0 ? p.U : p.w_end) + (size_t)t.u_row * p.stride + 80 * k0;
        const float fw = pass == 0 ? c1 : qw, fu = pass == 0 ? 1.f : neta;
#pragma unroll
        for (int j = 0; j < KS; ++j) {   // a k-step's 80 parameters through the warp's own buffer: whole lines out
          float* st = sm.zpart[warp];
          const int at = 2 * tt * kC + g;
          const float2 wa = w01[32 * j], wb = sm.ws23[g & 1][k0 + j][tt];
          st[at] = fmaf(fu, U[j][0], fw * wa.x);
          st[at + kC] = fmaf(fu, U[j][1], fw * wa.y);
          if (two) {
            st[at + 8] = fmaf(fu, U[j][2], fw * wb.x);
            st[at + kC + 8] = fmaf(fu, U[j][3], fw * wb.y);
          }
          __syncwarp();
          if (lane < 20) *reinterpret_cast<float4*>(row + 80 * j + 4 * lane) = *reinterpret_cast<const float4*>(st + 4 * lane);
          __syncwarp();
        }
      }
    }
  }
  if (!ok && p.status && lane == 0) atomicOr(p.status, 1u);
  if (!ok && warp == NW)   // copies still in flight target this CTA's shared memory: a bounded chance to land
    for (int s = 0; s < kRing; ++s) {
      mbar_wait_limit(&sm.full[s], 0, 1u << 16);
      mbar_wait_limit(&sm.full[s], 1, 1u << 16);
    }
  if (threadIdx.x == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = n; rec.flags = 1;
    p.trig[t.seq] = rec;
  }
}

template <class S>
cudaError_t launch(const RoundLaunch& p, cudaStream_t s) {
  static bool opted_in[64] = {};   // more than 48 KB of shared memory has to be asked for once per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool known = dev >= 0 && dev < 64;
  if (!known || !opted_in[dev]) {
    e = cudaFuncSetAttribute(lr_block_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(typename S::Smem));
    if (e != cudaSuccess) return e;
    if (known) opted_in[dev] = true;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.n_tasks, 1, 1);
  cfg.blockDim = dim3(S::kThreads, 1, 1);
  cfg.dynamicSmemBytes = sizeof(typename S::Smem);
  cfg.stream = s;
  // the grid may start under the tail of the aggregation kernel ahead of it and waits before reading its output
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lr_block_kernel<S>, p);
}

}  // namespace

cudaError_t launch_lr_block_rounds(const RoundLaunch& p, bool crowded, cudaStream_t s) {
  if (crowded) return p.l2 != 0.f ? launch<Shape<7, 14, true>>(p, s) : launch<Shape<7, 14, false>>(p, s);
  return p.l2 != 0.f ? launch<Shape<14, 7, true>>(p, s) : launch<Shape<14, 7, false>>(p, s);
}

}  // namespace aet
