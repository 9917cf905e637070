// Local-SGD round of one client for the LeNet-shaped classifier 28x28x1 -> conv 6 -> conv 16 -> 120 -> 84 -> 10 on a
// cluster of 8 or 4 CTAs of 16 warps: convolutions split by samples, the widest dense layer split by its outputs.
//
// Algorithm 3, MainComputeNode, inner loop with xi a minibatch: g = mean gradient (+ lambda W on weights), w_c -= eta_i g,
// U_i += g, repeated s_{i,c} / B times; then (c, U_i, i) is sent.
//
// Splitting the whole model by samples (cnn_kernel.cu) moves 44,426 gradients out of every CTA and as many weights into
// it per iteration, through L2.  Here only what is small moves, by st.async into the peers' shared memory, each hand-over
// counted by an mbarrier at the receiver:
//   pooled maps q2 (256 per sample) to everybody;  every CTA has 120 / CL outputs of the first dense layer, for all samples;
//   its h1 to everybody;                            layers 2, 3 and the softmax run in every CTA alike (same order: same bits);
//   its part of dq2 to the samples' CTAs;           which go on through the convolutions;
//   the convolutions' gradients (2,566) to the CTAs that own a slice of them, and the new weights back to everybody.
// Nothing is reused before its readers are done because each step needs the one before from all CTAs.  All weights stay in
// shared memory, all update sums in the registers of the threads that own the parameters, for the whole round.
//
// Products are bf16 on operands in three parts (mma_common.cuh; rms error of a round 0.5e-7 to 1.1e-7 as with fp32 FMAs, 1.1e-7 to
// 1.5e-7 with two tf32 parts), convolutions as implicit GEMMs:
//   conv 2      Z[16 x 64] = W2[16 x 150] im2col(q1)           M = output planes exactly; the bias is tap 150 with input 1
//   its dW      dW2[16 x 150] = dz2[16 x 64] im2col(q1)^T      accumulators stay in registers over the samples
//   its dIn     col[150 x 64] = W2^T dz2, then every output gathers its up to 25 entries of col
//   conv 1      FMAs (6 planes would fill 6 of 16 rows);  its dW[26 x 6] = im2col(x)^T dz1, dz1 formed from dq1 and sign bits
// What bounds it: the chain of some fifteen short phases and five hand-overs per iteration, not any one unit (about 55 K
// cycles).  Measured: 16 clients, minibatch 16, 12 rounds, 18.9 -> 7.5 ms against the split by samples.
#include <cuda_runtime.h>

#include "aet_kernels.h"
#include "aet_rng.h"
#include "lr_common.cuh"
#include "mma_common.cuh"

namespace aet {
namespace {

using lr::kWaitLimit;
using lr::mbar_expect_tx;
using lr::mbar_init;
using lr::smem_addr;
using mma::Parts;
using mma::parts;
using mma::parts_t;

constexpr int kWarps = 16, kThreads = kWarps * 32;
constexpr int kS = 28, kC1 = 6, kP1 = 12, kC2 = 16, kFlat = 256, kF1 = 120, kF2 = 84, kN = 10;
constexpr int kX = kS * kS, kQ1 = kC1 * kP1 * kP1;      // values of a row, of the first pooled maps
constexpr int kPw2 = 152, kW2c = kC2 * kPw2, kW1c = 256;   // conv 2: [plane][tap, bias, 0]; conv 1: [tap, bias][8 planes, 6 used]
constexpr int kQuads = (kW2c + kW1c) / 4;               // the convolutions' parameters as 16-byte pieces
constexpr int kPq2 = 264, kPh1 = 120, kPh2 = 88, kPdz = 72, kPcol = 72;   // row pitches: fragment loads hit different banks
constexpr int kMaxPer = 4;                              // samples per CTA
// offsets in the parameter vector
constexpr int kOW1 = 0, kOb1 = 150, kOW2 = 156, kOb2 = 2556, kOF1 = 2572, kObF1 = kOF1 + kFlat * kF1, kOF2 = kObF1 + kF1,
              kObF2 = kOF2 + kF1 * kF2, kOF3 = kObF2 + kF2, kObF3 = kOF3 + kF2 * kN, kP = kObF3 + kN;
static_assert(kP == 44426, "the LeNet shape");
static_assert(kF1 / 8 % 2 == 1 && kPh2 / 8 % 2 == 1, "the dense layers' last step is one of eight");

// ---- fragments (lane = 4 g + tt; the k index of a step is read as pairs 2 tt | 2 tt + 1 unless said otherwise) ----------
// An operand's pair of k values in three bf16 parts, split by rounding (the convolutions' gathered inputs by cutting)
struct FA { Parts lo, hi; };   // rows g and g + 8
struct FB { Parts v; };
__device__ __forceinline__ FA a_rows(const float* w, int pitch, int g, int tt) {   // [row][k]
  const float2 a = *reinterpret_cast<const float2*>(w + g * pitch + 2 * tt), b = *reinterpret_cast<const float2*>(w + (g + 8) * pitch + 2 * tt);
  return {parts(a.x, a.y), parts(b.x, b.y)};
}
__device__ __forceinline__ FA a_cols(const float* w, int pitch, int g, int tt) {   // [k][row]
  const float* p = w + 2 * tt * pitch + g;
  return {parts(p[0], p[pitch]), parts(p[8], p[pitch + 8])};
}
__device__ __forceinline__ FA a_cols_k(const float* w, int pitch, int g, int tt) {   // [k][row], k = tt | tt + 4
  const float* p = w + tt * pitch + g;
  return {parts(p[0], p[4 * pitch]), parts(p[8], p[4 * pitch + 8])};
}
__device__ __forceinline__ FB b_rows(const float* x, int pitch, int g, int tt) {   // [column][k]
  const float2 a = *reinterpret_cast<const float2*>(x + g * pitch + 2 * tt);
  return {parts(a.x, a.y)};
}
__device__ __forceinline__ FB b_cols_k(const float* x, int pitch, int g, int tt) {   // [k][column], k = tt | tt + 4
  const float* p = x + tt * pitch + g;
  return {parts(p[0], p[4 * pitch])};
}
// Eight k: the leading parts by themselves, two pairs of the small ones as one k index of 16
__device__ __forceinline__ void mul3(float (&d)[4], float (&x)[4], float (&y)[4], const FA& a, const FB& b) {
  const uint32_t ca[4] = {a.lo.c, a.hi.c, a.lo.a, a.hi.a}, bb[4] = {a.lo.b, a.hi.b, a.lo.b, a.hi.b};
  mma::mma_bf16_k8(d, a.lo.a, a.hi.a, b.v.a);
  mma::mma_bf16(x, ca, b.v.a, b.v.c);
  mma::mma_bf16(y, bb, b.v.b, b.v.a);
  mma::mma_bf16_k8(x, a.lo.a, a.hi.a, b.v.b);
}
__device__ __forceinline__ void mul(float (&d)[4], float (&x)[4], const FA& a, const FB& b) { mul3(d, x, x, a, b); }
// Sixteen k: two steps of eight as one
__device__ __forceinline__ void mul6(float (&d)[4], float (&x)[4], float (&y)[4], const FA& a0, const FB& b0, const FA& a1, const FB& b1) {
  const uint32_t a[4] = {a0.lo.a, a0.hi.a, a1.lo.a, a1.hi.a}, b[4] = {a0.lo.b, a0.hi.b, a1.lo.b, a1.hi.b}, c[4] = {a0.lo.c, a0.hi.c, a1.lo.c, a1.hi.c};
  mma::mma_bf16(x, c, b0.v.a, b1.v.a);
  mma::mma_bf16(d, a, b0.v.a, b1.v.a);
  mma::mma_bf16(y, a, b0.v.c, b1.v.c);
  mma::mma_bf16(x, b, b0.v.b, b1.v.b);
  mma::mma_bf16(y, b, b0.v.a, b1.v.a);
  mma::mma_bf16(x, a, b0.v.b, b1.v.b);
}
__device__ __forceinline__ void mul2(float (&d)[4], float (&x)[4], const FA& a0, const FB& b0, const FA& a1, const FB& b1) { mul6(d, x, x, a0, b0, a1, b1); }
__device__ __forceinline__ void send1(uint32_t addr, float v, uint32_t bar) {   // 4 bytes to a peer
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}

template <int CL, int BT>
struct Lay {   // shared memory, in floats
  static constexpr int N1 = kF1 / CL, MT1 = (N1 + 15) / 16, Bp = 8 * BT;
  static constexpr int kPer = Bp / CL;   // samples per CTA at most
  static constexpr int kPd1 = 16 * MT1 + 8;
  static constexpr int wc = 0, w1 = wc + kW2c + kW1c, w2 = w1 + 16 * MT1 * kPq2, w3 = w2 + 88 * kPh1, b1 = w3 + kF2 * kN,
                       b2 = b1 + 16 * MT1, b3 = b2 + 96, x = b3 + 16, q1 = x + kPer * kX, m1 = q1 + kPer * kQ1,
                       m2 = m1 + kPer * kQ1 / 4, dz2 = m2 + kPer * kFlat / 4, dq1 = dz2 + kC2 * kPdz, dense = dq1 + (kPer > 1 ? 2 : 1) * kQ1;
  // q2, h1, h2, dh2 of all samples; once the dense layers are done the convolutions' gradient parts lie there
  static constexpr int q2 = dense, h1 = q2 + Bp * kPq2, h2 = h1 + Bp * kPh1, dh2 = h2 + Bp * kPh2, dense_end0 = dh2 + Bp * kPh2 + 8;
  static constexpr int g2 = dense, g1 = g2 + 2 * kW2c, dense_end1 = g1 + kWarps * kW1c;
  static constexpr int dense_end = dense_end0 > dense_end1 ? dense_end0 : dense_end1;
  static constexpr int z3 = dense_end, dh1 = z3 + Bp * 12, ing = dh1 + Bp * kPd1, col = ing + 4 * kQuads;
  // col; before it the parts of the first dense layer's outputs, the pooled maps on their way out, and the parts of dq2
  static constexpr int kCol = kPcol * 150, kPart = kWarps * 16 * MT1 * Bp, kInD = CL * kPer * kFlat;
  static constexpr int colsz = kCol > kPart ? (kCol > kInD ? kCol : kInD) : (kPart > kInD ? kPart : kInD);
  static constexpr int off = col + colsz, idx = off + 76, bars = idx + 2 * 64, total = bars + 16;
  static constexpr bool fits = kPer <= kMaxPer && total * 4 <= 227 * 1024;
  static_assert(x % 4 == 0 && q1 % 4 == 0 && dz2 % 4 == 0 && dense % 4 == 0 && z3 % 4 == 0 && ing % 4 == 0 && col % 4 == 0 && bars % 2 == 0, "alignment");
};

template <int CL, int BT>
__global__ void __launch_bounds__(kThreads, 1) cnn_mma_kernel(CnnLaunch p) {
  typedef Lay<CL, BT> M;
  constexpr int N1 = M::N1, MT1 = M::MT1, Bp = M::Bp, kPer = M::kPer, kPd1 = M::kPd1, kOwn = kQuads / CL;
  extern __shared__ __align__(128) float sm[];
  const TaskDesc t = p.r.tasks[p.r.task_begin + blockIdx.x / CL];
  if (!debug_task_ok(p.r, t)) return;   // the whole cluster alike
  const int rank = (int)mma::cluster_rank();
  if (t.steps == 0) {
    if (rank == 0) publish_empty_round(p.r, t, (uint32_t)kP);
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tt = lane & 3;
  const int B = (int)p.shape.batch, per = (B + CL - 1) / CL;
  const int b0 = min(B, rank * per), nb = min(B, b0 + per) - b0;   // this CTA's samples
  const float eta = t.eta, lambda = p.r.l2;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(sm + M::bars);   // q2, h1, dq2, convolution gradients, convolution weights
  int* const idx = reinterpret_cast<int*>(sm + M::idx);               // [64] row numbers of the own samples, labels of all: by parity
  uint16_t* const off = reinterpret_cast<uint16_t*>(sm + M::off);     // where tap k of an output of conv 2 finds its input
  uint8_t* const m1 = reinterpret_cast<uint8_t*>(sm + M::m1);         // signs of the four outputs behind a pooled one
  uint8_t* const m2 = reinterpret_cast<uint8_t*>(sm + M::m2);

#pragma unroll 1
  for (int i = tid; i < M::total; i += kThreads) sm[i] = 0.f;
  __syncthreads();
#pragma unroll 1
  for (int k = tid; k < kPw2; k += kThreads) off[k] = k < 150 ? (uint16_t)((k / 25) * 144 + ((k % 25) / 5) * 12 + k % 5) : 0;
  if (tid == 0) {
#pragma unroll 1
    for (int i = 0; i < 5; ++i) mbar_init(&bars[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  mma::cluster_sync();
  const uint32_t bytes[5] = {(uint32_t)(B * kFlat * 4), (uint32_t)(kF1 * Bp * 4), (uint32_t)(CL * nb * kFlat * 4), (uint32_t)(CL * kOwn * 16), (uint32_t)(kQuads * 16)};
  if (tid == 0) {
#pragma unroll 1
    for (int i = 0; i < 5; ++i)
      if (bytes[i]) mbar_expect_tx(&bars[i], bytes[i]);
  }
  // A thread whose wait has given up waits no more and runs through on whatever is there, but neither arms a barrier (a second arrival
  // on one that is short of bytes would be invalid) nor sends: whoever depends on it gives up in turn, the status word is set, and
  // every CTA of the cluster reaches the end.
  bool ok = true;
  auto wait = [&](int i, uint32_t parity) {
    const uint32_t at = smem_addr(&bars[i]);
#pragma unroll 1
    for (uint32_t k = 0; ok; ++k) {
      if (mma::try_wait_cluster(at, parity)) break;
      if (k >= kWaitLimit) ok = false;
    }
  };

  // ---- start model: snapshot minus own update sums still in flight ----
  const float* snap = p.r.snaps + (size_t)t.snap_slot * p.r.stride;
  auto start_value = [&](int at) {
    float v = snap[at];
#pragma unroll 1
    for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
      const InflightRef ref = p.r.inflight[t.inflight_off + f];
      v = fmaf(-ref.eta, p.r.U[(size_t)ref.row * p.r.stride + at], v);
    }
    return v;
  };
  // value of a convolution parameter's place in the slice layout: its place in the parameter vector, -1 for padding
  auto conv_at = [&](int e) {
    if (e < kW2c) {
      const int c = e / kPw2, k = e - c * kPw2;
      return k < 150 ? kOW2 + c * 150 + k : (k == 150 ? kOb2 + c : -1);
    }
    const int q = e - kW2c, tap = q >> 3, c = q & 7;
    return c >= kC1 || tap > 25 ? -1 : (tap < 25 ? kOW1 + c * 25 + tap : kOb1 + c);
  };
  {
    constexpr int kTrip = 4;
    auto fill = [&](int count, auto place, auto dest) {   // kTrip loads on their way before the first store
#pragma unroll 1
      for (int e0 = tid; e0 < count; e0 += kTrip * kThreads) {
        float v[kTrip];
#pragma unroll
        for (int q = 0; q < kTrip; ++q) {
          const int e = e0 + q * kThreads, at = e < count ? place(e) : -1;
          v[q] = at >= 0 ? start_value(at) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < kTrip; ++q)
          if (e0 + q * kThreads < count) sm[dest(e0 + q * kThreads)] = v[q];
      }
    };
    fill(kW2c + kW1c, conv_at, [&](int e) { return M::wc + e; });
    fill(kFlat * N1, [&](int e) { return kOF1 + (e / N1) * kF1 + rank * N1 + e % N1; }, [&](int e) { return M::w1 + (e % N1) * kPq2 + e / N1; });
    fill(kF1 * kF2, [&](int e) { return kOF2 + e; }, [&](int e) { return M::w2 + (e % kF2) * kPh1 + e / kF2; });
    fill(kF2 * kN, [&](int e) { return kOF3 + e; }, [&](int e) { return M::w3 + e; });
    fill(N1, [&](int e) { return kObF1 + rank * N1 + e; }, [&](int e) { return M::b1 + e; });
    fill(kF2, [&](int e) { return kObF2 + e; }, [&](int e) { return M::b2 + e; });
    fill(kN, [&](int e) { return kObF3 + e; }, [&](int e) { return M::b3 + e; });
  }
  const ClientData cd = p.r.clients[t.client];
  const uint64_t key = p.r.sample_keys[t.client];
  const float* xrows = reinterpret_cast<const float*>(cd.x);
  auto draw_rows = [&](uint32_t it) {   // row numbers and labels of iteration it (labels of every sample: the dense layers need them)
    if (tid < B) {
      const uint32_t id = sample_index(draw(key, t.sample_ctr0 + (uint64_t)it * B + tid), cd.n);
      if (tid >= b0 && tid < b0 + nb) idx[(it & 1) * 64 + tid - b0] = (int)id;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(idx + (it & 1) * 64 + 32 + tid)), "l"(cd.y + id) : "memory");
    }
  };
  auto copy_rows = [&](uint32_t it) {
#pragma unroll 1
    for (int e = tid; e < nb * (kX / 4); e += kThreads) {
      const int b = e / (kX / 4), c = e - b * (kX / 4);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(sm + M::x + 4 * e)), "l"(xrows + (size_t)idx[(it & 1) * 64 + b] * kX + 4 * c) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  draw_rows(0);
  __syncthreads();
  copy_rows(0);

  // update sums of the parameters this thread owns: first dense layer [tile][k tile], second dense layer (a tile in
  // CL-th rounds of the tile loop), third layer and small biases, first layer's biases, a piece of the convolutions
  constexpr int kR2 = (6 + CL - 1) / CL;
  float u1[MT1][2][4] = {}, u2[kR2][4] = {}, u3[3] = {}, ub1 = 0.f, uc[4] = {}, wcv[4] = {};
  if (tid < kOwn) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int at = conv_at(4 * (rank * kOwn + tid) + i);
      wcv[i] = at >= 0 ? start_value(at) : 0.f;
    }
  }

#pragma unroll 1
  for (uint32_t it = 0; it < t.steps; ++it) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (it) {
      wait(4, (it - 1) & 1);
      if (ok && tid == 0) mbar_expect_tx(&bars[4], bytes[4]);
    }
    if (it + 1 < t.steps) draw_rows(it + 1);
    __syncthreads();

    // ================= conv 1, ReLU, pooling: two planes of a pooled output per thread =================
#pragma unroll 1
    for (int e = tid; e < nb * 432; e += kThreads) {
      const int b = e / 432, r = e - b * 432, grp = r / 144, pos = r - grp * 144, py = pos / kP1, px = pos - py * kP1;
      const float* xp = sm + M::x + b * kX + 2 * py * kS + 2 * px;
      const float* w = sm + M::wc + kW2c + 2 * grp;
      float patch[6][6], z[2][4];
#pragma unroll
      for (int i = 0; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const float2 v = *reinterpret_cast<const float2*>(xp + i * kS + 2 * j);
          patch[i][2 * j] = v.x; patch[i][2 * j + 1] = v.y;
        }
      {
        const float2 bias = *reinterpret_cast<const float2*>(w + 25 * 8);
#pragma unroll
        for (int q = 0; q < 4; ++q) { z[0][q] = bias.x; z[1][q] = bias.y; }
      }
#pragma unroll
      for (int dy = 0; dy < 5; ++dy)
#pragma unroll
        for (int dx = 0; dx < 5; ++dx) {
          const float2 wv = *reinterpret_cast<const float2*>(w + (dy * 5 + dx) * 8);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float v = patch[dy + (q >> 1)][dx + (q & 1)];
            z[0][q] = fmaf(wv.x, v, z[0][q]); z[1][q] = fmaf(wv.y, v, z[1][q]);
          }
        }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t bits = 0;
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (z[c][q] > 0.f) { bits |= 1u << q; sum += z[c][q]; }
        }
        const int at = b * kQ1 + (2 * grp + c) * 144 + pos;
        sm[M::q1 + at] = 0.25f * sum;
        m1[at] = (uint8_t)bits;
      }
    }
    __syncthreads();

    // ================= conv 2, ReLU, pooling: a warp takes two rows of a sample's 8 x 8 outputs, all planes =================
    // (with at most two samples two warps share an item, each with half of the taps)
    constexpr bool kShare = kPer <= 2;
    float acc2[2][4] = {}, crs2[2][4] = {};
    const int e_half = kShare ? warp >> 3 : 0;
    auto conv2 = [&](int b, int yp, int s0, int s1, float (&acc)[2][4], float (&crs)[2][4]) {
      const float* q = sm + M::q1 + b * kQ1 + 2 * yp * kP1 + g;
      auto taps = [&](int s, FA& a, FB (&f)[2]) {
        a = a_rows(sm + M::wc + 8 * s, kPw2, g, tt);
        const uint32_t o2 = *reinterpret_cast<const uint32_t*>(off + 8 * s + 2 * tt);
        const float* i0 = q + (o2 & 0xFFFF);
        const float* i1 = q + (o2 >> 16);
        const bool last = s == kPw2 / 8 - 1 && tt == 3;   // taps 150 (the bias input) and 151
#pragma unroll
        for (int r = 0; r < 2; ++r) f[r] = {parts_t(last ? 1.f : i0[kP1 * r], last ? 0.f : i1[kP1 * r])};
      };
      FA a0, a1;
      FB f0[2], f1[2];
#pragma unroll 3
      for (int s = s0; s + 1 < s1; s += 2) {
        taps(s, a0, f0);
        taps(s + 1, a1, f1);
#pragma unroll
        for (int r = 0; r < 2; ++r) {   // added up in fp32: the tensor cores would cut a sum of positive inputs always the same way
          float d[4] = {};
          mul2(d, crs[r], a0, f0[r], a1, f1[r]);
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] += d[c];
        }
      }
      if ((s1 - s0) & 1) {
        taps(s1 - 1, a0, f0);
#pragma unroll
        for (int r = 0; r < 2; ++r) mul(acc[r], crs[r], a0, f0[r]);
      }
    };
    if (kShare) {
      const int e = warp & 7;
      if (e < 4 * nb) {
        if (e_half == 0) conv2(e >> 2, e & 3, 0, 10, acc2, crs2);
        else conv2(e >> 2, e & 3, 10, kPw2 / 8, acc2, crs2);
        if (e_half) {
          float* d = sm + M::col + kWarps * 64 + e * 256 + lane;
#pragma unroll
          for (int i = 0; i < 8; ++i) d[32 * i] = acc2[i >> 2][i & 3] + crs2[i >> 2][i & 3];
        }
      }
      __syncthreads();
    }
#pragma unroll 1
    for (int e = warp; e < 4 * nb; e += kWarps) {
      const int b = e >> 2, yp = e & 3;
      float acc[2][4] = {}, crs[2][4] = {};
      if (kShare) {
        const float* d = sm + M::col + kWarps * 64 + e * 256 + lane;
#pragma unroll
        for (int i = 0; i < 8; ++i) { acc[i >> 2][i & 3] = acc2[i >> 2][i & 3] + crs2[i >> 2][i & 3]; crs[i >> 2][i & 3] = d[32 * i]; }
      } else {
        conv2(b, yp, 0, kPw2 / 8, acc, crs);
      }
      float* st = sm + M::col + warp * 64;
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // planes g and g + 8; columns 2 tt, 2 tt + 1 of rows 2 yp, 2 yp + 1
        uint32_t bits = 0;
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float z = acc[i >> 1][2 * h + (i & 1)] + crs[i >> 1][2 * h + (i & 1)];
          if (z > 0.f) { bits |= 1u << i; sum += z; }
        }
        m2[b * kFlat + (g + 8 * h) * 16 + yp * 4 + tt] = (uint8_t)bits;
        st[(g + 8 * h) * 4 + tt] = 0.25f * sum;
      }
      __syncwarp();
      const float4 v = *reinterpret_cast<const float4*>(st + 4 * (lane & 15));
      const uint32_t at = smem_addr(sm + M::q2 + (b0 + b) * kPq2 + (lane & 15) * 16 + yp * 4);
#pragma unroll
      for (int r = 0; r < CL; r += 2)
        if (ok) mma::send_peer(mma::peer_addr(at, r + (lane >> 4)), v, mma::peer_addr(smem_addr(&bars[0]), r + (lane >> 4)));
      __syncwarp();
    }

    // ================= dense 1: own outputs, all samples; the warps share the 256 inputs =================
    wait(0, it & 1);
    if (ok && tid == 0 && it + 1 < t.steps) mbar_expect_tx(&bars[0], bytes[0]);
    {
      float acc[MT1][BT][4] = {}, crs[MT1][BT][4] = {};
      const int k = 16 * warp;
      FA a[MT1][2];
#pragma unroll
      for (int i = 0; i < MT1; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) a[i][h] = a_rows(sm + M::w1 + 16 * i * kPq2 + k + 8 * h, kPq2, g, tt);
#pragma unroll
      for (int b = 0; b < BT; ++b) {
        const FB f0 = b_rows(sm + M::q2 + 8 * b * kPq2 + k, kPq2, g, tt), f1 = b_rows(sm + M::q2 + 8 * b * kPq2 + k + 8, kPq2, g, tt);
#pragma unroll
        for (int i = 0; i < MT1; ++i) mul2(acc[i][b], crs[i][b], a[i][0], f0, a[i][1], f1);
      }
      __syncthreads();   // staged pooled maps have left the area the parts go to
      float* part = sm + M::col + warp * 16 * MT1 * Bp;
#pragma unroll
      for (int i = 0; i < MT1; ++i)
#pragma unroll
        for (int b = 0; b < BT; ++b)
#pragma unroll
          for (int r = 0; r < 2; ++r)
            *reinterpret_cast<float2*>(part + (16 * i + g + 8 * r) * Bp + 8 * b + 2 * tt) =
                make_float2(acc[i][b][2 * r] + crs[i][b][2 * r], acc[i][b][2 * r + 1] + crs[i][b][2 * r + 1]);
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < N1 * Bp; e += kThreads) {
      const int n = e / Bp, b = e % Bp;
      float v = sm[M::b1 + n];
#pragma unroll
      for (int w = 0; w < kWarps; ++w) v += sm[M::col + w * 16 * MT1 * Bp + e];
      v = fmaxf(v, 0.f);
      const uint32_t at = smem_addr(sm + M::h1 + b * kPh1 + rank * N1 + n);
#pragma unroll
      for (int r = 0; r < CL; ++r)
        if (ok) send1(mma::peer_addr(at, r), v, mma::peer_addr(smem_addr(&bars[1]), r));
    }
    wait(1, it & 1);
    if (ok && tid == 0 && it + 1 < t.steps) mbar_expect_tx(&bars[1], bytes[1]);

    // ================= dense 2, dense 3, softmax, in every CTA =================
#pragma unroll 1
    for (int e = warp; e < 6 * BT; e += kWarps) {
      const int i = e % 6, b = e / 6;
      float acc[3][4] = {};
      auto w_at = [&](int s) { return a_rows(sm + M::w2 + 16 * i * kPh1 + 8 * s, kPh1, g, tt); };
      auto h_at = [&](int s) { return b_rows(sm + M::h1 + 8 * b * kPh1 + 8 * s, kPh1, g, tt); };
#pragma unroll
      for (int s = 0; s + 1 < kF1 / 8; s += 2) mul6(acc[0], acc[1], acc[2], w_at(s), h_at(s), w_at(s + 1), h_at(s + 1));
      mul3(acc[0], acc[1], acc[2], w_at(kF1 / 8 - 1), h_at(kF1 / 8 - 1));
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int n = 16 * i + g + ((c & 2) ? 8 : 0), s = 8 * b + 2 * tt + (c & 1);
        if (n < kPh2) sm[M::h2 + s * kPh2 + n] = n < kF2 ? fmaxf(acc[0][c] + (acc[1][c] + acc[2][c]) + sm[M::b2 + n], 0.f) : 0.f;
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < Bp * kN * 2; e += kThreads) {   // two lanes per logit (whole warps: Bp is a multiple of 8, 160 | Bp * 20)
      const int o = e >> 1, b = o / kN, c = o % kN, i0 = (e & 1) * (kF2 / 2);
      const float* h = sm + M::h2 + b * kPh2 + i0;
      const float* w = sm + M::w3 + i0 * kN + c;
      float v0 = 0.f, v1 = 0.f;
#pragma unroll 7
      for (int i = 0; i < kF2 / 2; i += 2) { v0 = fmaf(h[i], w[i * kN], v0); v1 = fmaf(h[i + 1], w[(i + 1) * kN], v1); }
      float v = v0 + v1;
      v += __shfl_xor_sync(0xffffffffu, v, 1);
      if (!(e & 1)) sm[M::z3 + b * 12 + c] = v + sm[M::b3 + c];
    }
    __syncthreads();
    if (tid < 4 * Bp) {   // dZ = (p - onehot) / B; four lanes per sample
      const int s = tid >> 2, q = tid & 3;
      float* z = sm + M::z3 + s * 12;
      float v[3], mx = -3e38f, sum = 0.f;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        v[i] = q + 4 * i < kN ? z[q + 4 * i] : -3e38f;
        mx = fmaxf(mx, v[i]);
      }
      mx = fmaxf(mx, lr::shx(mx, 1));
      mx = fmaxf(mx, lr::shx(mx, 2));
#pragma unroll
      for (int i = 0; i < 3; ++i) { v[i] = lr::ex2((v[i] - mx) * lr::kLog2e); sum += v[i]; }
      sum += lr::shx(sum, 1);
      sum += lr::shx(sum, 2);
      const float fb = s < B ? 1.f / (float)B : 0.f, inv = 1.f / sum;
      const int y = idx[(it & 1) * 64 + 32 + s];
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (q + 4 * i < kN) z[q + 4 * i] = (v[i] * inv - (q + 4 * i == y ? 1.f : 0.f)) * fb;
    }
    __syncthreads();

    // ================= backward through the dense layers =================
#pragma unroll 1
    for (int e = tid; e < Bp * kPh2; e += kThreads) {   // dh2
      const int b = e / kPh2, i = e % kPh2;
      float v = 0.f;
      if (i < kF2 && sm[M::h2 + e] > 0.f) {
        const float* dz = sm + M::z3 + b * 12;
        const float* w = sm + M::w3 + i * kN;
#pragma unroll
        for (int c = 0; c < kN; ++c) v = fmaf(dz[c], w[c], v);
      }
      sm[M::dh2 + e] = v;
    }
    __syncthreads();
    if (warp < 4) {   // dh1 of the own outputs
#pragma unroll 1
      for (int e = warp; e < MT1 * BT; e += 4) {
        const int i = e / BT, b = e % BT;
        float acc[3][4] = {};
        auto w_at = [&](int s) { return a_cols(sm + M::w2 + 8 * s * kPh1 + rank * N1 + 16 * i, kPh1, g, tt); };
        auto d_at = [&](int s) { return b_rows(sm + M::dh2 + 8 * b * kPh2 + 8 * s, kPh2, g, tt); };
#pragma unroll
        for (int s = 0; s + 1 < kPh2 / 8; s += 2) mul6(acc[0], acc[1], acc[2], w_at(s), d_at(s), w_at(s + 1), d_at(s + 1));
        mul3(acc[0], acc[1], acc[2], w_at(kPh2 / 8 - 1), d_at(kPh2 / 8 - 1));
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int n = 16 * i + g + ((c & 2) ? 8 : 0), s = 8 * b + 2 * tt + (c & 1);
          sm[M::dh1 + s * kPd1 + n] = n < N1 && sm[M::h1 + s * kPh1 + rank * N1 + n] > 0.f ? acc[0][c] + (acc[1][c] + acc[2][c]) : 0.f;
        }
      }
    } else {          // dense 3 and the biases of layers 2 and 3
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int e = tid - 128 + 384 * r;
        float gr = 0.f;
        if (e < kF2 * kN) {
          const int i = e / kN, c = e % kN;
          float g4[4] = {};   // four short sums: fewer roundings on a long one
#pragma unroll
          for (int b = 0; b < Bp; ++b) g4[b & 3] = fmaf(sm[M::h2 + b * kPh2 + i], sm[M::z3 + b * 12 + c], g4[b & 3]);
          gr = (g4[0] + g4[1]) + (g4[2] + g4[3]);
          const float w = sm[M::w3 + e];
          gr = fmaf(lambda, w, gr);
          sm[M::w3 + e] = fmaf(-eta, gr, w);
        } else if (e < kF2 * kN + kF2 + kN) {
          const int q = e - kF2 * kN;
          const float* d = q < kF2 ? sm + M::dh2 + q : sm + M::z3 + q - kF2;
          const int pitch = q < kF2 ? kPh2 : 12;
          float g4[4] = {};
#pragma unroll
          for (int b = 0; b < Bp; ++b) g4[b & 3] += d[b * pitch];
          gr = (g4[0] + g4[1]) + (g4[2] + g4[3]);
          float* w = q < kF2 ? sm + M::b2 + q : sm + M::b3 + q - kF2;
          *w = fmaf(-eta, gr, *w);
        }
        u3[r] += gr;
      }
    }
    __syncthreads();
    {   // this CTA's part of dq2, 16 inputs per warp, to the samples' CTAs
      float acc[BT][4] = {}, crs[BT][4] = {};
#pragma unroll
      for (int s = 0; s < 2 * MT1; s += 2) {
        const FA a0 = a_cols(sm + M::w1 + 8 * s * kPq2 + 16 * warp, kPq2, g, tt), a1 = a_cols(sm + M::w1 + 8 * (s + 1) * kPq2 + 16 * warp, kPq2, g, tt);
#pragma unroll
        for (int b = 0; b < BT; ++b)
          mul2(acc[b], crs[b], a0, b_rows(sm + M::dh1 + 8 * b * kPd1 + 8 * s, kPd1, g, tt), a1, b_rows(sm + M::dh1 + 8 * b * kPd1 + 8 * (s + 1), kPd1, g, tt));
      }
      const uint32_t inv = (1u << 16) / (uint32_t)per + 1;
#pragma unroll
      for (int b = 0; b < BT; ++b)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int s = 8 * b + 2 * tt + q;
          if (s < B) {
            const uint32_t to = ((uint32_t)s * inv) >> 16;
            const uint32_t at = mma::peer_addr(smem_addr(sm + M::col + (rank * kPer + s - (int)to * per) * kFlat + 16 * warp + g), to);
            const uint32_t bar = mma::peer_addr(smem_addr(&bars[2]), to);
            if (!ok) continue;
            send1(at, acc[b][q] + crs[b][q], bar);
            send1(at + 32, acc[b][2 + q] + crs[b][2 + q], bar);
          }
        }
    }
    __syncwarp();   // the warp has read its 16 inputs' weights, which nobody else reads: update them
#pragma unroll
    for (int i = 0; i < MT1; ++i) {
      float acc[2][4] = {}, crs[2][4] = {};
      auto d_at = [&](int s) { return a_cols_k(sm + M::dh1 + 8 * s * kPd1 + 16 * i, kPd1, g, tt); };
      auto q_at = [&](int s, int h) { return b_cols_k(sm + M::q2 + 8 * s * kPq2 + 16 * warp + 8 * h, kPq2, g, tt); };
#pragma unroll
      for (int s = 0; s + 1 < BT; s += 2) {
        const FA a0 = d_at(s), a1 = d_at(s + 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) mul2(acc[h], crs[h], a0, q_at(s, h), a1, q_at(s + 1, h));
      }
      if (BT % 2) {
        const FA a = d_at(BT - 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) mul(acc[h], crs[h], a, q_at(BT - 1, h));
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          float2* w = reinterpret_cast<float2*>(sm + M::w1 + (16 * i + g + 8 * r) * kPq2 + 16 * warp + 8 * h + 2 * tt);
          float2 v = *w;
          const float g0 = fmaf(lambda, v.x, acc[h][2 * r] + crs[h][2 * r]), g1 = fmaf(lambda, v.y, acc[h][2 * r + 1] + crs[h][2 * r + 1]);
          v.x = fmaf(-eta, g0, v.x); v.y = fmaf(-eta, g1, v.y);
          *w = v;
          u1[i][h][2 * r] += g0; u1[i][h][2 * r + 1] += g1;
        }
    }
#pragma unroll
    for (int r0 = 0; r0 < 6; r0 += 3) {   // dense 2: 6 x 15 tiles, the products of three before their first update (stores would hold the loads back)
      float acc[3][4] = {}, crs[3][4] = {};
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int e = min(warp + kWarps * (r0 + r), 89), j = e / 6, i = e - 6 * j;
        auto d_at = [&](int s) { return a_cols_k(sm + M::dh2 + 8 * s * kPh2 + 16 * i, kPh2, g, tt); };
        auto h_at = [&](int s) { return b_cols_k(sm + M::h1 + 8 * s * kPh1 + 8 * j, kPh1, g, tt); };
#pragma unroll
        for (int s = 0; s + 1 < BT; s += 2) mul2(acc[r], crs[r], d_at(s), h_at(s), d_at(s + 1), h_at(s + 1));
        if (BT % 2) mul(acc[r], crs[r], d_at(BT - 1), h_at(BT - 1));
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int e = warp + kWarps * (r0 + r), j = e / 6, i = e - 6 * j;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int n = 16 * i + g + 8 * q;
          if (e < 90 && n < kF2) {
            float2* w = reinterpret_cast<float2*>(sm + M::w2 + n * kPh1 + 8 * j + 2 * tt);
            float2 v = *w;
            const float g0 = fmaf(lambda, v.x, acc[r][2 * q] + crs[r][2 * q]), g1 = fmaf(lambda, v.y, acc[r][2 * q + 1] + crs[r][2 * q + 1]);
            v.x = fmaf(-eta, g0, v.x); v.y = fmaf(-eta, g1, v.y);
            *w = v;
            if ((r0 + r) % CL == rank) { u2[(r0 + r) / CL][2 * q] += g0; u2[(r0 + r) / CL][2 * q + 1] += g1; }
          }
        }
      }
    }
    if (tid < N1) {
      float g4[4] = {};
#pragma unroll
      for (int b = 0; b < Bp; ++b) g4[b & 3] += sm[M::dh1 + b * kPd1 + tid];
      const float gr = (g4[0] + g4[1]) + (g4[2] + g4[3]);
      sm[M::b1 + tid] = fmaf(-eta, gr, sm[M::b1 + tid]);
      ub1 += gr;
    }

    // ================= backward through the convolutions, sample by sample =================
    float vq[kMaxPer / 2] = {};   // dq2 / 4 of sample e / 256, input e % 256, e = tid + 512 r
    if (nb > 0) {
      wait(2, it & 1);
      if (ok && tid == 0 && it + 1 < t.steps) mbar_expect_tx(&bars[2], bytes[2]);
#pragma unroll
      for (int r = 0; r < kMaxPer / 2; ++r) {
        const int e = tid + kThreads * r;
        if (e < nb * kFlat) {
          float v = 0.f;
#pragma unroll
          for (int q = 0; q < CL; ++q) v += sm[M::col + q * kPer * kFlat + e];
          vq[r] = 0.25f * v;
        }
      }
    }
    float a2[3][4] = {}, x2[3][4] = {};   // conv 2's gradient: tile pairs (taps 8 (q / 2) .., half q % 2 of the rows), q = warp + 16 i
    float a1[2][4] = {}, x1[2][4] = {};   // conv 1's: taps x planes, over the warp's share of the outputs
    int o2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) o2[i] = off[min(8 * ((warp + kWarps * i) >> 1) + g, kPw2 - 1)];
    auto put_dz2 = [&](int b) {   // dz2 = [z2 > 0] dq2 / 4
#pragma unroll
      for (int r = 0; r < kMaxPer / 2; ++r) {
        const int e = tid + kThreads * r;
        if ((e >> 8) == b) {
          const int k = e & 255, c = k >> 4, py = (k >> 2) & 3, px = k & 3;
          const uint32_t bits = m2[e];
          float2* d = reinterpret_cast<float2*>(sm + M::dz2 + c * kPdz + 16 * py + 2 * px);
          d[0] = make_float2(bits & 1 ? vq[r] : 0.f, bits & 2 ? vq[r] : 0.f);
          d[4] = make_float2(bits & 4 ? vq[r] : 0.f, bits & 8 ? vq[r] : 0.f);
        }
      }
    };
    // Conv 1's gradient of the samples from s0 (an even one) to s1 (at most two): dW1^T[tap x plane] += im2col(x)^T dz1,
    // eight outputs of a row a step; dz1 from dq1 and the sign bits.
    auto conv1_grad = [&](int s0, int s1) {
      const bool plane = g < kC1;
      const int tap1 = g + 8, tap2 = g + 16;
      const int oa = (g / 5) * kS + g % 5, ob = (tap1 / 5) * kS + tap1 % 5, oc = (tap2 / 5) * kS + tap2 % 5, od = 4 * kS + 4;
#pragma unroll 2
      for (int u = warp; u < 36 * (s1 - s0); u += kWarps) {
        const int hi = u >= 36 ? 1 : 0, v36 = u - 36 * hi, py = v36 / 3, px = 4 * (v36 - 3 * py) + tt;
        const float* xp = sm + M::x + (s0 + hi) * kX + 2 * px;
        const int at = (plane ? g : 0) * 144 + py * kP1 + px;
        const float v = plane ? 0.25f * sm[M::dq1 + hi * kQ1 + at] : 0.f;
        const uint32_t bits = m1[(s0 + hi) * kQ1 + at];
        FA lo[2], up[2];   // taps 0 .. 15; taps 16 .. 23, then 24, the bias (an input of 1) and none
        FB f[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float* xi = xp + (2 * py + h) * kS;
          f[h] = {parts(bits & (1u << (2 * h)) ? v : 0.f, bits & (2u << (2 * h)) ? v : 0.f)};
          lo[h] = {parts_t(xi[oa], xi[oa + 1]), parts_t(xi[ob], xi[ob + 1])};
          const float t0 = g == 0 ? xi[od] : (g == 1 ? 1.f : 0.f), t1 = g == 0 ? xi[od + 1] : (g == 1 ? 1.f : 0.f);
          up[h] = {parts_t(xi[oc], xi[oc + 1]), parts_t(t0, t1)};
        }
        mul2(a1[0], x1[0], lo[0], f[0], lo[1], f[1]);
        mul2(a1[1], x1[1], up[0], f[0], up[1], f[1]);
      }
    };
    __syncthreads();   // dq2's parts have been read: col may take their place
    if (nb > 0) put_dz2(0);
    __syncthreads();
#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
      const float* q1 = sm + M::q1 + b * kQ1;
      // col[tap x output] = W2^T dz2: items of 16 taps x 16 outputs; the warps with fewer gradient tiles take more
      {
        const int first = warp < 6 ? 2 * warp : 12 + 3 * (warp - 6), n = min(40, first + (warp < 6 ? 2 : 3));
#pragma unroll 1
        for (int e = first; e < n; ++e) {
          const int i = e >> 2, y = 2 * (e & 3);
          const FA f0 = a_cols_k(sm + M::wc + 16 * i, kPw2, g, tt), f1 = a_cols_k(sm + M::wc + 8 * kPw2 + 16 * i, kPw2, g, tt);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float acc[4] = {}, crs[4] = {};
            mul2(acc, crs, f0, b_cols_k(sm + M::dz2 + 8 * (y + h), kPdz, g, tt), f1, b_cols_k(sm + M::dz2 + 8 * kPdz + 8 * (y + h), kPdz, g, tt));
            float* d = sm + M::col + (16 * i + g) * kPcol + 8 * (y + h) + 2 * tt;
            if (16 * i + g < 150) *reinterpret_cast<float2*>(d) = make_float2(acc[0] + crs[0], acc[1] + crs[1]);
            if (16 * i + g + 8 < 150) *reinterpret_cast<float2*>(d + 8 * kPcol) = make_float2(acc[2] + crs[2], acc[3] + crs[3]);
          }
        }
      }
      // dW2[plane x tap] += dz2 im2col(q1)^T over four rows of outputs
      const int y0 = 4 * (warp & 1);   // (the same half for all of a warp's tiles)
#pragma unroll
      for (int y = 0; y < 4; y += 2) {
        const FA f0 = a_rows(sm + M::dz2 + 8 * (y0 + y), kPdz, g, tt), f1 = a_rows(sm + M::dz2 + 8 * (y0 + y + 1), kPdz, g, tt);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const int q = warp + kWarps * i;
          if (q < 38) {
            const int n = 8 * (q >> 1) + g;
            const float* in = q1 + o2[i] + 2 * tt + (y0 + y) * kP1;
            float v0 = in[0], v1 = in[1], v2 = in[kP1], v3 = in[kP1 + 1];
            if (n >= 150) v0 = v1 = v2 = v3 = n == 150 ? 1.f : 0.f;   // the bias
            mul2(a2[i], x2[i], f0, {parts_t(v0, v1)}, f1, {parts_t(v2, v3)});
          }
        }
      }
      __syncthreads();
      if (b + 1 < nb) put_dz2(b + 1);
#pragma unroll 1
      for (int e = tid; e < kQ1; e += kThreads) {   // dq1: every input of conv 2 adds up the entries of col it is part of
        const int c = e / 144, r = e - 144 * c, y = r / kP1, x = r - kP1 * y;
        const float* cp = sm + M::col + c * 25 * kPcol + y * 8 + x;
        float v = 0.f, w = 0.f;
#pragma unroll
        for (int dy = 0; dy < 5; ++dy) {
          const bool in_y = (uint32_t)(y - dy) < 8u;
#pragma unroll
          for (int dx = 0; dx < 5; ++dx)
            if (in_y && (uint32_t)(x - dx) < 8u) {
              const float q = cp[(dy * 5 + dx) * kPcol - 8 * dy - dx];
              if (dx & 1) w += q; else v += q;
            }
        }
        sm[M::dq1 + (b & 1) * kQ1 + e] = v + w;
      }
      __syncthreads();
      if ((b & 1) || b + 1 == nb) conv1_grad(b & ~1, b + 1);   // (the barriers of the next sample lie before dq1 is written again)
    }
    __syncthreads();   // the rows have been read
    if (it + 1 < t.steps) copy_rows(it + 1);

    // ================= the convolutions' gradients to their owners, the new weights back =================
    // (the dense layers' activations are dead: every CTA has sent its part of dq2 and used its own)
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int q = warp + kWarps * i;
      if (q < 38) {
        float* d = sm + M::g2 + (q & 1) * kW2c + g * kPw2 + 8 * (q >> 1) + 2 * tt;
        *reinterpret_cast<float2*>(d) = make_float2(a2[i][0] + x2[i][0], a2[i][1] + x2[i][1]);
        *reinterpret_cast<float2*>(d + 8 * kPw2) = make_float2(a2[i][2] + x2[i][2], a2[i][3] + x2[i][3]);
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      float* d = sm + M::g1 + warp * kW1c + (16 * i + g) * 8 + 2 * tt;
      *reinterpret_cast<float2*>(d) = make_float2(a1[i][0] + x1[i][0], a1[i][1] + x1[i][1]);
      *reinterpret_cast<float2*>(d + 64) = make_float2(a1[i][2] + x1[i][2], a1[i][3] + x1[i][3]);
    }
    __syncthreads();
#pragma unroll 1
    for (int e = tid; e < kQuads; e += kThreads) {
      float4 v;
      if (e < kW2c / 4) {
        const float4 a = *reinterpret_cast<const float4*>(sm + M::g2 + 4 * e), b = *reinterpret_cast<const float4*>(sm + M::g2 + kW2c + 4 * e);
        v = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
      } else {
        v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
          const float4 a = *reinterpret_cast<const float4*>(sm + M::g1 + w * kW1c + 4 * e - kW2c);
          v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
        }
      }
      const int to = e / kOwn;
      if (ok) mma::send_peer(mma::peer_addr(smem_addr(sm + M::ing + (rank * kOwn + e - to * kOwn) * 4), to), v, mma::peer_addr(smem_addr(&bars[3]), to));
    }
    if (tid < kOwn) {
      wait(3, it & 1);
      if (ok && tid == 0 && it + 1 < t.steps) mbar_expect_tx(&bars[3], bytes[3]);
      const int e0 = 4 * (rank * kOwn + tid);
      float gr[4] = {};
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(sm + M::ing + (r * kOwn + tid) * 4);
        gr[0] += v.x; gr[1] += v.y; gr[2] += v.z; gr[3] += v.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int e = e0 + i;
        const bool bias = e < kW2c ? e % kPw2 >= 150 : (e - kW2c) >> 3 >= 25;
        if (!bias) gr[i] = fmaf(lambda, wcv[i], gr[i]);
        wcv[i] = fmaf(-eta, gr[i], wcv[i]);
        uc[i] += gr[i];
      }
      if (it + 1 < t.steps) {   // (the last iteration's are not needed any more)
        const float4 v = make_float4(wcv[0], wcv[1], wcv[2], wcv[3]);
        const uint32_t at = smem_addr(sm + M::wc + e0);
#pragma unroll
        for (int r = 0; r < CL; ++r)
          if (ok) mma::send_peer(mma::peer_addr(at, r), v, mma::peer_addr(smem_addr(&bars[4]), r));
      }
    }
  }

  // ---- event trigger: h reached s_{i,c}; publish U_i (and the end model) ----
  __syncthreads();
  {
    // a round whose hand-overs gave up leaves NaN behind as well as the status bit
    const float bad = ok ? 0.f : __int_as_float(0x7FFFFFFF);
    float* U = p.r.U + (size_t)t.u_row * p.r.stride;
    float* W = p.r.w_end ? p.r.w_end + (size_t)t.u_row * p.r.stride : nullptr;
    auto publish = [&](int at, float u, float w) {
      U[at] = u + bad;
      if (W) W[at] = w + bad;
    };
    if (tid < kOwn) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int at = conv_at(4 * (rank * kOwn + tid) + i);
        if (at >= 0) publish(at, uc[i], wcv[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < MT1; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int n = 16 * i + g + ((q & 2) ? 8 : 0), k = 16 * warp + 8 * h + 2 * tt + (q & 1);
          if (n < N1) publish(kOF1 + k * kF1 + rank * N1 + n, u1[i][h][q], sm[M::w1 + n * kPq2 + k]);
        }
    if (tid < N1) publish(kObF1 + rank * N1 + tid, ub1, sm[M::b1 + tid]);
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      const int e = warp + kWarps * r;
      if (r % CL == rank && e < 90) {
        const int j = e / 6, i = e - 6 * j;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int n = 16 * i + g + ((q & 2) ? 8 : 0), k = 8 * j + 2 * tt + (q & 1);
          if (n < kF2) publish(kOF2 + k * kF2 + n, u2[r / CL][q], sm[M::w2 + n * kPh1 + k]);
        }
      }
    }
    if (rank == 0 && warp >= 4) {
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int e = tid - 128 + 384 * r, q = e - kF2 * kN;
        if (q < 0) publish(kOF3 + e, u3[r], sm[M::w3 + e]);
        else if (q < kF2) publish(kObF2 + q, u3[r], sm[M::b2 + q]);
        else if (q < kF2 + kN) publish(kObF3 + q - kF2, u3[r], sm[M::b3 + q - kF2]);
      }
    }
  }
  if (!ok && p.r.status && lane == 0) atomicOr(p.r.status, 1u);
  if (tid == 0 && rank == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = t.steps * (uint32_t)B; rec.flags = 1;
    p.r.trig[t.seq] = rec;
  }
  mma::cluster_sync();   // no CTA leaves while a peer may still send to it
  if (!ok) lr::linger();
}

template <int CL, int BT>
cudaError_t launch(const CnnLaunch& p, cudaStream_t s) {
  if constexpr (!Lay<CL, BT>::fits) {
    return cudaErrorInvalidConfiguration;
  } else {
    constexpr size_t smem = (size_t)Lay<CL, BT>::total * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(cnn_mma_kernel<CL, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.r.n_tasks * CL, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cnn_mma_kernel<CL, BT>, p);
  }
}

constexpr bool kFits[2][3] = {{Lay<8, 1>::fits, Lay<8, 2>::fits, Lay<8, 3>::fits}, {Lay<4, 1>::fits, Lay<4, 2>::fits, Lay<4, 3>::fits}};

}  // namespace

// CTAs per round-task for this launch; 0: not a shape, minibatch or launch for this kernel.  Eight if the device runs a cluster for
// every round-task at once (20 iterations at minibatch 16: 15 clients 0.65 ms, 16 clients 1.26 in two waves and 1.00 on four), else
// four.  Two waves of either are still several times faster than the general kernel (35 clients 1.98 ms, 38 clients there 10.4).
cudaError_t cnn_mma_cluster(const CnnShape& s, uint32_t n_tasks, uint32_t* cluster) {
  constexpr uint32_t lenet[7] = {kS, 1, kC1, kC2, kF1, kF2, kN};
  *cluster = 0;
#pragma unroll 1
  for (int i = 0; i < 7; ++i)
    if (s.dims[i] != lenet[i]) return cudaSuccess;
  const uint32_t bt = (s.batch + 7) / 8;
  if (bt > 3) return cudaSuccess;
  uint32_t sms = 0, eights = 0;
  cudaError_t e = clusters_at_once(1, &sms);
  if (e == cudaSuccess) e = clusters_at_once(8, &eights);
  if (e != cudaSuccess) return e;
  if (kFits[0][bt - 1] && n_tasks <= eights) *cluster = 8;
  else if (kFits[1][bt - 1] && n_tasks * 4 <= sms) *cluster = 4;
  else if (kFits[0][bt - 1] && eights && n_tasks * 8 <= sms) *cluster = 8;
  return cudaSuccess;
}

cudaError_t launch_cnn_mma_rounds(const CnnLaunch& p, uint32_t cluster, cudaStream_t s) {
  const uint32_t bt = (p.shape.batch + 7) / 8;
  if (cluster == 8) return bt == 1 ? launch<8, 1>(p, s) : bt == 2 ? launch<8, 2>(p, s) : launch<8, 3>(p, s);
  return bt == 1 ? launch<4, 1>(p, s) : bt == 2 ? launch<4, 2>(p, s) : launch<4, 3>(p, s);
}

}  // namespace aet
