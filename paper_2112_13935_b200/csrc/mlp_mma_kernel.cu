// Local-SGD round of one client for ReLU MLPs on minibatches of up to 64 samples (fp32, or bf16 operands with fp32
// masters): the first layer stays on the chip for the whole round, spread over a cluster.
//
// Algorithm 3, MainComputeNode, inner loop with xi a minibatch: g = mean gradient (+ lambda W), w_c -= eta_i g,
// U_i += g, repeated s_{i,c} / B times; then (c, U_i, i) is sent.
//
// A cluster of CL CTAs of 16 warps per round-task.  CTA r owns a range of the inputs (whole units of 16); it copies only
// these columns of the minibatch rows (one iteration ahead) and holds the rows of W_0 they meet - in transposed fragments,
// each thread its own entries, in TENSOR MEMORY used as a register file of 128 words per thread (tcgen05.ld / st; what
// does not fit goes on in shared memory): nothing of W_0 moves between start and trigger.  Per iteration:
//   1  Z_0^T += W_0^T X^T over the CTA's inputs (warp = hidden tile x input part), summed over the parts in shared
//      memory, each CTA's share sent to the CTA that owns the hidden row (st.async, counted by an mbarrier there);
//   2  the owner adds the CTAs' parts in rank order, bias, ReLU, and sends its rows of A_0 to every CTA;
//   3  every CTA runs the narrow layers, the softmax and the backward pass down to dZ_0 redundantly (same inputs, same
//      order: the same bits in every CTA);
//   4  dW_0^T = dZ_0^T X over the CTA's inputs: the accumulator fragment is the thread's own piece of W_0^T - update in place.
//      With bf16 operands the next iteration's step 1 rides along: an entry of W_0 is read and written once per iteration
//      (3.4 -> 3.1 ms at 12 clients of 3072-128-32-10).  fp32 keeps two passes: cross terms and split dZ_0 together do not
//      fit the registers without giving up the loads in flight (32.9 instead of 32.5 ms).
// The hand-overs need no cluster barrier: a CTA sends its part of Z_0 for the next iteration only after it has all of A_0
// of this one, which the owners sent after taking everybody's part.
//
// Products are m16n8k16 bf16.  fp32 operands go in as three bf16 parts each, six products in place of one (mma_common.cuh):
// rows and dZ lie in shared memory as three planes, split once where they are written (rows when an iteration begins); weights and
// activations are split on every read (three planes of A_0 for every peer: 37.3 instead of 31 ms for 32 clients).  One round's update sums are then as close to fp64 as sums of fp32 FMAs (0.7e-7 to
// 1e-7 rms; 2.5e-7 with two tf32 parts) and no slower: a split row is read by every hidden tile, forward and backward.  The transposed orientation puts
// hidden units on M, samples (forward) or inputs (gradient) on N: the fragment of a thread is the same in both products.
// tcgen05 would need W_0 as an operand in shared memory (bf16 image or hi/lo pair) rewritten every iteration and 64-row
// tiles; at 16-64 samples per iteration the warp-level instructions' rate (1,024 bf16 multiply-adds per clock
// and SM) is not what limits a round: hand-overs, updates and the narrow layers are.
//
// Update sums are accumulated beside the weights (W_0's in the thread's own words, the narrow layers' in shared memory).
// bf16 shapes that mlp_derives_w0 names have no room for W_0's: theirs is (W_start - W_end) / eta, and the narrow layers' lie
// in the tensor memory that frees.
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
using lr::mbar_expect_tx;
using lr::mbar_init;
using lr::smem_addr;
using mma::ldmatrix4;
using mma::ldmatrix4t;
using mma::mma_bf16;
using mma::pack_bf16;
using mma::Parts;
using mma::parts;
using mma::parts_t;

constexpr int kWarps = 16, kThreads = kWarps * 32;
constexpr int kTmemWords = 128;     // per thread: 512 columns over the four warps that share 32 lanes
constexpr int kMaxL = AET_MAX_LAYERS;

struct MmaPlan {
  int nl, d[8], B, Bp, bt;
  int CL, units, upc, upw;          // 16-input units: all, per CTA, per warp
  int MT, WM, WK;                   // hidden tiles of 16; warps over tiles, over input parts
  int rgs;                          // hidden rows owned per CTA, in groups of 8
  int bufs, xpitch;                 // minibatch columns: buffers (two; fp32 one if no more fit) of planes; elements per row
  int ap[kMaxL], zp[kMaxL], wp[kMaxL], np[kMaxL];   // pitches of A_l, dZ_l, W_l (l >= 1), padded rows of W_l
  int ext;                          // words per thread beyond tensor memory
  // offsets in floats
  int o_x, o_in, o_part, o_a[kMaxL], o_z[kMaxL], o_w[kMaxL], o_u[kMaxL], o_b, o_ub, o_gb, o_gb2, nb, o_logit, o_ext, o_idx, o_bar, total;
  int useg, us[kMaxL];              // W_0's sum derived: first 4-word piece of the narrow layers' update sums, of layer l's
  int imt[kMaxL], iitems[kMaxL], kp[kMaxL];   // ceil(2^20 / tiles of outputs | items); parts of the inputs
  int boff[kMaxL];                  // of layer l's biases in the bias arrays
};

__host__ __device__ inline int up(int v, int m) { return (v + m - 1) / m * m; }

// Whether and how a shape runs on clusters of cl CTAs with `bufs` buffers for minibatch columns; total == 0: it does not.
MmaPlan lay_out(const MlpShape& s, int cl, int bufs) {
  MmaPlan p{};
  const bool bf = s.precision == 1;
  p.nl = (int)s.n_layers;
  for (int i = 0; i <= p.nl; ++i) p.d[i] = (int)s.dims[i];
  p.B = (int)s.batch;
  p.Bp = up(p.B, bf ? 16 : 8);
  p.bt = p.Bp / 8;
  p.CL = cl;
  p.MT = (p.d[1] + 15) / 16;
  if (p.B > 64 || p.MT > 16 || (!bf && (p.MT > 8)) || p.d[p.nl] > 32 || (bf && p.d[0] % 8)) return p;
  p.WM = p.MT;
  p.WK = kWarps / p.WM;
  p.units = (p.d[0] + 15) / 16;
  p.upc = (p.units + cl - 1) / cl;
  p.upw = (p.upc + p.WK - 1) / p.WK;
  if (cl > 1 && p.upc * (cl - 1) >= p.units) return p;   // the last CTA would have nothing
  const bool derive = bf && mlp_derives_w0(s);
  const int words = p.upw * 8 * (derive ? 1 : 2);
  p.useg = words / 4;
  p.ext = words > kTmemWords ? words - kTmemWords : 0;
  p.rgs = (2 * p.MT + cl - 1) / cl;
  int o = 0;
  auto take = [&](int floats) { const int at = o; o += up(floats, 4); return at; };
  const int planes = bf ? 1 : 3;     // of bf16
  p.xpitch = 16 * p.upc + 8;         // 8 mod 16 elements: fragment loads hit different banks
  p.o_bar = take(16);
  p.o_idx = take(4 * 64);
  p.bufs = bufs;
  p.o_x = take(bufs * planes * p.Bp * p.xpitch / 2);
  p.o_in = take(cl * p.rgs * 8 * p.Bp);
  const int part = (p.WK - 1) * p.WM * p.bt * 128;
  for (int l = 0; l < p.nl; ++l) {
    const int n = up(p.d[l + 1], 16);
    p.ap[l] = n + 8;
    p.zp[l] = bf ? n + 8 : 8 * (p.bt | 1);   // dZ: bf16 [sample][n], fp32 [n][sample] (an odd number of 16-byte pieces)
    if (l + 1 < p.nl) p.o_a[l] = take(p.Bp * p.ap[l] / (bf ? 2 : 1));
    else if (l == 0) p.o_a[0] = take(p.Bp * p.ap[0]);   // no hidden layer: the logits, fp32
    if (l > 0) {
      p.o_z[l] = take(bf ? p.Bp * p.zp[l] / 2 : planes * n * p.zp[l] / 2);
      p.wp[l] = up(p.d[l], 16) + 8;
      p.np[l] = n;
      p.o_w[l] = take(n * p.wp[l]);
      if (!derive) p.o_u[l] = take(n * p.wp[l]);
    }
  }
  // dZ_0 and the partial products of the input parts are never needed at the same time
  const int z0 = bf ? p.Bp * p.zp[0] / 2 : planes * 16 * p.MT * p.zp[0] / 2, least = kWarps * 128;
  const int area = part > z0 ? (part > least ? part : least) : (z0 > least ? z0 : least);
  p.o_part = p.o_z[0] = take(area);
  for (int l = 1; l < p.nl; ++l) {
    auto inv = [](int d) { return ((1 << 20) + d - 1) / d; };
    const int mt = p.np[l] / 16, items = mt * p.bt, ks = up(p.d[l], 16) / 16;
    p.imt[l] = inv(mt); p.iitems[l] = inv(items);
    p.kp[l] = items >= kWarps ? 1 : (kWarps / items < ks ? kWarps / items : ks);
  }
  if (derive) {   // the narrow layers' update sums beside W_0 in tensor memory, a piece per tile of 16 x 8
    int at = p.useg;
    for (int l = 1; l < p.nl; ++l) {
      p.us[l] = at;
      at += (p.np[l] / 16 * (up(p.d[l], 16) / 8) + kWarps - 1) / kWarps;
    }
    p.us[0] = at;   // (the end)
    if (p.ext || 4 * at > kTmemWords) return p;
  }
  int nb = 0;
  for (int l = 0; l < p.nl; ++l) { p.boff[l] = nb; nb += up(p.d[l + 1], 16); }
  p.nb = nb;
  p.o_b = take(nb); p.o_ub = take(nb); p.o_gb = take(nb); p.o_gb2 = take(nb);
  // with two hidden layers a barrier lies between the last use of the logits and dZ_0: they share its area
  p.o_logit = !bf && p.nl > 2 && least + p.Bp * 33 <= area ? p.o_part + least : take(p.Bp * 33);
  p.o_ext = take(p.ext * kThreads);
  p.total = o;
  if ((size_t)o * 4 > 227 * 1024) p.total = 0;
  return p;
}
MmaPlan make_plan(const MlpShape& s, int cl) {
  const MmaPlan p = lay_out(s, cl, 2);
  return p.total || s.precision == 1 ? p : lay_out(s, cl, 1);
}

// ---- fragments -----------------------------------------------------------------------------------------------------
__device__ __forceinline__ void ldmatrix2t(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}

typedef __nv_bfloat16 T;
__device__ __forceinline__ void ldmatrix2(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}

// Operand fragments of a k-step of 16 in NP parts (bf16 operands one, fp32 three); arrays in shared memory are NP planes,
// `plane` elements apart.
template <int NP> struct FragA { uint32_t v[NP][4]; };
template <int NP> struct FragB { uint32_t v[NP][2]; };
template <int NP> __device__ __forceinline__ void set_pair(FragA<NP>& f, int i, float lo, float hi) {   // weights
  if constexpr (NP == 1) {
    f.v[0][i] = pack_bf16(lo, hi);
  } else {
    const Parts p = parts(lo, hi);
    f.v[0][i] = p.a; f.v[1][i] = p.b; f.v[2][i] = p.c;
  }
}

// d[i] += a b[i] for N column tiles; three parts: all but the leading product into x1 and x2.  Term by term, so that no
// instruction waits for the one before it.
template <int N>
__device__ __forceinline__ void products(float (&d)[N][4], float (&x1)[N][4], float (&x2)[N][4], const FragA<3>& a, const FragB<3> (&b)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(x1[i], a.v[2], b[i].v[0][0], b[i].v[0][1]);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(x2[i], a.v[0], b[i].v[2][0], b[i].v[2][1]);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(d[i], a.v[0], b[i].v[0][0], b[i].v[0][1]);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(x1[i], a.v[1], b[i].v[1][0], b[i].v[1][1]);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(x2[i], a.v[1], b[i].v[0][0], b[i].v[0][1]);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(x1[i], a.v[0], b[i].v[1][0], b[i].v[1][1]);
}
template <int N>
__device__ __forceinline__ void products(float (&d)[N][4], float (&)[N][4], float (&)[N][4], const FragA<1>& a, const FragB<1> (&b)[N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) mma_bf16(d[i], a.v[0], b[i].v[0][0], b[i].v[0][1]);
}
// ... over eight k (an odd number of sample tiles as k): the first halves of the fragments, two pairs of parts as one k index of 16
__device__ __forceinline__ void product_k8(float (&d)[4], float (&x1)[4], float (&x2)[4], const FragA<3>& a, const FragB<3>& b) {
  const uint32_t a20[4] = {a.v[2][0], a.v[2][1], a.v[0][0], a.v[0][1]}, a11[4] = {a.v[1][0], a.v[1][1], a.v[1][0], a.v[1][1]};
  mma_bf16(x1, a20, b.v[0][0], b.v[2][0]);
  mma_bf16(x2, a11, b.v[1][0], b.v[0][0]);
  mma::mma_bf16_k8(d, a.v[0][0], a.v[0][1], b.v[0][0]);
  mma::mma_bf16_k8(x1, a.v[0][0], a.v[0][1], b.v[1][0]);
}
// One tile by itself: an accumulator per product, so that none waits for another of its k-step
template <int NP> struct Acc { float v[NP == 1 ? 1 : 6][4] = {}; };
__device__ __forceinline__ void product(Acc<1>& d, const FragA<1>& a, const FragB<1>& b) { mma_bf16(d.v[0], a.v[0], b.v[0][0], b.v[0][1]); }
__device__ __forceinline__ void product(Acc<3>& d, const FragA<3>& a, const FragB<3>& b) {
  mma_bf16(d.v[0], a.v[0], b.v[0][0], b.v[0][1]);
  mma_bf16(d.v[1], a.v[1], b.v[0][0], b.v[0][1]);
  mma_bf16(d.v[2], a.v[0], b.v[1][0], b.v[1][1]);
  mma_bf16(d.v[3], a.v[1], b.v[1][0], b.v[1][1]);
  mma_bf16(d.v[4], a.v[2], b.v[0][0], b.v[0][1]);
  mma_bf16(d.v[5], a.v[0], b.v[2][0], b.v[2][1]);
}
__device__ __forceinline__ void product_k8(Acc<3>& d, const FragA<3>& a, const FragB<3>& b) { product_k8(d.v[0], d.v[4], d.v[3], a, b); }
__device__ __forceinline__ float value(const Acc<1>& d, int c) { return d.v[0][c]; }
__device__ __forceinline__ float value(const Acc<3>& d, int c) { return d.v[0][c] + ((d.v[1][c] + d.v[2][c]) + (d.v[3][c] + (d.v[4][c] + d.v[5][c]))); }

// First operand from an fp32 weight array [row][k] (rows g, g + 8; the k index of a step is read as pairs 2t | 2t + 1)
template <int NP> __device__ __forceinline__ void load_w(FragA<NP>& f, const float* w, int pitch, int g, int tt) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 a = *reinterpret_cast<const float2*>(w + g * pitch + 8 * h + 2 * tt), b = *reinterpret_cast<const float2*>(w + (g + 8) * pitch + 8 * h + 2 * tt);
    set_pair(f, 2 * h, a.x, a.y); set_pair(f, 2 * h + 1, b.x, b.y);
  }
}
// First operand W^T: rows are the k index of an fp32 array [n][row], k = n in pairs
template <int NP> __device__ __forceinline__ void load_wt(FragA<NP>& f, const float* w, int pitch, int g, int tt) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float* p = w + (8 * h + 2 * tt) * pitch + g;
    set_pair(f, 2 * h, p[0], p[pitch]); set_pair(f, 2 * h + 1, p[8], p[pitch + 8]);
  }
}
// Second operand from samples [sample][k], column = sample g
template <int NP> __device__ __forceinline__ void load_s(FragB<NP>& f, const T* x, int plane, int pitch, int lane) {
  const uint32_t at = smem_addr(x + (lane & 7) * pitch + (lane & 8));
#pragma unroll
  for (int q = 0; q < NP; ++q) ldmatrix2(f.v[q], at + 2u * q * plane);
}
// ... N tiles of eight samples
template <int NP, int N> __device__ __forceinline__ void load_sn(FragB<NP> (&f)[N], const T* x, int plane, int pitch, int lane) {
#pragma unroll
  for (int b = 0; b + 1 < N; b += 2) {
    const uint32_t at = smem_addr(x + (8 * b + (lane >> 4) * 8 + (lane & 7)) * pitch + (lane & 8));
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      uint32_t r[4];
      ldmatrix4(r, at + 2u * q * plane);
      f[b].v[q][0] = r[0]; f[b].v[q][1] = r[1]; f[b + 1].v[q][0] = r[2]; f[b + 1].v[q][1] = r[3];
    }
  }
  if (N % 2) load_s(f[N - 1], x + 8 * (N - 1) * pitch, plane, pitch, lane);
}
// Second operand from an array [sample][n], k = sample, column = n
template <int NP> __device__ __forceinline__ void load_st(FragB<NP>& f, const T* x, int plane, int pitch, int lane) {
  const uint32_t at = smem_addr(x + (lane & 15) * pitch);
#pragma unroll
  for (int q = 0; q < NP; ++q) ldmatrix2t(f.v[q], at + 2u * q * plane);
}
// dZ_l: bf16 [sample][n], fp32 [n][sample] in planes - there the two samples of an accumulator fragment are one word of a plane.
// As first operand dZ^T: rows n, k = sample
__device__ __forceinline__ void load_zt(FragA<1>& f, const T* z, int k, int n, int, int pitch, int lane) {
  const int i = lane >> 3, r = lane & 7;
  ldmatrix4t(f.v[0], smem_addr(z + (k + (i >> 1) * 8 + r) * pitch + n + (i & 1) * 8));
}
__device__ __forceinline__ void load_zt(FragA<3>& f, const T* z, int k, int n, int plane, int pitch, int lane) {
  const uint32_t at = smem_addr(z + (n + (lane & 15)) * pitch + k + (lane >> 4) * 8);
#pragma unroll
  for (int q = 0; q < 3; ++q) ldmatrix4(f.v[q], at + 2u * q * plane);
}
__device__ __forceinline__ void load_zt_k8(FragA<3>& f, const T* z, int k, int n, int plane, int pitch, int lane) {
  const uint32_t at = smem_addr(z + (n + (lane & 15)) * pitch + k);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    uint32_t r[2];
    ldmatrix2(r, at + 2u * q * plane);
    f.v[q][0] = r[0]; f.v[q][1] = r[1];
  }
}
// ... as second operand: k = n, columns the N tiles of eight samples from s on
template <int N> __device__ __forceinline__ void load_zb(FragB<1> (&f)[N], const T* z, int k, int s, int, int pitch, int lane) {
  load_sn(f, z + s * pitch + k, 0, pitch, lane);
}
template <int N> __device__ __forceinline__ void load_zb(FragB<3> (&f)[N], const T* z, int k, int s, int plane, int pitch, int lane) {
#pragma unroll
  for (int b = 0; b + 1 < N; b += 2) {
    const uint32_t at = smem_addr(z + (k + (lane & 15)) * pitch + s + 8 * b + (lane >> 4) * 8);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      uint32_t r[4];
      ldmatrix4t(r, at + 2u * q * plane);
      f[b].v[q][0] = r[0]; f[b].v[q][1] = r[1]; f[b + 1].v[q][0] = r[2]; f[b + 1].v[q][1] = r[3];
    }
  }
  if (N % 2) load_st(f[N - 1], z + k * pitch + s + 8 * (N - 1), plane, pitch, lane);
}
// two samples s, s + 1 (s even) of column n
__device__ __forceinline__ void put_z(FragA<1>, T* z, int s, int n, int, int pitch, float v0, float v1) {
  z[s * pitch + n] = __float2bfloat16_rn(v0);
  z[(s + 1) * pitch + n] = __float2bfloat16_rn(v1);
}
__device__ __forceinline__ void put_z(FragA<3>, T* z, int s, int n, int plane, int pitch, float v0, float v1) {
  const Parts p = parts(v0, v1);
  T* at = z + n * pitch + s;
  *reinterpret_cast<uint32_t*>(at) = p.a;
  *reinterpret_cast<uint32_t*>(at + plane) = p.b;
  *reinterpret_cast<uint32_t*>(at + 2 * plane) = p.c;
}
// ... two column tiles side by side
template <int NP> __device__ __forceinline__ void load_st2(FragB<NP> (&f)[2], const T* x, int plane, int pitch, int lane) {
  const uint32_t at = smem_addr(x + (lane & 15) * pitch + (lane >> 4) * 8);
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    uint32_t r[4];
    ldmatrix4t(r, at + 2u * q * plane);
    f[0].v[q][0] = r[0]; f[0].v[q][1] = r[1]; f[1].v[q][0] = r[2]; f[1].v[q][1] = r[3];
  }
}
template <int NP> __device__ __forceinline__ void load_st2_k8(FragB<NP> (&f)[2], const T* x, int plane, int pitch, int lane) {
  const uint32_t at = smem_addr(x + (lane & 7) * pitch + (lane & 8));
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    uint32_t r[2];
    ldmatrix2t(r, at + 2u * q * plane);
    f[0].v[q][0] = r[0]; f[1].v[q][0] = r[1];
  }
}
// Weights and dZ are split by rounding, rows and activations by cutting: of the terms that the products leave out one side
// always has a random sign.
// Activations: bf16, or fp32 as they are; second operands from them, split (cut) on the way
__device__ __forceinline__ void put_a(T* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void put_a(float* p, float v) { *p = v; }
__device__ __forceinline__ void set_pair(FragB<3>& f, int i, float lo, float hi) {
  const Parts p = parts_t(lo, hi);
  f.v[0][i] = p.a; f.v[1][i] = p.b; f.v[2][i] = p.c;
}
__device__ __forceinline__ void load_a(FragB<1>& f, const T* x, int pitch, int lane) { load_s(f, x, 0, pitch, lane); }
__device__ __forceinline__ void load_a(FragB<3>& f, const float* x, int pitch, int lane) {   // [sample][k], column = sample g
  const float* p = x + (lane >> 2) * pitch + 2 * (lane & 3);
  const float2 a = *reinterpret_cast<const float2*>(p), b = *reinterpret_cast<const float2*>(p + 8);
  set_pair(f, 0, a.x, a.y);
  set_pair(f, 1, b.x, b.y);
}
__device__ __forceinline__ void load_at(FragB<1>& f, const T* x, int pitch, int lane) { load_st(f, x, 0, pitch, lane); }
__device__ __forceinline__ void load_at(FragB<3>& f, const float* x, int pitch, int lane) {   // [sample][n], k = sample, column = n
  const float* p = x + 2 * (lane & 3) * pitch + (lane >> 2);
  set_pair(f, 0, p[0], p[pitch]);
  set_pair(f, 1, p[8 * pitch], p[9 * pitch]);
}
__device__ __forceinline__ void load_at_k8(FragB<3>& f, const float* x, int pitch, int lane) {
  const float* p = x + 2 * (lane & 3) * pitch + (lane >> 2);
  set_pair(f, 0, p[0], p[pitch]);
}
__device__ __forceinline__ float get(const float* p) { return *p; }
__device__ __forceinline__ float get(const T* p) { return __bfloat162float(*p); }

// ---- a thread's own words: tensor memory, then shared memory ----------------------------------------------------------
struct Own {
  uint32_t tmem;     // this thread's lane and first column
  float* ext;        // word i at ext[i * kThreads]
  // the words of a group; they may be used after wait() (other work goes between the two)
  __device__ __forceinline__ void issue(int group, uint32_t (&r)[8]) const {
    if (group < kTmemWords / 8) {
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                   : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                   : "r"(tmem + 8u * group) : "memory");
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) r[i] = __float_as_uint(ext[(8 * group - kTmemWords + i) * kThreads]);
    }
  }
  __device__ __forceinline__ void wait(uint32_t (&r)[8], float (&v)[8]) const {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]) : : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
  }
  __device__ __forceinline__ void store(int group, const float (&v)[8]) const {
    if (group < kTmemWords / 8) {
      asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                   ::"r"(tmem + 8u * group), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
                     "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])) : "memory");
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) ext[(8 * group - kTmemWords + i) * kThreads] = v[i];
    }
  }
  __device__ __forceinline__ void load4(int piece, float (&v)[4]) const {
    uint32_t r[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(tmem + 4u * piece) : "memory");
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
  }
  __device__ __forceinline__ void store4(int piece, const float (&v)[4]) const {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};\n\ttcgen05.wait::st.sync.aligned;"
                 ::"r"(tmem + 4u * piece), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])) : "memory");
  }
  __device__ __forceinline__ void store_wait() const { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
};

// n / d for 0 <= n < 2^13 by a multiplication with ceil(2^20 / d) (d <= 128: exact); a hardware division of integers is
// some twenty dependent instructions, and every phase of the narrow layers needs a few
__device__ __forceinline__ int div20(int n, int inv) { return (int)(((uint32_t)n * (uint32_t)inv) >> 20); }

struct MmaLaunch {
  RoundLaunch r;
  MmaPlan m;
};

// SUM: W_0's update sum is accumulated
template <bool BF, int BT, bool SUM>
__global__ void __launch_bounds__(kThreads, 1) mlp_mma_kernel(const __grid_constant__ MmaLaunch p) {
  constexpr int NP = BF ? 1 : 3, kStep = 16;
  extern __shared__ __align__(128) float smem[];
  const MmaPlan& m = p.m;
  // the number of sample tiles is a constant: run-time guards around single instructions cut the code into blocks of
  // one instruction each (three times slower)
  constexpr int bt = BT, Bp = 8 * BT;
  const int CL = m.CL, B = m.B, nl = m.nl, N1 = m.d[1], D0 = m.d[0];

  const TaskDesc t = p.r.tasks[p.r.task_begin + blockIdx.x / CL];
  if (!debug_task_ok(p.r, t)) return;   // the whole cluster alike
  const uint32_t rank = CL > 1 ? mma::cluster_rank() : 0;
  if (t.steps == 0) {
    int P = 0;
#pragma unroll 1
    for (int l = 0; l < nl; ++l) P += m.d[l] * m.d[l + 1] + m.d[l + 1];
    if (rank == 0) publish_empty_round(p.r, t, (uint32_t)P);
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tt = lane & 3;
  const float eta = t.eta, lambda = p.r.l2;

  T* const xb0 = reinterpret_cast<T*>(smem + m.o_x);
  const int xpl = Bp * m.xpitch;   // distance of the planes
  float* const inbox = smem + m.o_in;
  float* const part = smem + m.o_part;
  float* const bias = smem + m.o_b;
  float* const ubias = smem + m.o_ub;
  float* const gbias = smem + m.o_gb;
  float* const logit = smem + m.o_logit;
  int* const idx = reinterpret_cast<int*>(smem + m.o_idx);        // [2][64] row numbers, then [2][64] labels
  uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + m.o_bar);   // [0] parts of Z_0, [1] A_0
  uint32_t* const tmem_at = reinterpret_cast<uint32_t*>(bars + 2);
  typedef typename std::conditional<BF, T, float>::type In;   // a client's values, and activations
  auto A = [&](int l) { return reinterpret_cast<In*>(smem + m.o_a[l]); };
  auto Z = [&](int l) { return reinterpret_cast<T*>(smem + m.o_z[l]); };
  auto zplane = [&](int l) { return up(m.d[l + 1], 16) * m.zp[l]; };   // (fp32)

  const int u0 = min(m.units, (int)rank * m.upc), nu = min(m.units, u0 + m.upc) - u0;   // this CTA's input units
  const int x0 = 16 * u0, nx = min(D0, x0 + 16 * nu) - x0;                              // ... and columns
  const int wm = warp % m.WM, wk = warp / m.WM;
  const bool mine = wk < m.WK;                                                          // (some warps hold no tile)
  const int w0 = mine ? min(nu, wk * m.upw) : nu, wn = min(nu, w0 + m.upw) - w0;        // this warp's units
  const int rg0 = min(2 * m.MT, (int)rank * m.rgs), nrg = min(2 * m.MT, rg0 + m.rgs) - rg0;   // owned groups of 8 hidden rows

#pragma unroll 1
  for (int i = tid; i < m.total; i += kThreads) smem[i] = 0.f;
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tmem_at)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (CL > 1) mma::cluster_sync(); else __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t in_bytes = (uint32_t)(CL * nrg * 8 * Bp * 4), a_bytes = (uint32_t)(16 * m.MT * Bp * (nl > 1 ? sizeof(In) : sizeof(float)));
  if (tid == 0) {
    if (nrg > 0) mbar_expect_tx(&bars[0], in_bytes);
    mbar_expect_tx(&bars[1], a_bytes);
  }

  Own own;
  own.tmem = *tmem_at + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * kTmemWords;
  own.ext = smem + m.o_ext + tid;
  const int ug = m.upw;   // first group of W_0's update sum

  // A thread whose wait has given up waits no more and runs through on whatever is there, but neither arms a barrier (a second arrival
  // on one that is short of bytes would be invalid) nor sends: whoever depends on it gives up in turn, the status word is set, and
  // every CTA of the cluster reaches the end.
  bool ok = true;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    const uint32_t at = smem_addr(bar);
#pragma unroll 1
    for (uint32_t i = 0; ok; ++i) {
      if (mma::try_wait_cluster(at, parity)) break;
      if (i >= kWaitLimit) ok = false;
    }
  };

  const ClientData cd = p.r.clients[t.client];
  const uint64_t key = p.r.sample_keys[t.client];
  // Row numbers and labels of iteration it, then this CTA's columns of its rows into a buffer (asynchronous copies).
  auto draw_rows = [&](uint32_t it) {
    if (tid < B) {
      const uint32_t id = sample_index(draw(key, t.sample_ctr0 + (uint64_t)it * B + tid), cd.n);
      idx[(it & 1) * 64 + tid] = (int)id;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(idx + 128 + (it & 1) * 64 + tid)), "l"(cd.y + id) : "memory");
    }
  };
  constexpr int kChunk = 16 / (int)sizeof(In);
  const bool whole = (D0 * sizeof(In)) % 16 == 0;
  auto rows_of = [&](uint32_t it) { return xb0 + (m.bufs > 1 ? (it & 1) : 0) * NP * xpl; };
  // bf16: into their buffer (asynchronous copies); fp32: into L2, to be fetched and split when there is time
  auto copy_rows = [&](uint32_t it) {
    T* x = rows_of(it);
    const In* src = reinterpret_cast<const In*>(cd.x) + x0;
#pragma unroll 1
    for (int r = warp; r < B; r += kWarps) {
      const In* row = src + (size_t)idx[(it & 1) * 64 + r] * D0;
      if (!BF) {
        for (int c = 32 * lane; c < nx; c += 1024) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + c));
      } else if (whole) {
#pragma unroll 1
        for (int c = lane * kChunk; c < nx; c += 32 * kChunk)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(x + r * m.xpitch + c)), "l"(row + c) : "memory");
      } else {
#pragma unroll 1
        for (int c = lane; c < nx; c += 32) x[r * m.xpitch + c] = row[c];
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // fp32: the columns of iteration it, split into their planes
  const int quads = 4 * nu;
  const uint32_t iquads = quads ? 0xFFFFFFFFu / (uint32_t)quads + 1 : 0;   // e / quads = high word of e iquads (e quads < 2^32)
  auto split_rows = [&](uint32_t it) {
    T* const X = rows_of(it);
    const float* src = reinterpret_cast<const float*>(cd.x) + x0;
    constexpr int kTrip = 4;
#pragma unroll 1
    for (int e0 = tid; e0 < B * quads; e0 += kTrip * kThreads) {   // kTrip loads on their way before the first is split
      float4 v[kTrip];
      int at[kTrip];
#pragma unroll
      for (int q = 0; q < kTrip; ++q) {
        const int e = e0 + q * kThreads, r = (int)__umulhi((uint32_t)e, iquads), c = 4 * (e - r * quads);
        v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        at[q] = e < B * quads ? r * m.xpitch + c : -1;
        if (at[q] >= 0) {
          const float* from = src + (size_t)idx[(it & 1) * 64 + r] * D0 + c;
          if (whole) {
            if (c < nx) v[q] = __ldg(reinterpret_cast<const float4*>(from));
          } else {
            if (c < nx) v[q].x = __ldg(from);
            if (c + 1 < nx) v[q].y = __ldg(from + 1);
            if (c + 2 < nx) v[q].z = __ldg(from + 2);
            if (c + 3 < nx) v[q].w = __ldg(from + 3);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < kTrip; ++q)
        if (at[q] >= 0) {
          const Parts a = parts_t(v[q].x, v[q].y), b = parts_t(v[q].z, v[q].w);
          T* x = X + at[q];
          *reinterpret_cast<uint2*>(x) = make_uint2(a.a, b.a);
          *reinterpret_cast<uint2*>(x + xpl) = make_uint2(a.b, b.b);
          *reinterpret_cast<uint2*>(x + 2 * xpl) = make_uint2(a.c, b.c);
        }
    }
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
  // Parameter of W_0 behind word i of group (unit) u: hidden unit n, input x; false if there is none
  auto place = [&](int u, int i, size_t& at) {
    const int n = 16 * wm + g + ((i & 2) ? 8 : 0), x = 16 * (u0 + w0 + u) + 2 * tt + (i & 1) + ((i & 4) ? 8 : 0);
    at = (size_t)x * N1 + n;
    return n < N1 && x < D0;
  };
  // W_start of `n` groups from `first` on: all loads of a chunk on their way before the first is used
  constexpr int kChunkG = 4;
  auto start_groups = [&](int first, int n, float (&v)[kChunkG][8]) {
#pragma unroll
    for (int q = 0; q < kChunkG; ++q)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        size_t at;
        v[q][i] = q < n && place(first + q, i, at) ? snap[at] : 0.f;
      }
#pragma unroll 1
    for (uint32_t f = 0; f < t.inflight_cnt; ++f) {
      const InflightRef ref = p.r.inflight[t.inflight_off + f];
      const float* us = p.r.U + (size_t)ref.row * p.r.stride;
      float x[kChunkG][8];
#pragma unroll
      for (int q = 0; q < kChunkG; ++q)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          size_t at;
          x[q][i] = q < n && place(first + q, i, at) ? us[at] : 0.f;
        }
#pragma unroll
      for (int q = 0; q < kChunkG; ++q)
#pragma unroll
        for (int i = 0; i < 8; ++i) v[q][i] = fmaf(-ref.eta, x[q][i], v[q][i]);
    }
  };
  draw_rows(0);
#pragma unroll 1
  for (int g0 = 0; g0 < wn; g0 += kChunkG) {
    const int n = min(kChunkG, wn - g0);
    float v[kChunkG][8], zero[8] = {};
    start_groups(g0, n, v);
#pragma unroll
    for (int q = 0; q < kChunkG; ++q)
      if (q < n) {
        own.store(g0 + q, v[q]);
        if (SUM) own.store(ug + g0 + q, zero);
      }
  }
  if (!SUM) {
    const float zero[4] = {};
#pragma unroll 1
    for (int q = m.useg; q < m.us[0]; ++q) own.store4(q, zero);
  }
  own.store_wait();
  {
    size_t o = (size_t)D0 * N1;
#pragma unroll 1
    for (int l = 0; l < nl; ++l) {
      const int K = m.d[l], N = m.d[l + 1];
      if (l > 0) {
#pragma unroll 1
        for (int e0 = tid; e0 < K * N; e0 += 8 * kThreads) {
          float v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = e0 + q * kThreads < K * N ? start_value(o + e0 + q * kThreads) : 0.f;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int e = e0 + q * kThreads;
            if (e < K * N) smem[m.o_w[l] + (e % N) * m.wp[l] + e / N] = v[q];
          }
        }
        o += (size_t)K * N;
      }
#pragma unroll 1
      for (int e = tid; e < N; e += kThreads) bias[m.boff[l] + e] = start_value(o + e);
      o += N;
    }
  }
  __syncthreads();
  if (BF) copy_rows(0);
  else if (m.bufs > 1) split_rows(0);

  // Where this lane's row of Z_0 (g, or g + 8 for odd lanes) goes: its owner's inbox and barrier (warps of the first part).
  uint32_t row_at, row_bar;
  {
    const int rg = min(2 * wm + (tt & 1), 2 * m.MT - 1);
    const uint32_t to = (uint32_t)(rg / m.rgs);
    row_at = mma::peer_addr(smem_addr(inbox + ((int)rank * m.rgs * 8 + (rg % m.rgs) * 8 + g) * Bp + 4 * (tt >> 1)), to);
    row_bar = mma::peer_addr(smem_addr(&bars[0]), to);
  }
  const int own_q = tid / Bp, own_b = tid - own_q * Bp;   // this thread's owned rows and sample in step 2

  float acc[BT][4], crs[BT][4];   // this warp's part of Z_0^T; (fp32) the cross terms
  auto clear = [&]() {
#pragma unroll
    for (int b = 0; b < BT; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) { acc[b][c] = 0.f; crs[b][c] = 0.f; }
  };
  auto forward = [&](const T* xu, const float (&w)[8]) {   // one unit of inputs
    FragA<NP> a;
#pragma unroll
    for (int i = 0; i < 4; ++i) set_pair(a, i, w[2 * i], w[2 * i + 1]);
    if constexpr (BF) {
      FragB<NP> f[BT];
      load_sn(f, xu, xpl, m.xpitch, lane);
      products(acc, crs, crs, a, f);
    } else {   // sample tiles two at a time: room for their three parts
#pragma unroll
      for (int b = 0; b < BT; b += 2) {
        if (b + 1 < BT) {
          FragB<NP> f[2];
          load_sn(f, xu + 8 * b * m.xpitch, xpl, m.xpitch, lane);
          products(reinterpret_cast<float (&)[2][4]>(acc[b]), reinterpret_cast<float (&)[2][4]>(crs[b]), reinterpret_cast<float (&)[2][4]>(crs[b]), a, f);
        } else {
          FragB<NP> f[1];
          load_sn(f, xu + 8 * b * m.xpitch, xpl, m.xpitch, lane);
          products(reinterpret_cast<float (&)[1][4]>(acc[b]), reinterpret_cast<float (&)[1][4]>(crs[b]), reinterpret_cast<float (&)[1][4]>(crs[b]), a, f);
        }
      }
    }
  };
  auto forward_all = [&](const T* X) {
    clear();
#pragma unroll 1
    for (int u = 0; u < wn; ++u) {
      uint32_t r[8];
      float w[8];
      own.issue(u, r);
      own.wait(r, w);
      forward(X + 16 * (w0 + u), w);
    }
  };

  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();   // the first rows are in
  if (BF) forward_all(rows_of(0));

#pragma unroll 1
  for (uint32_t it = 0; it < t.steps; ++it) {
    // ================= 1: this CTA's part of Z_0^T =================
    if (it + 1 < t.steps) draw_rows(it + 1);
    __syncthreads();   // everybody is out of the last pass: the buffer of its rows and the area of dZ_0 are free
    if (!BF) {
      if (it + 1 < t.steps) copy_rows(it + 1);
      if (m.bufs == 1) {   // no second buffer: the rows come in now
        split_rows(it);
        __syncthreads();
      }
      forward_all(rows_of(it));
    }
    {
      if (!BF) {
#pragma unroll
        for (int b = 0; b < BT; ++b)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[b][c] += crs[b][c];
      }
      if (m.WK > 1) {
        if (mine && wk > 0) {
          float* pp = part + ((wk - 1) * m.WM + wm) * bt * 128 + lane;
#pragma unroll
          for (int b = 0; b < BT; ++b)
#pragma unroll
              for (int c = 0; c < 4; ++c) pp[(b * 4 + c) * 32] = acc[b][c];
        }
        __syncthreads();
      }
      if (wk == 0) {
#pragma unroll 1
        for (int k = 1; k < m.WK; ++k) {
          const float* q = part + ((k - 1) * m.WM + wm) * bt * 128 + lane;
#pragma unroll
          for (int b = 0; b < BT; ++b)
#pragma unroll
              for (int c = 0; c < 4; ++c) acc[b][c] += q[(b * 4 + c) * 32];
        }
#pragma unroll
        for (int b = 0; b < BT; ++b) {
          // neighbouring lanes trade pairs: the even one then has four samples of row g, the odd one of row g + 8
          const bool odd = tt & 1;
          const float r0 = __shfl_xor_sync(0xffffffffu, odd ? acc[b][0] : acc[b][2], 1), r1 = __shfl_xor_sync(0xffffffffu, odd ? acc[b][1] : acc[b][3], 1);
          if (ok) mma::send_peer(row_at + 32u * b, odd ? make_float4(r0, r1, acc[b][2], acc[b][3]) : make_float4(acc[b][0], acc[b][1], r0, r1), row_bar);
        }
      }
    }

    if (it + 1 < t.steps) {   // the next rows, under the hand-over
      if (BF) copy_rows(it + 1);
      else if (m.bufs > 1) split_rows(it + 1);
    }

    // ================= 2: owned rows: sum over the CTAs, bias, ReLU; A_0 (or the logits) to every CTA =================
    if (nrg > 0) {
      wait(&bars[0], it & 1);
      if (ok && tid == 0 && it + 1 < t.steps) mbar_expect_tx(&bars[0], in_bytes);
      // (without hidden layers these are the logits: fp32 whatever the operands.)  A lane's words are a packet to each peer, and
      // packets are what a hand-over takes its time for: 16 bytes each, four rows of a sample or eight in bf16.
      constexpr int kRows = BF ? 8 : 4;
      const uint32_t bar = smem_addr(&bars[1]);
      int q = own_q, b = own_b;
#pragma unroll 1
      for (int e = tid; e < nrg * (8 / kRows) * Bp; e += kThreads) {
        if (e >= kThreads) { q = e / Bp; b = e - q * Bp; }
        const int n = 8 * rg0 + kRows * q;
        float v[kRows];
#pragma unroll
        for (int i = 0; i < kRows; i += 4) {
          const float4 b4 = *reinterpret_cast<const float4*>(bias + n + i);
          v[i] = b4.x; v[i + 1] = b4.y; v[i + 2] = b4.z; v[i + 3] = b4.w;
        }
        const float* in = inbox + kRows * q * Bp + b;
#pragma unroll 4
        for (int r = 0; r < CL; ++r, in += m.rgs * 8 * Bp)
#pragma unroll
          for (int i = 0; i < kRows; ++i) v[i] += in[i * Bp];
        if (nl > 1) {
#pragma unroll
          for (int i = 0; i < kRows; ++i) v[i] = fmaxf(v[i], 0.f);
        }
        if (BF && nl > 1) {
          const uint32_t at = smem_addr(A(0) + b * m.ap[0] + n);
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = pack_bf16(v[(2 * i) % kRows], v[(2 * i + 1) % kRows]);
#pragma unroll 1
          for (int r = 0; r < CL; ++r)
            if (ok) mma::send_peer(mma::peer_addr(at, r), make_float4(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]), __uint_as_float(w[3])), mma::peer_addr(bar, r));
        } else {
#pragma unroll
          for (int i = 0; i < kRows; i += 4) {
            const uint32_t at = smem_addr(smem + m.o_a[0] + b * m.ap[0] + n + i);
#pragma unroll 1
            for (int r = 0; r < CL; ++r)
              if (ok) mma::send_peer(mma::peer_addr(at, r), make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]), mma::peer_addr(bar, r));
          }
        }
      }
    }
    wait(&bars[1], it & 1);
    if (ok && tid == 0 && it + 1 < t.steps) mbar_expect_tx(&bars[1], a_bytes);

    // ================= 3: narrow layers, redundantly in every CTA =================
#pragma unroll 1
    for (int l = 1; l < nl; ++l) {
      const int mt = m.np[l] / 16, ks = up(m.d[l], kStep) / kStep, items = mt * bt;
      const bool last = l + 1 == nl;
      // few output tiles: several warps share one, each with its part of the inputs.  (The area of the partial Z_0 is
      // free: A_0 is complete, so every part has been sent.)
      const int kp = m.kp[l];
#pragma unroll 1
      for (int e = warp; e < items * kp; e += kWarps) {
        const int part_k = kp > 1 ? div20(e, m.iitems[l]) : 0, item = e - part_k * items, b = div20(item, m.imt[l]), i = item - b * mt;
        Acc<NP> acc;
        const float* w = smem + m.o_w[l] + 16 * i * m.wp[l];
        const In* a = A(l - 1) + 8 * b * m.ap[l - 1];
        const int per = (ks + kp - 1) / kp, k1 = min(ks, per * (part_k + 1));
#pragma unroll 4
        for (int k = per * part_k; k < k1; ++k) {
          FragA<NP> fa;
          FragB<NP> fb;
          load_w(fa, w + k * kStep, m.wp[l], g, tt);
          load_a(fb, a + k * kStep, m.ap[l - 1], lane);
          product(acc, fa, fb);
        }
        if (kp > 1) {
#pragma unroll
          for (int c = 0; c < 4; ++c) part[e * 128 + c * 32 + lane] = value(acc, c);
          continue;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int n = 16 * i + g + ((c & 2) ? 8 : 0), s = 8 * b + 2 * tt + (c & 1);
          const float v = value(acc, c) + bias[m.boff[l] + n];
          if (!last) put_a(A(l) + s * m.ap[l] + n, fmaxf(v, 0.f));
          else if (n < m.d[nl]) logit[s * 33 + n] = v;
        }
      }
      __syncthreads();
      if (kp > 1) {
#pragma unroll 1
        for (int e = tid; e < items * 128; e += kThreads) {
          const int item = e >> 7, c = (e >> 5) & 3, b = div20(item, m.imt[l]), i = item - b * mt;
          const int n = 16 * i + g + ((c & 2) ? 8 : 0), s = 8 * b + 2 * tt + (c & 1);
          float v = bias[m.boff[l] + n];
#pragma unroll 1
          for (int k = 0; k < kp; ++k) v += part[k * items * 128 + e];
          if (!last) put_a(A(l) + s * m.ap[l] + n, fmaxf(v, 0.f));
          else if (n < m.d[nl]) logit[s * 33 + n] = v;
        }
        __syncthreads();
      }
    }
    {   // softmax cross-entropy: dZ = (p - onehot) / B; four lanes per sample
      const int C = m.d[nl], s = tid >> 2, q = tid & 3;
      if (s < Bp) {
        const float* z = nl > 1 ? logit + s * 33 : smem + m.o_a[0] + s * m.ap[0];
        T* dz = BF ? Z(nl - 1) + s * m.zp[nl - 1] : Z(nl - 1) + s;
        const int zpl = zplane(nl - 1);
        float v[8], mx = -3e38f, sum = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          v[i] = q + 4 * i < C ? z[q + 4 * i] : -3e38f;
          mx = fmaxf(mx, v[i]);
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (4 * i < C) { v[i] = lr::ex2((v[i] - mx) * lr::kLog2e); sum += v[i]; }
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        const float fb = s < B ? 1.f / (float)B : 0.f, inv = 1.f / sum;
        const int y = idx[128 + (it & 1) * 64 + s];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int c = q + 4 * i;
          if (4 * i >= up(C, 16)) continue;
          const float d = c < C ? (v[i] * inv - (c == y ? 1.f : 0.f)) * fb : 0.f;
          if constexpr (BF) {
            dz[c] = __float2bfloat16_rn(d);
          } else {
            const Parts p = parts(d, 0.f);
            T* at = dz + c * m.zp[nl - 1];
            at[0] = __ushort_as_bfloat16((unsigned short)p.a);
            at[zpl] = __ushort_as_bfloat16((unsigned short)p.b);
            at[2 * zpl] = __ushort_as_bfloat16((unsigned short)p.c);
          }
          if (c < C) logit[s * 33 + c] = d;   // unrounded, for the bias gradient (the four lanes have read the sample's logits)
        }
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int c = kWarps - 1 - warp; c < m.d[nl]; c += kWarps) {   // bias gradient of the last layer
      float v = 0.f;
#pragma unroll 1
      for (int s = lane; s < B; s += 32) v += logit[s * 33 + c];
#pragma unroll
      for (int k = 16; k; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
      if (lane == 0) gbias[m.boff[nl - 1] + c] = v;
    }
#pragma unroll 1
    for (int l = nl - 1; l >= 1; --l) {
      // dZ_{l-1}^T = [A_{l-1} > 0] W_l dZ_l^T: a warp takes 16 inputs and all samples, or half of them, and so has its
      // share of their bias gradients
      const int mi = up(m.d[l], 16) / 16, K = up(m.d[l + 1], kStep);
      constexpr int kHalf = BT % 2 == 0 ? BT / 2 : BT;
      const int halves = BT / kHalf;
#pragma unroll 1
      for (int e = warp; e < mi * halves; e += kWarps) {
        const int half = halves > 1 && e >= mi ? 1 : 0, i = e - half * mi, b0 = half * kHalf;
        float s0 = 0.f, s1 = 0.f;
        constexpr int kX = BF || kHalf > 4 ? 1 : 2;   // accumulators of the small terms
        float acc[kHalf][4] = {}, crs[kX][kHalf][4] = {};
#pragma unroll 1
        for (int k = 0; k < K; k += kStep) {
          FragA<NP> fa;
          FragB<NP> fb[kHalf];
          load_wt(fa, smem + m.o_w[l] + k * m.wp[l] + 16 * i, m.wp[l], g, tt);
          load_zb(fb, Z(l), k, 8 * b0, zplane(l), m.zp[l], lane);
          products(acc, crs[0], crs[kX - 1], fa, fb);
        }
#pragma unroll
        for (int b = 0; b < kHalf; ++b)
#pragma unroll
          for (int c = 0; c < 4; c += 2) {
            const int n = 16 * i + g + (c ? 8 : 0), s = 8 * (b0 + b) + 2 * tt;
            float v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q)
              v[q] = get(A(l - 1) + (s + q) * m.ap[l - 1] + n) > 0.f ? acc[b][c + q] + (BF ? 0.f : kX > 1 ? crs[0][b][c + q] + crs[kX - 1][b][c + q] : crs[0][b][c + q]) : 0.f;
            put_z(FragA<NP>(), Z(l - 1), s, n, zplane(l - 1), m.zp[l - 1], v[0], v[1]);
            if (c) s1 += v[0] + v[1]; else s0 += v[0] + v[1];
          }
        s0 += __shfl_xor_sync(0xffffffffu, s0, 1); s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
        s0 += __shfl_xor_sync(0xffffffffu, s0, 2); s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
        if (tt == 0) {
          float* gb = smem + (half ? m.o_gb2 : m.o_gb) + m.boff[l - 1] + 16 * i + g;
          gb[0] = s0; gb[8] = s1;
        }
      }
      if (l == 1) asm volatile("cp.async.wait_group 0;" ::: "memory");   // the next rows, for everybody behind this barrier
      __syncthreads();
      // dW_l^T = dZ_l^T A_{l-1}, update
      const int mt = m.np[l] / 16, ni = up(m.d[l], 16) / 8;
#pragma unroll 1
      for (int e = warp; e < mt * ni; e += kWarps) {
        const int j = div20(e, m.imt[l]), i = e - j * mt;
        Acc<NP> acc;
        FragA<NP> fa;
        FragB<NP> fb;
#pragma unroll 2
        for (int k = 0; k + kStep <= Bp; k += kStep) {
          load_zt(fa, Z(l), k, 16 * i, zplane(l), m.zp[l], lane);
          load_at(fb, A(l - 1) + k * m.ap[l - 1] + 8 * j, m.ap[l - 1], lane);
          product(acc, fa, fb);
        }
        if constexpr (BT % 2 != 0) {
          constexpr int k = Bp - 8;
          load_zt_k8(fa, Z(l), k, 16 * i, zplane(l), m.zp[l], lane);
          load_at_k8(fb, A(l - 1) + k * m.ap[l - 1] + 8 * j, m.ap[l - 1], lane);
          product_k8(acc, fa, fb);
        }
        float uq[4];
        if (!SUM) own.load4(m.us[l] + (e >> 4), uq);
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2) {
          const int at = (16 * i + g + 8 * r2) * m.wp[l] + 8 * j + 2 * tt, c = 2 * r2;
          float2* w = reinterpret_cast<float2*>(smem + m.o_w[l] + at);
          float2 wv = *w;
          const float g0 = fmaf(lambda, wv.x, value(acc, c)), g1 = fmaf(lambda, wv.y, value(acc, c + 1));
          wv.x = fmaf(-eta, g0, wv.x); wv.y = fmaf(-eta, g1, wv.y);
          *w = wv;
          if (!SUM) {
            uq[c] += g0; uq[c + 1] += g1;
          } else {
            float2* u = reinterpret_cast<float2*>(smem + m.o_u[l] + at);
            float2 uv = *u;
            uv.x += g0; uv.y += g1;
            *u = uv;
          }
        }
        if (!SUM) own.store4(m.us[l] + (e >> 4), uq);
      }
    }
    // biases: every layer's gradient is in (the barriers above lie between)
    if (nl == 1) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
    }
#pragma unroll 1
    for (int e = tid; e < m.nb; e += kThreads) {
      const float gb = gbias[e] + smem[m.o_gb2 + e];
      bias[e] = fmaf(-eta, gb, bias[e]);
      ubias[e] += gb;
    }

    // ================= 4: dW_0^T over this CTA's inputs, update in place; bf16: the next Z_0 in the same pass =================
    if (wn > 0) {
      const bool more = it + 1 < t.steps;
      const T* X = rows_of(it);
      const T* Xn = rows_of(it + 1);
      if (BF) clear();
      constexpr int kBk = BT / 2;   // whole k-steps over the samples; an odd tile goes by itself
      constexpr bool kHold = BF || BT <= 4;   // room for all of dZ_0's fragments
      const int zpl = zplane(0);
      FragA<NP> a[kHold ? (BT + 1) / 2 : 1];
      if (kHold) {
#pragma unroll
        for (int k = 0; k < kBk; ++k) load_zt(a[kHold ? k : 0], Z(0), k * kStep, 16 * wm, zpl, m.zp[0], lane);
        if constexpr (BT % 2 != 0) load_zt_k8(a[kHold ? kBk : 0], Z(0), kBk * kStep, 16 * wm, zpl, m.zp[0], lane);
      }
#pragma unroll 1
      for (int u = 0; u < wn; ++u) {
        const T* xu = X + 16 * (w0 + u);
        uint32_t r[8], rs[8];
        own.issue(u, r);
        if (SUM) own.issue(ug + u, rs);
        float d[2][4] = {}, x1[2][4] = {};
#pragma unroll
        for (int k = 0; k < kBk; ++k) {
          if (!kHold) load_zt(a[0], Z(0), k * kStep, 16 * wm, zpl, m.zp[0], lane);
          FragB<NP> f[2];
          load_st2(f, xu + k * kStep * m.xpitch, xpl, m.xpitch, lane);
          products(d, x1, x1, a[kHold ? k : 0], f);
        }
        if constexpr (BT % 2 != 0) {
          if (!kHold) load_zt_k8(a[0], Z(0), kBk * kStep, 16 * wm, zpl, m.zp[0], lane);
          FragB<NP> f[2];
          load_st2_k8(f, xu + kBk * kStep * m.xpitch, xpl, m.xpitch, lane);
          product_k8(d[0], x1[0], x1[0], a[kHold ? kBk : 0], f[0]);
          product_k8(d[1], x1[1], x1[1], a[kHold ? kBk : 0], f[1]);
        }
        float w[8], us[8];
        own.wait(r, w);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          us[i] = fmaf(lambda, w[i], (BF ? d[i >> 2][i & 3] : d[i >> 2][i & 3] + x1[i >> 2][i & 3]));   // the gradient
          w[i] = fmaf(-eta, us[i], w[i]);
        }
        own.store(u, w);
        if (SUM) {
          float v[8];
          own.wait(rs, v);
#pragma unroll
          for (int i = 0; i < 8; ++i) us[i] += v[i];
          own.store(ug + u, us);
        }
        if (BF && more) forward(Xn + 16 * (w0 + u), w);
      }
      own.store_wait();
    }
  }

  // ---- event trigger: h reached s_{i,c}; publish U_i (and the end model) ----
  __syncthreads();
  {
    // a round whose hand-overs gave up leaves NaN behind as well as the status bit
    const float bad = ok ? 0.f : __int_as_float(0x7FFFFFFF);
    float* Urow = p.r.U + (size_t)t.u_row * p.r.stride;
    float* wrow = p.r.w_end ? p.r.w_end + (size_t)t.u_row * p.r.stride : nullptr;
    const float inv_eta = 1.f / eta;
#pragma unroll 1
    for (int g0 = 0; g0 < wn; g0 += kChunkG) {
      const int n = min(kChunkG, wn - g0);
      float us[kChunkG][8];
      if (!SUM) start_groups(g0, n, us);
#pragma unroll
      for (int q = 0; q < kChunkG; ++q)
        if (q < n) {
          float w[8];
          uint32_t r[8];
          own.issue(g0 + q, r);
          own.wait(r, w);
          if (SUM) {
            own.issue(ug + g0 + q, r);
            own.wait(r, us[q]);
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) us[q][i] = (us[q][i] - w[i]) * inv_eta;
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            size_t at;
            if (!place(g0 + q, i, at)) continue;
            Urow[at] = us[q][i] + bad;
            if (wrow) wrow[at] = w[i] + bad;
          }
        }
    }
    if (rank == 0) {
      size_t o = (size_t)D0 * N1;
#pragma unroll 1
      for (int l = 0; l < nl; ++l) {
        const int K = m.d[l], N = m.d[l + 1];
        if (l > 0) {
#pragma unroll 1
          for (int e = tid; e < K * N; e += kThreads) {
            const int at = (e % N) * m.wp[l] + e / N;
            if (SUM) Urow[o + e] = smem[m.o_u[l] + at] + bad;
            if (wrow) wrow[o + e] = smem[m.o_w[l] + at] + bad;
          }
          if (!SUM) {
            const int mt = m.np[l] / 16, tiles = mt * (up(K, 16) / 8);
#pragma unroll 1
            for (int e = warp; e < tiles; e += kWarps) {
              const int j = div20(e, m.imt[l]), i = e - j * mt;
              float uq[4];
              own.load4(m.us[l] + (e >> 4), uq);
#pragma unroll
              for (int c = 0; c < 4; ++c) {
                const int n = 16 * i + g + ((c & 2) ? 8 : 0), k = 8 * j + 2 * tt + (c & 1);
                if (n < N && k < K) Urow[o + (size_t)k * N + n] = uq[c] + bad;
              }
            }
          }
          o += (size_t)K * N;
        }
#pragma unroll 1
        for (int e = tid; e < N; e += kThreads) {
          Urow[o + e] = ubias[m.boff[l] + e] + bad;
          if (wrow) wrow[o + e] = bias[m.boff[l] + e] + bad;
        }
        o += N;
      }
    }
  }
  if (!ok && p.r.status && lane == 0) atomicOr(p.r.status, 1u);
  if (tid == 0 && rank == 0) {
    TriggerRec rec;
    rec.client = t.client; rec.round = t.round; rec.samples_done = t.steps * (uint32_t)B; rec.flags = 1;
    p.r.trig[t.seq] = rec;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (CL > 1) mma::cluster_sync(); else __syncthreads();   // no CTA leaves while a peer may still send to it
  if (!ok) lr::linger();
  __syncwarp();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_at) : "memory");
}

template <bool BF, int BT, bool SUM>
cudaError_t launch(const MmaLaunch& p, cudaStream_t s) {
  const size_t smem = (size_t)p.m.total * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(mlp_mma_kernel<BF, BT, SUM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(p.r.n_tasks * p.m.CL, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.m.CL;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.m.CL > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, mlp_mma_kernel<BF, BT, SUM>, p);
}

// The widest cluster of which the device runs one for every round-task of the launch at once; where there is none, the smallest
// power of two that holds the first layer.  Widths that are no powers of two count where the inputs' units ask for them: the 49 of
// 784 inputs leave the last of eight CTAs nothing, but are seven for each of seven (12 clients of 784-100-37-10, four -> seven CTAs:
// 3.0 -> 2.5 ms).
cudaError_t pick_plan(const MlpShape& s, uint32_t n_tasks, MmaPlan* out) {
  *out = MmaPlan{};
#pragma unroll 1
  for (int cl = 8; cl >= 1; --cl) {
    const MmaPlan p = make_plan(s, cl);
    if (!p.total) continue;
    uint32_t fit = 0;
    if (const cudaError_t e = clusters_at_once((uint32_t)cl, &fit)) return e;
    if (n_tasks <= fit || !(cl & (cl - 1))) *out = p;
    if (n_tasks <= fit) break;
  }
  return cudaSuccess;
}

}  // namespace

bool mlp_mma_eligible(const MlpShape& shape) {
#pragma unroll 1
  for (int cl = 8; cl >= 1; cl >>= 1)
    if (make_plan(shape, cl).total) return true;
  return false;
}

cudaError_t launch_mlp_mma_rounds(const MlpLaunch& p, cudaStream_t s) {
  MmaLaunch q;
  q.r = p.r;
  if (const cudaError_t e = pick_plan(p.shape, p.r.n_tasks, &q.m)) return e;
  if (!q.m.total) return cudaErrorInvalidConfiguration;
  if (p.shape.precision == 0) {
    switch (q.m.bt) {
      case 1: return launch<false, 1, true>(q, s);
      case 2: return launch<false, 2, true>(q, s);
      case 3: return launch<false, 3, true>(q, s);
      case 4: return launch<false, 4, true>(q, s);
      case 5: return launch<false, 5, true>(q, s);
      case 6: return launch<false, 6, true>(q, s);
      case 7: return launch<false, 7, true>(q, s);
      default: return launch<false, 8, true>(q, s);
    }
  }
  const bool sum = !mlp_derives_w0(p.shape);
  switch (q.m.bt) {
    case 2: return sum ? launch<true, 2, true>(q, s) : launch<true, 2, false>(q, s);
    case 4: return sum ? launch<true, 4, true>(q, s) : launch<true, 4, false>(q, s);
    case 6: return sum ? launch<true, 6, true>(q, s) : launch<true, 6, false>(q, s);
    default: return sum ? launch<true, 8, true>(q, s) : launch<true, 8, false>(q, s);
  }
}

}  // namespace aet
