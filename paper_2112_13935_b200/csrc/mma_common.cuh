// Warp-level tensor-core products of fp32 operands for the round kernels: m16n8k16 bf16 instructions on operands in three parts,
// m16n8k8 tf32 instructions on operands in two, and the cluster-scope barrier wrappers the kernels that split one round-task over
// CTAs use.
//
// Why mma.sync here and not tcgen05: the contractions of a batch-1 regression block are 16 samples x 10 classes
// (and 16 x 16 Gram matrices).  tcgen05 needs M >= 64, its operands in shared memory in both orientations and its
// results fetched back from tensor memory; here the update sum's accumulator fragment IS the operand fragment of
// the next logits product (see frag order below), so nothing moves between the two products of a block.
// Measured on this part: m16n8k8 tf32 issues every 8 cycles per scheduler (512 multiply-adds per clock and SM),
// 21 cycles latency.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace aet {
namespace mma {

// Two tf32 operands for one fp32 value, v = hi + lo: the tensor cores read the top 19 bits of a word.
//   split    hi = nearest tf32, lo = the remainder (signed): hi.hi + hi.lo + lo.hi keeps a product to about 2^-22
//   split_t  hi = v as it stands (its top 19 bits are read), lo = what that leaves out: one logic operation and one
//            subtraction.  What the product loses of v is below 2^-21 and 2^-23 on average, an fp32 unit in the last place;
//            used for the Gram matrices (small corrections) and the crowded regression's logits: errors there move a softmax, not a
//            sum that is kept.
// Measured: cvt.rna.tf32 costs a scheduler 4 cycles, the logic operation 2; crowded regression rounds spent 45 % of
// the integer pipe and 44 % of their instructions on the former.
struct Split { uint32_t hi, lo; };
__device__ __forceinline__ Split split(float v) {
  Split s;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(s.hi) : "f"(v));
  s.lo = __float_as_uint(v - __uint_as_float(s.hi));
  return s;
}
__device__ __forceinline__ Split split_t(float v) {
  Split s;
  s.hi = __float_as_uint(v);
  s.lo = __float_as_uint(v - __uint_as_float(s.hi & 0xFFFFE000u));
  return s;
}
// as split (ties away from zero), by an addition on the bits: half of the cost of the conversion
__device__ __forceinline__ Split split_r(float v) {
  Split s;
  s.hi = (__float_as_uint(v) + 0x1000u) & 0xFFFFE000u;
  s.lo = __float_as_uint(v - __uint_as_float(s.hi));
  return s;
}
// d[16 x 8] += a[16 x 8] b[8 x 8]; lane = 4 g + t.  a0 (row g, k t), a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4);
// b0 (k t, col g), b1 (t + 4, g); d0 (row g, col 2t), d1 (g, 2t + 1), d2 (g + 8, 2t), d3 (g + 8, 2t + 1).
__device__ __forceinline__ void tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ---- bf16: m16n8k16, pairs in one register --------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two fp32 values as three bf16 each, a + b + c, exactly: 8 + 8 + 8 bits of significand, pairs in one register.
//   parts    nearest at each step (remainders of either sign)
//   parts_t  cut at each step: no conversions, only logic and two subtractions per value
// aa + (ab + ba) + (ac + bb + ca) leaves 2^-25 of a product out, of random sign where at least one side is rounded.  Against
// sums of fp32 FMAs (0.5e-7 to 1.0e-7 rms for 32 terms, 2.3e-7 to 5.0e-7 for 784; two tf32 parts: 0.9e-7 to 1.3e-7, cut 2.0e-7
// to 2.3e-7): 0.3e-7 to 0.5e-7 for 32, and the leading products of 8 x 8 bits barely feel that the tensor cores cut instead
// of rounding, so that 128 terms in one accumulator are still below FMAs (0.5e-7 to 1.2e-7 against 1.0e-7 to 2.0e-7).  The
// tensor work is that of three tf32 products.
struct Parts { uint32_t a, b, c; };
__device__ __forceinline__ float lo_of(uint32_t pair) { return __uint_as_float(pair << 16); }
__device__ __forceinline__ float hi_of(uint32_t pair) { return __uint_as_float(pair & 0xFFFF0000u); }
__device__ __forceinline__ Parts parts(float x, float y) {
  Parts p;
  p.a = pack_bf16(x, y);
  x -= lo_of(p.a); y -= hi_of(p.a);
  p.b = pack_bf16(x, y);
  p.c = pack_bf16(x - lo_of(p.b), y - hi_of(p.b));
  return p;
}
__device__ __forceinline__ Parts parts_t(float x, float y) {
  Parts p;
  p.a = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
  x -= hi_of(__float_as_uint(x)); y -= hi_of(__float_as_uint(y));
  p.b = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
  x -= hi_of(__float_as_uint(x)); y -= hi_of(__float_as_uint(y));
  p.c = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
  return p;
}
// m16n8k8: a0 (row g, k 2t | 2t + 1), a1 (g + 8, the same); b0 (k 2t | 2t + 1, col g)
__device__ __forceinline__ void mma_bf16_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(b0));
}
__device__ __forceinline__ void ldmatrix4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// ---- cluster helpers -----------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t saddr, uint32_t rank) {   // shared::cluster address of a peer's copy
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// 16 bytes into a peer's shared memory; they count towards the transaction bytes of a barrier there (no fence needed)
__device__ __forceinline__ void send_peer(uint32_t addr, float4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ float ld_peer(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void arrive_peer(uint32_t bar) {   // release at cluster scope
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace mma
}  // namespace aet
