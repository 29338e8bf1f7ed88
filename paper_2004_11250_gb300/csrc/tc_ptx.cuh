// Inline-PTX helpers shared by the tensor-core convolution kernels: shared
// memory matrix descriptors, mbarriers, tcgen05 MMA / TMEM access and named
// barriers.  Everything here is a thin wrapper over one PTX instruction.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

namespace ppc_ptx {

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, K-major, no swizzle: core matrices of 8 rows
// x 16 bytes; lbo = byte distance between the two K halves, sbo = 128 between
// groups of 8 rows; bit 46 = descriptor version of this architecture.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)(128 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor: D f32, A and B tf32, both K-major, shape M x N.
__host__ __device__ constexpr uint32_t idesc_tf32(int m, int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Instruction descriptor: D f32, A and B f16 (kind::f16), both K-major, shape M x N.
__host__ __device__ constexpr uint32_t idesc_f16(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t a, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count));
}
__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(a), "r"(parity)
               : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(uint32_t a) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t a, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes) : "memory");
}

// Named barrier 1 over the first NT threads of the CTA (the loader warps).
// Every one of those threads must reach each use.
template <int NT>
__device__ __forceinline__ void group_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}
// OR of v over the same NT threads (a barrier too), so all of them take the same branch.
template <int NT>
__device__ __forceinline__ bool group_any(bool v) {
  uint32_t r;
  asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; bar.red.or.pred q, 1, %2, p; selp.u32 %0, 1, 0, q; }"
               : "=r"(r)
               : "r"((uint32_t)v), "n"(NT)
               : "memory");
  return r != 0;
}

__device__ __forceinline__ void tm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_ld16(uint32_t ta, float (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(ta));
}
__device__ __forceinline__ void tm_ld8(uint32_t ta, float (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(ta));
}
__device__ __forceinline__ void tm_ld(uint32_t ta, float (&v)[16]) { tm_ld16(ta, v); }
__device__ __forceinline__ void tm_ld(uint32_t ta, float (&v)[8]) { tm_ld8(ta, v); }
__device__ __forceinline__ void mma_tf32(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p; }" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// CTA pairs (cta_group::2, issued by one thread of the even CTA of the pair):
// an M = 256 MMA whose A rows 0-127 and 128-255 come from the two CTAs' shared
// memory at the same address, whose B columns 0 .. N/2-1 and N/2 .. N-1 come
// likewise from the two CTAs, and whose D rows land in each CTA's own TMEM.
__device__ __forceinline__ void mma_tf32_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p; }" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_f16_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
// arrives on the mbarrier at this shared address in every CTA of the cluster
// named by mask, once the pair's earlier MMAs are complete
__device__ __forceinline__ void mma_commit_pair(uint32_t bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"(mask)
      : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the shared::cluster address of this CTA's shared address a in cluster CTA rank
__device__ __forceinline__ uint32_t map_rank(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
// arrive (release at cluster scope) on an mbarrier of another CTA of the cluster
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// the same with the default scope: hands over operands that the async proxy reads (after fence.proxy.async) or
// tensor memory; it does not wait for the thread's global stores, as the cluster-scope release does
__device__ __forceinline__ void mbar_arrive_pair(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// Two fp32 operations per instruction (each element rounded as the scalar one).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// tf32 split of an fp32 value: hi keeps the sign, exponent and 10 explicit
// mantissa bits (exact in tf32); lo = v - hi is exact in fp32.
__device__ __forceinline__ float tf32_hi(float v) { return __uint_as_float(__float_as_uint(v) & 0xFFFFE000u); }

// fp16 split of 8 fp32 values scaled by sc (a power of two): hi = f16(v sc) and
// lo = f16((v sc - hi) * 2^11), rounded to nearest, 8 halves per 16 bytes in the
// values' order (the K-major row of a kind::f16 operand).  v sc - hi is exact in
// fp32.  Returns a word that is nonzero when some hi half is infinite or NaN,
// i.e. |v sc| >= 65520 (fp16 overflow) or v is not a number: for every half the
// exponent field plus one carries into the cleared sign bit exactly when it is
// all ones.
__device__ __forceinline__ uint32_t split_f16x8(const float* v, float sc, uint4& h, uint4& l) {
  uint32_t hw[4], lw[4];
  uint32_t bad = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float a = v[2 * k] * sc, b = v[2 * k + 1] * sc;
    const __half2 hh = __floats2half2_rn(a, b);
    const float2 hf = __half22float2(hh);
    const __half2 ll = __floats2half2_rn((a - hf.x) * 2048.f, (b - hf.y) * 2048.f);
    hw[k] = *reinterpret_cast<const uint32_t*>(&hh);
    lw[k] = *reinterpret_cast<const uint32_t*>(&ll);
    bad |= ((hw[k] & 0x7FFF7FFFu) + 0x04000400u) & 0x80008000u;
  }
  h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
  l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
  return bad;
}

// The same split with packed fp32 operations and the range test as a running maximum of |hi| (NaN propagates): the
// caller tests the result with f16_max_bad once at the end.
__device__ __forceinline__ void split_f16x8_max(const float* v, float sc, uint4& h, uint4& l, __half2& mx) {
  uint32_t hw[4], lw[4];
  const uint64_t s2 = pack2(sc, sc), m1 = pack2(-1.f, -1.f), e2 = pack2(2048.f, 2048.f);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint64_t vs = mul2(pack2(v[2 * k], v[2 * k + 1]), s2);
    float a, b;
    unpack2(vs, a, b);
    const __half2 hh = __floats2half2_rn(a, b);
    const float2 hf = __half22float2(hh);
    unpack2(mul2(fma2(pack2(hf.x, hf.y), m1, vs), e2), a, b);
    const __half2 ll = __floats2half2_rn(a, b);
    hw[k] = *reinterpret_cast<const uint32_t*>(&hh);
    lw[k] = *reinterpret_cast<const uint32_t*>(&ll);
    mx = __hmax2_nan(mx, __habs2(hh));
  }
  h = make_uint4(hw[0], hw[1], hw[2], hw[3]);
  l = make_uint4(lw[0], lw[1], lw[2], lw[3]);
}
// nonzero when some |hi| in the running maximum was infinite or NaN
__device__ __forceinline__ bool f16_max_bad(__half2 mx) {
  const uint32_t w = *reinterpret_cast<const uint32_t*>(&mx);
  return (((w & 0x7FFF7FFFu) + 0x04000400u) & 0x80008000u) != 0;
}

}  // namespace ppc_ptx
