// Device helpers shared by the tensor-core translation kernels (m2l_tc.cu,
// m2l_cx.cu): shared-memory matrix descriptors, mbarrier waits with a time
// limit, asynchronous copies, tcgen05 MMA issue and tensor-memory loads, and
// the scaled FP16 split.  Written from the PTX ISA (tcgen05, mbarrier,
// cp.async, cp.async.bulk, red).
#pragma once
#include <cuda_fp16.h>

#include <cstdint>

#include "common.h"

namespace dfmm {
namespace tc {

constexpr unsigned long long kWaitNs = 200000000ull;   // 0.2 s bound on every wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of fp16 element (row, k) of a tile in the canonical K-major
// layout without swizzle: 8-row x 16-byte core matrices, K-adjacent cores
// 128 B apart, 8-row groups `sbo` bytes apart
__host__ __device__ __forceinline__ uint32_t kmaj_off(int row, int k, int sbo) {
  return (uint32_t)((row >> 3) * sbo + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor of that layout: start, LBO = 128 B, SBO,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(128u >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1u << 46;
  return d;
}

// descriptor of a K-major tile with the 128-byte swizzle: rows of 128 bytes,
// 8-row groups 1024 B apart, the 16-byte piece p of row r at r * 128 +
// ((p ^ (r & 7)) << 4); the tile is 1024-byte aligned, saddr may add 32-byte K steps
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1u << 46;
  d |= (uint64_t)2u << 61;
  return d;
}
__host__ __device__ __forceinline__ uint32_t sw128_off(int row, int piece) {
  return (uint32_t)(row * 128 + ((piece ^ (row & 7)) << 4));
}

// instruction descriptor, kind::f16: D f32, A and B f16, both K-major,
// M = 128, N = n; neg_a negates A
__device__ __forceinline__ uint32_t idesc_f16(int n, bool neg_a = false) {
  return (1u << 4) | ((neg_a ? 1u : 0u) << 13) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for the phase with the given parity to complete.  Gives up (false)
// after kWaitNs, or as soon as another CTA has reported a timeout, and then
// reports the timeout itself.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned* status) {
  if (mbar_try_wait(bar, parity)) return true;
  unsigned long long t0 = globaltimer();
  while (!mbar_try_wait(bar, parity)) {
    if (globaltimer() - t0 > kWaitNs || (*(volatile unsigned*)status & kStatusTimeout)) {
      atomicOr(status, kStatusTimeout);
      return false;
    }
  }
  return true;
}

// Wait without giving up early on another CTA's report (used only to let a
// CTA's own copies and MMAs land before it frees its memory); time-limited.
__device__ __forceinline__ bool mbar_wait_drain(uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  unsigned long long t0 = globaltimer();
  while (!mbar_try_wait(bar, parity))
    if (globaltimer() - t0 > kWaitNs) return false;
  return true;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void cp_async16(uint32_t saddr, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(saddr), "l"(g) : "memory");
}
// 16 zero bytes (source size 0: nothing is read)
__device__ __forceinline__ void cp_async16_zero(uint32_t saddr, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, 0;" ::"r"(saddr), "l"(g) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// bulk global -> shared copy of `bytes` (multiple of 16), completing on `bar`
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// ---- issue by a whole warp ----
// The MMA warp runs its loop converged and one elected lane issues: ring positions and
// descriptors are then uniform over the warp and stay in uniform registers, which the MMA
// reads.  Issued from one diverged thread, every descriptor went through a register
// move of its own and an MMA took 115 to 140 clocks to issue whatever its size.

// 1 on one lane of the (converged) warp
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p;
}
// mbar_wait by all lanes together, with one result
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, unsigned* status) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const unsigned long long t0 = globaltimer();
  for (;;) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const bool late = globaltimer() - t0 > kWaitNs || (*(volatile unsigned*)status & kStatusTimeout);
    if (__any_sync(0xffffffffu, late)) {
      atomicOr(status, kStatusTimeout);
      return false;
    }
  }
}
__device__ __forceinline__ void mma_f16_by(uint32_t lead, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                           uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n @q tcgen05.mma.cta_group::1.kind::f16 "
      "[%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lead));
}
__device__ __forceinline__ void mma_commit_by(uint32_t lead, uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 "
      "[%0];\n}\n" ::"r"(bar),
      "r"(lead)
      : "memory");
}

// 16 lanes x 32 columns of one accumulator (.16x256b, 4 repetitions): thread t
// gets lane t/4 (r[4j], r[4j+1]) and lane t/4 + 8 (r[4j+2], r[4j+3]) at columns
// 8j + 2 (t % 4) + {0, 1}
__device__ __forceinline__ void tmem_ld16x256_x4(uint32_t ta, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(ta));
}

struct Ring {   // position in a ring of shared-memory slots, and the parity of its current use
  int st = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int n) {
    if (++st == n) { st = 0; ph ^= 1u; }
  }
};

// column / nrhs for a tile column below 128 and 1 <= nrhs <= 64 by multiplication:
// exact, since 127 * 63 < 2^16 (a division per gathered row took 3.5k clocks of a 12k-clock tile)
__device__ __forceinline__ uint32_t rhs_magic(int nrhs) { return (65535u + (uint32_t)nrhs) / (uint32_t)nrhs; }
__device__ __forceinline__ int div_rhs(int col, uint32_t magic) { return (int)(((uint32_t)col * magic) >> 16); }

// fire-and-forget adds of two / four floats to global memory (no value returned)
__device__ __forceinline__ void red_add2(float* p, float a, float b) {
  asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void red_add4(float* p, float a, float b, float c, float d) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

// smallest power of two >= m (1 for m == 0)
__device__ __forceinline__ float pow2_above(float m) {
  if (!(m > 0.f)) return 1.f;
  int e;
  frexpf(m, &e);
  return ldexpf(1.f, e);
}

__device__ __forceinline__ void split_h(float v, __half& h, __half& l) {
  h = __float2half_rn(v);
  l = __float2half_rn(v - __half2float(h));
}

}  // namespace tc
}  // namespace dfmm
