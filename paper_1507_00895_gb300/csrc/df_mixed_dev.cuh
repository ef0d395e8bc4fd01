// Helpers of the mixed-precision ladder kernels (DF_FP32_IR) and of the tensor-core products:
// FP32 complex arithmetic, exponents, swizzled operand rows, and the tcgen05 (5th-generation
// tensor core) instructions.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>

#include "df_internal.cuh"

namespace df {


constexpr int kTile = 4;          // rows and columns per thread of the relaid S (df_mixed64_dev.cuh)
constexpr int kPanel = 8;         // pivot columns per Gauss-Jordan panel

// padded order classes of the mixed ladders: 16, 32, 64, 128
__host__ __device__ inline int mixed_pad(int n) {
  int np = 16;
  while (np < n) np *= 2;
  return np;
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cfmaf2(float2 a, float2 b, float2 c) {   // c + a b
  return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}
// 2^e as a float for e >= -126 (0 below: the terms it scales are < 2^-100 of the result)
__device__ __forceinline__ float pow2f(int e) {
  return e < -126 ? 0.f : __int_as_float((e + 127) << 23);
}

// exponent e with |v| < 2^e (v != 0): unbiased exponent + 1
__device__ __forceinline__ int exp_bound_f32(float v) {
  const unsigned bits = __float_as_uint(v) & 0x7FFFFFFFu;
  if (bits == 0) return -1000;
  const int E = (int)(bits >> 23);
  return (E == 0 ? -126 : E - 127) + 1;
}

// operand rows of 64 16-bit values (32 words): word w of row r stored at
// w ^ ((r & 7) << 2), the 128-byte swizzle of the descriptors below
__device__ __forceinline__ int swz(int row, int k) {
  return row * 64 + ((((k >> 1) ^ ((row & 7) << 2))) << 1) + (k & 1);
}

// ---- tcgen05 (5th-generation tensor core) helpers ----
// Operands are K-major bf16 tiles in shared memory with 128-byte rows in the
// 128-byte swizzle (16-byte chunk c of row r at chunk c ^ (r & 7); 8-row groups
// 1024 bytes apart, group base 1024-aligned) -- the layout swz() writes.  The
// FP32 accumulators live in tensor memory (TMEM): row i of D in TMEM lane i,
// column j in TMEM column (base + j).
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t umma_desc_sw128(unsigned saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// instruction descriptor, kind::f16: bf16 A and B (K-major), FP32 D, M x N
__host__ __device__ constexpr unsigned umma_idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}
__device__ __forceinline__ void umma_bf16(unsigned dtmem, uint64_t a, uint64_t b, unsigned idesc, unsigned acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// arrive on mbar once every MMA issued so far by this thread has completed
__device__ __forceinline__ void umma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
               : "memory");
}
// bounded wait for the completion of the given parity; false if it gave up
// after `spins` polls
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, unsigned parity, unsigned spins = kMbarSpin) {
  const unsigned a = smem_u32(mbar);
  for (unsigned it = 0; it < spins; ++it) {
    unsigned done;
    asm volatile(
        "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void tc05_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc05_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic-proxy shared-memory writes -> visible to the tensor core's reads
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// 16 consecutive FP32 columns of this thread's TMEM lane (warp w reads lanes 32 (w % 4) ..)
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float* v) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
// TMEM allocation of a fixed power-of-two column count (warp 0 calls alloc/dealloc)
template <int COLS>
__device__ __forceinline__ void tmem_alloc_cols(unsigned* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "n"(COLS)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int COLS>
__device__ __forceinline__ void tmem_dealloc_cols(unsigned taddr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "n"(COLS) : "memory");
}

}  // namespace df
