// FP32-accurate products on the tensor cores from three bf16 parts per value (tcgen05, sm_103a):
// shared by the triangular solves (tc_solve.cu) and the trailing update of large matrices
// (tc_gemm96.cu).
#pragma once

#include <cstdint>

#include <cuda_bf16.h>

namespace lsms {
namespace tb {

constexpr int NP = 3;  // bf16 parts per value, weight classes per accumulator
constexpr long long kWaitLimit = 1ll << 24;           // bounded mbarrier wait: polls,
constexpr unsigned long long kWaitNs = 2000000000ull;  // and nanoseconds

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t phase);
// Wait for a phase, bounded in polls and in time (a poll may suspend the thread for long).
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t phase) {
  unsigned long long t0 = 0;
  for (long long q = 0; q < kWaitLimit; ++q) {
    if (mbar_try_wait(smem_u32(mbar), phase)) return true;
    if ((q & 63) == 63) {
      unsigned long long t;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
      if (t0 == 0) t0 = t;
      else if (t - t0 > kWaitNs) return false;
    }
  }
  return false;
}
// The same by a whole warp, with the same answer in every lane.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* mbar, uint32_t phase) {
  return __all_sync(0xffffffffu, mbar_wait(mbar, phase));
}

// K-major, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// kind::f16 with bf16 A and B: D f32, both K-major, N and M.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mbar)) : "memory");
}
// arrival when every product issued so far by this thread is complete
__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(mbar), "r"(phase)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {  // completed by tcgen05.wait::ld
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(taddr));
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// The three bf16 parts of two values as packed pairs; the remainders are exact in FP32.
__device__ __forceinline__ void split3(float x0, float x1, uint32_t (&p)[NP]) {
#pragma unroll
  for (int s = 0; s < NP; ++s) {
    p[s] = bf16_pair(x0, x1);
    if (s + 1 < NP) {
      x0 -= __uint_as_float(p[s] << 16);
      x1 -= __uint_as_float(p[s] & 0xffff0000u);
    }
  }
}

}  // namespace tb
}  // namespace lsms
