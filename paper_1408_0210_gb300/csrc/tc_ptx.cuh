// tc_ptx.cuh -- the mbarrier, bulk-copy and tcgen05 instructions that the
// tensor-core kernels share, and their bounded waits.
#pragma once
#include <cuda.h>

#include "internal.h"

namespace eifmm {

constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t a, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(a), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try(uint32_t a, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(a), "r"(parity)
      : "memory");
  return ok;
}
// Bounded wait; returns false (and records `code`) after `limit` cycles.
__device__ __forceinline__ bool mbar_wait_lim(uint32_t a, uint32_t parity, int* err, int code, long long limit) {
  const long long t0 = clock64();
  while (!mbar_try(a, parity)) {
    if (clock64() - t0 > limit) {
      atomicExch(err, code);
      return false;
    }
  }
  return true;
}
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, int* err, int code) {
  return mbar_wait_lim(a, parity, err, code, kWaitCycles);
}

// The producer's last act: every copy it issued has landed (each stage's
// last fill completed its phase) before the CTA may exit, also after an
// abort.  it = fills issued so far, ring of `stages`.  Bounded like every
// wait.
__device__ __forceinline__ void drain_fills(int it, int stages, const uint64_t* bars_full, int* err) {
  for (int k = 0; k < stages && k < it; ++k) {
    const int i = it - 1 - k;  // a recent fill
    mbar_wait(smem_u32(&bars_full[i % stages]), (uint32_t)((i / stages) & 1), err, 5);
  }
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            int c3, int c4, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(mbar)
      : "memory");
}

// Bounded wait that also gives up when another role has set *abort.
__device__ __forceinline__ bool mbar_wait_ab(uint32_t a, uint32_t parity, int* err, int code,
                                             volatile int* abort) {
  if (mbar_try(a, parity)) return true;  // the clock is read only when it has to wait
  const long long t0 = clock64();
  while (!mbar_try(a, parity)) {
    if (*abort) return false;
    if (clock64() - t0 > kWaitCycles) {
      atomicExch(err, code);
      *abort = 1;
      return false;
    }
  }
  return true;
}

// As mbar_wait_ab for a converged warp, with a vote on every branch, so that the
// control flow stays uniform for the compiler too: after a wait whose lanes
// might part, MMAs and commits are issued as by a diverged thread.  The residue GEMM
// at d = 193: 98 cycles per MMA and 263 per step before, 109 (the tensor rate) and
// 147 with it; M2L of 2^20 points 5.70 -> 5.13 ms, at d = 126 3.86 -> 3.30.  The
// FP32 tiers' kernels, whose steps are three times as long, gain nothing from it.
__device__ __forceinline__ bool mbar_wait_u(uint32_t a, uint32_t parity, int* err, int code,
                                            volatile int* abort) {
  if (__all_sync(0xffffffffu, mbar_try(a, parity))) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, mbar_try(a, parity))) {
    const bool late = clock64() - t0 > kWaitCycles;
    if (__any_sync(0xffffffffu, late || *abort)) {
      if (late) {
        atomicExch(err, code);
        *abort = 1;
      }
      return false;
    }
  }
  return true;
}

// Issue from a converged warp: one lane is elected once and only its
// instructions take effect.  The operands then stay in uniform registers: a
// loop that a single thread of a diverged warp runs needs about 100 cycles per
// MMA and 300 for a wait and a commit, this form 27 and 60, so that M = 128,
// N = 128 (64 cycles of the tensor pipe) runs at full rate.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p;
}
__device__ __forceinline__ void mma_commit_el(uint32_t mbar, uint32_t el) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(mbar),
      "r"(el)
      : "memory");
}
// kind::f16; the descriptors as their low and high words
__device__ __forceinline__ void mma_f16_el(uint32_t tmem, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                           uint32_t id, uint32_t acc, uint32_t el) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 a, b;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
      " setp.ne.b32 p, %6, 0;\n setp.ne.b32 q, %7, 0;\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(tmem),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(id), "r"(acc), "r"(el));
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn();  // cuTensorMapEncodeTiled of the loaded driver (m2l_tc.cu); null if absent

}  // namespace eifmm
