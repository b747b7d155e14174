// Inline-PTX helpers of the tensor-core kernels (sm_103a: tcgen05, mbarrier,
// bulk and tensor TMA) and the job decode of the trailing updates, shared by
// k_tc.cu and k_dz.cu.
#pragma once

#include <cuda.h>
#include <math.h>

#include "ahlp_internal.h"

namespace ahlp {

constexpr unsigned long long kWaitNs = 1000000000ull;   // 1 s


__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long globaltimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait for phase `parity` of the barrier; false when it ran out.  The
// timer is read only after some failed tries: most waits end at once, and one
// timer read per wait would sit between consecutive MMAs.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
#pragma unroll 1
  for (int i = 0; i < 16; ++i)
    if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  while (!mbar_try(bar, parity))
    if (globaltimer() - t0 > kWaitNs) return false;
  return true;
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes,
                                         uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor of a K-major operand without swizzling:
// 8-row x 16-byte core matrices, LBO = byte distance between core matrices
// adjacent in K, SBO = byte distance between adjacent 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version of the tcgen05 family
  return d;                 // base offset 0, absolute LBO, no swizzle
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::
                   "r"(bar)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// One update job of step k: block b, the row tile pair (I0, I0 + 1) (the
// second one only when has_i1) and the column tile J.  The jobs of a step are
// numbered block after block (joff: prefix over the blocks); inside a block
// with t trailing tiles, row pair R holds min(2R + 2, t) jobs, so the jobs
// before it number R(R + 1).
struct Job {
  int b, I0, J;
  bool has_i1;
};

__device__ __forceinline__ Job decode_job(const int *joff, int nblk, int k, const BlkInfo *blk,
                                          int q, const int4 *jt) {
  if (jt) {   // tile-sparse: the kept jobs of this step, in the dense order
    const int4 v = jt[q];
    Job j;
    j.b = v.x;
    j.I0 = v.y;
    j.J = v.z;
    j.has_i1 = v.w != 0;
    return j;
  }
  int lo = 0, hi = nblk;   // joff[lo] <= q < joff[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (joff[mid] <= q) lo = mid;
    else hi = mid;
  }
  const int t = blk[lo].T - k - 1;
  // largest R with R(R + 1) <= local: an FP32 estimate, corrected in integers
  // (an FP64 square root here costs every warp of every job ~25 instructions of
  // a pipe that issues one warp instruction in 64 clocks per partition)
  const long long local = q - joff[lo];
  long long R = (long long)((sqrtf(4.0f * (float)local + 1.0f) - 1.0f) * 0.5f);
  while (R * (R + 1) > local) --R;
  while ((R + 1) * (R + 2) <= local) ++R;
  Job j;
  j.b = lo;
  j.I0 = k + 1 + 2 * (int)R;
  j.J = k + 1 + (int)(local - R * (R + 1));
  j.has_i1 = 2 * R + 1 < t;
  return j;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// the driver's tensor-map encoder, or nullptr
EncodeTiledFn tensor_map_encoder();

}  // namespace ahlp
