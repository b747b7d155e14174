// Inline-PTX helpers of the tensor-core kernels (sm_103a: tcgen05, mbarrier,
// bulk and tensor TMA) and the job decode of the trailing updates, shared by
// k_tc.cu and k_dz.cu.
#pragma once

#include <cuda.h>
#include <math.h>

#include "ahlp_internal.h"

namespace ahlp {

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
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
  const unsigned long long t0 = global_ns();
  while (!mbar_try(bar, parity))
    if (global_ns() - t0 > kWaitLimitNs) return false;
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
// second one only when has_i1) and the column tile J.  Inside a block with t
// trailing tiles, row pair R holds min(2R + 2, t) jobs, so the jobs before it
// number R(R + 1).
struct Job {
  int b, I0, J;
  bool has_i1;
};

// The update jobs of one pivot step, shared by every tensor-core update kernel.
// The jobs that hold the next step's diagonal tiles come first, and the kernel
// counts them off in `ready`, so that the next step's diagonal factorisations
// (a chain of 64 dependent pivots that keeps a few CTAs busy for 20 to 75 us) run
// beside the rest of this update instead of after it: they are the next kernel in
// the stream, may be scheduled as soon as every CTA here has started, and need an
// SM with room.  A persistent update takes a whole SM per CTA, so the last
// `short_ctas` CTAs stop after `full` rounds, some time before the others end.
struct StepJobs {
  const int *joff;      // [nblk + 1] prefix of (jobs - 1) over the blocks, then the number of
                        // blocks with jobs and those blocks
  const BlkInfo *blk;
  const int4 *jt;       // this step's tile-sparse job table, or nullptr
  int nblk, k, njobs;
  int full, short_ctas;
  int *ready;           // [nblk] arrivals on the next diagonal tiles, or nullptr
  const int *miss;      // blocks whose next diagonal tile this step does not touch
  int nmiss;
};

// number of jobs of this CTA, and its j-th job
__device__ __forceinline__ int my_jobs(const StepJobs &S) {
  const int i = blockIdx.x, G = gridDim.x, g = G - S.short_ctas;
  if (i >= g) return S.full;
  const int rest = S.njobs - S.full * G - i;
  return S.full + (rest > 0 ? (rest - 1) / g + 1 : 0);
}

__device__ __forceinline__ int job_index(const StepJobs &S, int j) {
  const int i = blockIdx.x, G = gridDim.x;
  return j < S.full ? i + j * G : S.full * G + i + (j - S.full) * (G - S.short_ctas);
}

__device__ __forceinline__ Job decode_job(const StepJobs &S, int q) {
  if (S.jt) {   // tile-sparse: the kept jobs of this step
    const int4 v = S.jt[q];
    Job j;
    j.b = v.x;
    j.I0 = v.y;
    j.J = v.z;
    j.has_i1 = v.w != 0;
    return j;
  }
  const int nact = S.joff[S.nblk + 1];
  int lo;
  long long local;
  if (q < nact) {   // a block's first job: the next diagonal tile
    lo = S.joff[S.nblk + 2 + q];
    local = 0;
  } else {
    q -= nact;
    lo = 0;
    int hi = S.nblk;   // joff[lo] <= q < joff[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (S.joff[mid] <= q) lo = mid;
      else hi = mid;
    }
    local = q - S.joff[lo] + 1;
  }
  const int t = S.blk[lo].T - S.k - 1;
  // largest R with R(R + 1) <= local: an FP32 estimate, corrected in integers
  // (an FP64 square root here costs every warp of every job ~25 instructions of
  // a pipe that issues one warp instruction in 64 clocks per partition)
  long long R = (long long)((sqrtf(4.0f * (float)local + 1.0f) - 1.0f) * 0.5f);
  while (R * (R + 1) > local) --R;
  while ((R + 1) * (R + 2) <= local) ++R;
  Job j;
  j.b = lo;
  j.I0 = S.k + 1 + 2 * (int)R;
  j.J = S.k + 1 + (int)(local - R * (R + 1));
  j.has_i1 = 2 * R + 1 < t;
  return j;
}

// does this job hold the next step's diagonal tile, and is someone waiting for it
__device__ __forceinline__ bool next_diag(const StepJobs &S, const Job &jb) {
  return S.ready && jb.J == S.k + 1 && jb.I0 == S.k + 1;
}

// after the kernel's griddepcontrol.wait: let the next kernel's CTAs be scheduled,
// and count off the tiles that have no job (`arrivals` per tile)
__device__ __forceinline__ void jobs_begin(const StepJobs &S, int arrivals) {
  if (!S.ready) return;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < S.nmiss; i += blockDim.x) {
      __threadfence();
      atomicExch(&S.ready[S.miss[i]], arrivals);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// jobs of step k and the grid of its update kernel (k_tc.cu)
StepJobs step_jobs(ahlp_problem *p, int k, bool persistent, int diag_jobs, int per_sm,
                   int arrivals, LookAhead *la, int *grid);

// the driver's tensor-map encoder, or nullptr
EncodeTiledFn tensor_map_encoder();

}  // namespace ahlp
