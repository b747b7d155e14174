// Tensor-core trailing update of the FP64 block factors (sm_103a: tcgen05,
// tensor memory, tensor TMA): exact integer-digit products, in the spirit of
// Ozaki's error-free splitting.
//
// The FP64 pipe of this part does two multiply-adds per clock and SM, so the
// update C_IJ -= L_Ik L_Jk' of the batched partial Cholesky, nearly all the
// flops of a factor, is bound by it: 162 ms of the 185 ms an FP64 factor of
// 32 uneven blocks (500..4000 rows) took with FP64 arithmetic.  Here the panel
// kernel writes every entry of a finished panel tile as eight signed 8-bit
// digits under one exponent per row,
//     x_rk = 2^E_r sum_s d_s 2^(-7-8s),  s = 0..7,  -128 <= d_s <= 127,
// E_r one more than the exponent of the row's largest entry (so |d_0| <= 64
// and entries are kept to 2^-63 of the row's scale), each digit an FP16
// integer.  With D_q = sum_{s+t=q} sum_k d_s(r,k) d_t(c,k),
//     sum_k x_rk y_ck = 2^(E_r+E_c-14) sum_q 2^(-8q) D_q.
// Over 64 pivot columns |D_q| <= (q + 1) 2^20 < 2^24, so the tensor core's
// FP32 accumulation of FP16 products is exact.  The 36 digit products with
// s + t <= 7 are kept.  The dropped ones sum to about 7 2^20 2^-78 = 2^-55 of
// 2^(E_r + E_c) at most, which is 2^-51 of the product of the rows' largest
// entries at worst (E is up to two above an entry's binary magnitude); digits of
// mixed signs leave about 2^-61 of the scales, below the roundings of 64 chained
// FP64 multiply-adds.  The epilogue adds the eight D_q in 64-bit integers, rounded
// to units of 2^-58 of the scales (12 bits less than the sum holds), turns the sum
// into an FP64 number by shifts (a second rounding) and subtracts it from C with
// one FP64 operation per entry (a third).
// All of it is relative to the rows' scales, where FP64 arithmetic rounds each
// product relative to itself.  The block factors meet the same normwise backward
// error bound, and as preconditioners they take the same Krylov steps up to 16
// decades of D.  Behind clamped pivots, whose rows grow by orders of magnitude,
// they are worse; solves that fail then move to the FP64 pipe (solve_on_pipe,
// ipm_solve's safeguards).
//
// One persistent CTA per SM walks the step's jobs (128 x 64 tiles of C, job
// blockIdx.x + j * gridDim.x):
//   warp 0     producer: the digit planes of 16 pivot columns (A: 8 planes of
//              128 rows, B: 8 planes of 64 rows, 48 KB) per ring stage, two
//              tensor TMA copies each, four stages;
//   warp 1     MMA issuer: digit s of A against digits 0..7-s of B stacked
//              along N, up to four digits (N = 256) per instruction, so one
//              read of A's digit from shared memory serves up to four
//              products; D_q accumulates in TMEM columns 64q..64q+63 (all
//              512 columns);
//   warps 2-17 epilogue: four warps per TMEM lane quarter, 16 columns each.
//              A warp requests its entries of C before the products are
//              ready, reads and combines the accumulators (which frees tensor
//              memory for the next job's MMAs), then converts and subtracts.
// A step of 7174 jobs (32 uneven blocks) takes 354 us: C's read and write need
// 124 us of the measured copy bandwidth, the MMAs about 110 us and the FP64
// subtractions 111 us of the FP64 pipe, and they overlap little, because a job's
// products fill tensor memory until its epilogue has read them (907 clocks per
// slice of eight MMAs issued, 7.3 k clocks of epilogue per job).  Two accumulator
// sets of half a tile with A resident measured 358 to 387 us: the narrower
// MMAs cost what the overlap gained.
// mbarrier parities: the n-th use of a stage or of the accumulators waits
// phase n & 1 of its "full" barrier and the (n-1)-th completion of its
// "empty" one.  Every wait is bounded (1 s); on expiry status[4] is set, the
// operations in flight are waited for and tensor memory is freed.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "ahlp_internal.h"
#include "tcgen05.h"

namespace ahlp {

namespace {

constexpr int kDzEpiWarps = 16;
constexpr int kDzThreads = 64 + 32 * kDzEpiWarps;
constexpr int kDzM = 128, kDzN = 64;
constexpr int kDzSliceK = 16;                                  // pivot columns per ring stage
constexpr uint32_t kDzPlane = NB * kDzSliceK * 2;              // a digit of 64 rows: 2 KB
constexpr uint32_t kDzPlaneA = 2 * kDzPlane;
constexpr uint32_t kDzStage = kDzQ * (kDzPlaneA + kDzPlane);   // 48 KB
constexpr int kDzStages = 4;
constexpr uint32_t kDzSmem = kDzStages * kDzStage + 1024;

// kind::f16 instruction descriptor: FP32 accumulator, FP16 A and B, both
// K-major, M = 128, N = n
__device__ __forceinline__ constexpr uint32_t dz_idesc(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kDzM >> 4) << 24);
}

__device__ __forceinline__ void dz_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc,
                                       uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tm, int x, int y,
                                            int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float (&v)[2]) {
  uint32_t r0, r1;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(taddr));
  v[0] = __uint_as_float(r0);
  v[1] = __uint_as_float(r1);
}

// sum_q D_q 2^(44-8q) as a 64-bit integer (the last 12 bits of the eight-digit
// sum rounded away).  |D_q| <= (q + 1) 2^20, |D_0| <= 2^18, so the pairs fit 32 bits.
__device__ __forceinline__ long long dz_combine(const float (&D)[kDzQ]) {
  const int a = (__float2int_rn(D[0]) << 8) + __float2int_rn(D[1]);
  const int b = (__float2int_rn(D[2]) << 8) + __float2int_rn(D[3]);
  const int c = (__float2int_rn(D[4]) << 8) + __float2int_rn(D[5]);
  const int e = (__float2int_rn(D[6]) << 8) + __float2int_rn(D[7]);
  return ((long long)a << 36) + ((long long)b << 20) + ((long long)c << 4) +
         ((e + (1 << 11)) >> 12);
}

// p 2^(sc - 58) as an FP64 number, rounded to nearest; values below the
// normal range become zero.  A row with a NaN or an infinity carries the
// exponent kDzNotFinite, and every product with it is a NaN.
__device__ __forceinline__ double dz_scale(long long p, int sc) {
  const unsigned long long u = p < 0 ? 0ull - (unsigned long long)p : (unsigned long long)p;
  const int lz = __clzll((long long)u);
  const unsigned long long v = u << (lz & 63);
  const int be = sc - 58 + 63 - lz + 1023;   // biased exponent
  unsigned long long bits =
      ((unsigned long long)(unsigned)(be - 1) << 52) + (v >> 11) + ((v >> 10) & 1ull);
  if (be > 2046) bits = 0x7ff0000000000000ull;
  if (u == 0 || be < 1) bits = 0;
  if (sc >= kDzNotFinite / 2) bits = 0x7ff8000000000000ull;
  bits |= (unsigned long long)p & 0x8000000000000000ull;
  return __longlong_as_double((long long)bits);
}

struct DzArgs {
  const int *dexp;         // per slot 64 row exponents
  double *buf;             // the augmented matrices
  int *status;
  StepJobs S;
};

__global__ void __launch_bounds__(kDzThreads, 1)
    pchol_update_dz_kernel(const DzArgs args, const __grid_constant__ CUtensorMap mapA,
                           const __grid_constant__ CUtensorMap mapB) {
  pdl_wait();
  jobs_begin(args.S, kDzEpiWarps);
  extern __shared__ __align__(1024) unsigned char dz_raw[];
  __shared__ __align__(8) uint64_t full[kDzStages], empty[kDzStages], tfull, tempty;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  unsigned char *base = dz_raw + ((1024 - (smem_u32(dz_raw) & 1023)) & 1023);
  volatile int *vfail = &s_fail;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int myjobs = my_jobs(args.S);
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int i = 0; i < kDzStages; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), 1);
    }
    mbar_init(smem_u32(&tfull), 1);
    mbar_init(smem_u32(&tempty), kDzEpiWarps * 32);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // ---- producer: 16 pivot columns of one job per unit ----------------------
    if (lane == 0) {
      int u = 0;   // units issued
      for (int j = 0; j < myjobs && !*vfail; ++j) {
        const Job jb = decode_job(args.S, job_index(args.S, j));
        const BlkInfo &bi = args.S.blk[jb.b];
        const int npiv = min(NB, bi.p - args.S.k * NB), soff = (int)bi.soff;
        const int ns = (npiv + kDzSliceK - 1) / kDzSliceK;
        bool ok = true;
        for (int sl = 0; sl < ns; ++sl, ++u) {
          const int st = u % kDzStages;
          if (!mbar_wait(smem_u32(&empty[st]), ((u / kDzStages) & 1) ^ 1)) {
            ok = false;
            break;
          }
          const uint32_t sa = smem_u32(base + st * kDzStage);
          const uint32_t bar = smem_u32(&full[st]);
          mbar_expect_tx(bar, kDzStage);   // rows past the slots are zero-filled and count
          tma_load_3d(sa, &mapA, 0, soff + jb.I0, sl * kDzQ, bar);
          tma_load_3d(sa + kDzQ * kDzPlaneA, &mapB, 0, soff + jb.J, sl * kDzQ, bar);
        }
        if (!ok) {
          atomicExch(&s_fail, 1);
          break;
        }
      }
      if (*vfail)   // copies still in flight land before exit
        for (int v = u >= kDzStages ? u - kDzStages : 0; v < u; ++v)
          mbar_wait(smem_u32(&full[v % kDzStages]), (v / kDzStages) & 1);
    }
  } else if (warp == 1) {
    // ---- MMA issuer -----------------------------------------------------------
    if (lane == 0) {
      int u = 0, last = -1;   // last unit whose MMAs were committed
      for (int j = 0; j < myjobs && !*vfail; ++j) {
        const Job jb = decode_job(args.S, job_index(args.S, j));
        const int npiv = min(NB, args.S.blk[jb.b].p - args.S.k * NB);
        const int ns = (npiv + kDzSliceK - 1) / kDzSliceK;
        if (!mbar_wait(smem_u32(&tempty), (j & 1) ^ 1)) {
          atomicExch(&s_fail, 2);
          break;
        }
        bool ok = true;
        for (int sl = 0; sl < ns; ++sl, ++u) {
          const int st = u % kDzStages;
          if (!mbar_wait(smem_u32(&full[st]), (u / kDzStages) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(base + st * kDzStage), sb = sa + kDzQ * kDzPlaneA;
#pragma unroll
          for (int s = 0; s < kDzQ; ++s) {
            const uint64_t da = smem_desc(sa + s * kDzPlaneA, 128, 256);
#pragma unroll
            for (int t = 0; t < kDzQ - s; t += 4) {   // digits t .. t + n - 1 of B
              const int n = kDzQ - s - t < 4 ? kDzQ - s - t : 4;
              dz_mma(tmem + (s + t) * kDzN, da, smem_desc(sb + t * kDzPlane, 128, 256),
                     dz_idesc(n * kDzN), (sl | s) != 0);
            }
          }
          mma_commit(smem_u32(&empty[st]));   // stage free once these MMAs complete
          last = u;
        }
        if (!ok) {
          atomicExch(&s_fail, 2);
          break;
        }
        mma_commit(smem_u32(&tfull));
      }
      if (*vfail && last >= 0)   // MMAs in flight finish before tensor memory is freed
        mbar_wait(smem_u32(&empty[last % kDzStages]), (last / kDzStages) & 1);
    }
  } else {
    // ---- epilogue -------------------------------------------------------------
    const int quarter = warp & 3;                  // TMEM lanes 32 quarter .. + 31
    const int cbase = ((warp - 2) >> 2) * 16;      // this warp's 16 columns of the tile
    const int r = quarter * 32 + lane;             // row of the 128-row tile
    const uint32_t tw = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)cbase;
    for (int j = 0; j < myjobs; ++j) {
      const Job jb = decode_job(args.S, job_index(args.S, j));
      const BlkInfo &bi = args.S.blk[jb.b];
      const int a = bi.a;
      const long long lda = bi.lda, slot0 = bi.soff + jb.I0, slotJ = bi.soff + jb.J;
      const int grow = jb.I0 * NB + r, col0 = jb.J * NB + cbase;
      // columns of this row on or below the diagonal (a row inside the matrix)
      const int nc = grow < a ? min(16, grow - col0 + 1) : 0;
      double *g = args.buf + bi.base + (long long)col0 * lda + grow;
      double c[16];
#pragma unroll
      for (int v = 0; v < 16; ++v) c[v] = v < nc ? g[v * lda] : 0.0;
      const int er = (r < NB || jb.has_i1) ? args.dexp[slot0 * NB + r] : 0;
      const int ec = args.dexp[slotJ * NB + cbase + (lane & 15)];   // lane v: column cbase + v
      int ok = 0;
      if (lane == 0) ok = mbar_wait(smem_u32(&tfull), j & 1) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) {
        atomicExch(&s_fail, 3);
        break;
      }
      tc_fence_after();
      long long P[16];
#pragma unroll
      for (int v = 0; v < 16; v += 2) {
        float D2[kDzQ][2];
#pragma unroll
        for (int q = 0; q < kDzQ; ++q) tmem_ld2(tw + (uint32_t)(q * kDzN + v), D2[q]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          float D[kDzQ];
#pragma unroll
          for (int q = 0; q < kDzQ; ++q) D[q] = D2[q][w];
          P[v + w] = dz_combine(D);
        }
      }
      // accumulators read: the next job's MMAs may overwrite them
      tc_fence_before();
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty))
                   : "memory");
#pragma unroll
      for (int v = 0; v < 16; ++v) {
        const int sc = er + __shfl_sync(0xffffffffu, ec, v);
        if (v < nc) g[v * lda] = c[v] - dz_scale(P[v], sc);
      }
      if (next_diag(args.S, jb)) {
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(&args.S.ready[jb.b], 1);
      }
    }
  }
  __syncwarp();
  if (threadIdx.x == 0 && *vfail) atomicExch(&args.status[4], 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                 : "memory");
}

}  // namespace

// Digit staging (plane p of K slice sl of every slot: 2 KB at
// ((sl * kDzQ + p) * slots + slot)), job offsets and the two tensor maps over
// the staging.  False when the driver has no tensor-map encoder, or when the
// device has no room for the staging (64 KB per 64 rows): the FP64 pipe's
// updates need none.  Nothing is kept then, and the next factor tries again.
bool dz_setup(ahlp_problem *p) {
  if (p->dz_stage) return true;
  const EncodeTiledFn encode = tensor_map_encoder();
  if (!encode) return false;
  try {
    jobs_setup(p);
    AllocScope mem(p);
    const long long slots = std::max(p->stage_slots, 1LL);
    constexpr int planes = kDzQ * NB / kDzSliceK;
    __half *stage = static_cast<__half *>(dalloc_bytes(p, (size_t)slots * planes * kDzPlane));
    int *exps = static_cast<int *>(dalloc_bytes(p, (size_t)slots * NB * sizeof(int)));
    static_assert(sizeof(p->dz_map) == 2 * sizeof(CUtensorMap), "tensor map size");
    for (int w = 0; w < 2; ++w) {
      const cuuint64_t dims[3] = {kDzPlane / 8, (cuuint64_t)slots, (cuuint64_t)planes};
      const cuuint64_t strides[2] = {kDzPlane, (cuuint64_t)slots * kDzPlane};
      const cuuint32_t box[3] = {kDzPlane / 8, w == 0 ? 2u : 1u, (cuuint32_t)kDzQ};
      const cuuint32_t estr[3] = {1, 1, 1};
      CUtensorMap m;
      if (encode(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3, stage, dims, strides, box, estr,
                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
      memcpy(p->dz_map[w], &m, sizeof m);
    }
    ck(cudaFuncSetAttribute(pchol_update_dz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                            (int)kDzSmem),
       "FP64 tensor-core update shared memory");
    p->dz_exp = exps;
    p->dz_stage = stage;
    mem.keep = true;
    return true;
  } catch (const Fail &f) {
    if (f.code != AHLP_ERR_OOM) throw;
    return false;
  }
}

cudaError_t launch_update_dz(ahlp_problem *p, int k, cudaStream_t s, LookAhead *la) {
  if (p->tc_jobs[k] <= 0) return cudaSuccess;
  int grid = 0;
  DzArgs a{p->dz_exp, p->aug, p->status, StepJobs{}};
  a.S = step_jobs(p, k, true, 13, 1, kDzEpiWarps, la, &grid);
  CUtensorMap mA, mB;
  memcpy(&mA, p->dz_map[0], sizeof mA);
  memcpy(&mB, p->dz_map[1], sizeof mB);
  count_launch(), launch_pdl(pchol_update_dz_kernel, grid, kDzThreads, kDzSmem, s, a, mA, mB);
  return cudaGetLastError();
}

}  // namespace ahlp
