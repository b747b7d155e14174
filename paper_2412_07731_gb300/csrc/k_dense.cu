// Dense per-block kernels: formation of the augmented matrices, the batched
// tiled partial Cholesky, and the forward / backward solves with its factor.
//
// Every block i owns an augmented lower-triangular matrix
//     [ M_i   .  ]        M_i = A_i D_i A_i' + delta I      (m_i x m_i)
//     [ G_i'  C_i]        G_i = [W_i | A_i D_i U_i' | A_i D_i Fg_i']
// stored column-major.  Eliminating its first m_i pivots (the block factor and
// Schur-contribution steps of Alg. 2 in normal-equation form) leaves L_i on
// top, Y_i' = (L_i^-1 G_i)' below it and C_i - G_i' M_i^-1 G_i in the corner
// -- the block's Schur contribution.
//
// The factor is stored in FP64, FP32 or float-float (two FP32 words); in the
// mixed modes it only preconditions an FP64 Krylov solve.  Kernels shared by
// FP64 and FP32 are templated on the storage type; the FP32 and float-float
// trailing updates and the FP32 diagonal tile have their own kernels.
// Entries are always formed in FP64 and rounded once.
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>

#include "ahlp_internal.h"
#include "publish.h"

namespace ahlp {

namespace {

// --------------------------------------------------------------------------
// formation: one CTA per 64x64 lower tile, written exactly once
// --------------------------------------------------------------------------
template <typename T>
struct FormArgs {
  float *lo;   // float-float: receives v - (double)(float)v (nullptr otherwise)
  const FormTile *tiles;
  const long long *tile_ent;
  const int *ent_pos;
  const long long *ent_cb;
  const int *con_idx;
  const double *con_coef;
  const double *d;
  const BlkInfo *blk;
  T *aug;
  double *diag0;
  double *cdiag0;
  double delta;
};

template <typename T, bool kLo>
__global__ void __launch_bounds__(kThreads) form_aug_kernel(FormArgs<T> A) {
  pdl_begin();
  __shared__ T t[NB * NB];   // column-major tile
  __shared__ float tl[kLo ? NB * NB : 1];
  const FormTile ft = A.tiles[blockIdx.x];
  const BlkInfo bi = A.blk[ft.blk];
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    t[i] = T(0);
    if constexpr (kLo) tl[i] = 0.0f;
  }
  __syncthreads();
  const long long e0 = A.tile_ent[blockIdx.x], e1 = A.tile_ent[blockIdx.x + 1];
  for (long long e = e0 + threadIdx.x; e < e1; e += blockDim.x) {
    const int pos = A.ent_pos[e];
    const long long q0 = A.ent_cb[e], q1 = A.ent_cb[e + 1];
    double v = 0.0;
    for (long long q = q0; q < q1; ++q) {
      const int di = A.con_idx[q];
      const double cf = A.con_coef[q];
      v += (di >= 0) ? cf * A.d[di] : cf;
    }
    const int rt = (pos >> 8) & 0xff, ct = pos & 0xff;
    if (pos & (1 << 16)) {   // diagonal of M_i: regularise, remember for pivot test
      v += A.delta;
      A.diag0[bi.d0off + (long long)ft.I * NB + rt] = v;
    } else if (pos & (1 << 17)) {   // corner diagonal: reference for link / y_g pivots
      A.cdiag0[bi.cdoff + (long long)ft.I * NB + rt - bi.p] = v;
    }
    t[ct * NB + rt] = T(v);
    if constexpr (kLo) tl[ct * NB + rt] = (float)(v - (double)(float)v);
  }
  __syncthreads();
  const int r0 = ft.I * NB, c0 = ft.J * NB;
  const int nr = min(NB, bi.a - r0), nc = min(NB, bi.a - c0);
  const long long g0 = bi.base + (long long)c0 * bi.lda + r0;
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    const int r = i % NB, c = i / NB;
    if (r < nr && c < nc) {
      A.aug[g0 + (long long)c * bi.lda + r] = t[i];
      if constexpr (kLo) A.lo[g0 + (long long)c * bi.lda + r] = tl[i];
    }
  }
}

// d = x / z; on the block variables x / (z + rho_x x) with the factor's primal
// regularisation, i.e. D^-1 + rho_x (caps d at 1 / rho_x).  The linking
// variables get theirs in the Schur border (-D_0^-1 - rho).  With them, the
// two per-variable quotients every solve at this point needs (FP64 division
// is a long instruction sequence on this part): xinv = 1 / x and
// w = 1 / (1 / d + rho on the linking variables).
// It also clears the factor's status words, the corner diagonals and the counts of
// updated diagonal tiles.
__global__ void dscale_kernel(const double *x, const double *z, double *d, double *xinv,
                              double *w, long long n, double rho_x, double rho,
                              const unsigned char *is_x0, int *status, double *cdiag0,
                              long long ncd, int *ready, long long nready) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 8) status[i] = 0;
  for (long long q = i; q < ncd; q += (long long)gridDim.x * blockDim.x) cdiag0[q] = 0.0;
  for (long long q = i; q < nready; q += (long long)gridDim.x * blockDim.x) ready[q] = 0;
  if (i >= n) return;
  const double di = (rho_x > 0.0 && !is_x0[i]) ? x[i] / (z[i] + rho_x * x[i]) : x[i] / z[i];
  d[i] = di;
  xinv[i] = 1.0 / x[i];
  w[i] = 1.0 / (1.0 / di + (is_x0[i] ? rho : 0.0));
}

// --------------------------------------------------------------------------
// partial Cholesky, step k: diagonal tile
// --------------------------------------------------------------------------
// FP64 and float-float diagonal tiles.  The FP64 pipe takes one warp instruction
// per 64 clocks and partition (76 with all four busy), comparisons and
// conversions included, so the tile is bound by the FP64 instructions on its
// chain of 64 pivots, not by bandwidth.  Four 16-column panels; a panel is
// factored in registers by four warps, one per partition: every warp holds its
// own copy of the 16 x 16 diagonal block and 16 rows below it (lane = row and
// column parity, eight entries each), so no column waits for another warp.  A
// pivot costs its test in integers, one reciprocal square root (five FP64
// instructions), two scalings and the updates; the diagonal entries themselves
// follow at the end, all at once.  Then all eight warps apply the panel to the
// lower triangle right of it, lanes packed over the triangle.  51 us per tile on
// one CTA (76 us with FP64 pivot tests and the diagonal on the chain, 124 us with
// a barrier, a square root and a division per column).
// 1 / sqrt(p) of a positive finite p: y0 = rsqrtf of the mantissa (p scaled
// by an even power of two into [1, 4)), then Householder's third-order
// iteration y = y0 + y0 e (1/2 + 3/8 e), e = 1 - m y0^2, whose error is ~e^3.
__device__ __forceinline__ double rsqrt_f64(double p) {
  const int hi = __double2hiint(p);
  const int ex = hi >> 20;
  if (ex == 0 || ex >= 0x7ff) return rsqrt(p);   // subnormal or infinite
  const int k = (ex - 1023) >> 1;
  const int mh = hi - (k << 21), ml = __double2loint(p);
  const double m = __hiloint2double(mh, ml);   // [1, 4)
  // FP32 value of m from its bits (truncated), and y0's bits as FP64 (y0 in (1/2, 1])
  const float y = rsqrtf(__int_as_float(((mh - 0x38000000) << 3) | (int)((unsigned)ml >> 29)));
  const int yb = __float_as_int(y);
  const double y0 = __hiloint2double((yb >> 3) + 0x38000000, yb << 29);
  const double e = fma(-m * y0, y0, 1.0);
  const double r = fma(y0 * e, fma(0.375, e, 0.5), y0);
  return __hiloint2double(__double2hiint(r) - (k << 20), __double2loint(r));
}

constexpr int kPW = 16;   // panel width

// Start and end of a diagonal factorisation.  With la.ready the kernel runs beside
// the update of the step before: it was launched as that update's programmatic
// dependent, so the update's CTAs have all started (they never wait for this
// kernel, and everything before them is complete), a block waits for its own tile
// only, and the whole update is waited for at the end, on behalf of the panel
// kernel behind.  The wait is bounded (1 s), then status[4] is set.
__device__ __forceinline__ bool diag_begin(const LookAhead &la, bool active, int *status) {
  if (!la.ready || !active) {
    pdl_begin();
    return active;
  }
  if (threadIdx.x == 0) {
    const int *f = la.ready + blockIdx.x;
    const unsigned long long t0 = global_ns();
    for (int it = 0; load_relaxed(f) < la.target; ++it) {
      __nanosleep(100);
      if ((it & 31) == 31 && global_ns() - t0 > kWaitLimitNs) {
        atomicExch(&status[4], 1);
        break;
      }
    }
    __threadfence();   // the tile's writes, ordered before the count, are visible
  }
  __syncthreads();
  return true;
}

__device__ __forceinline__ void diag_end(const LookAhead &la) {
  if (la.ready) pdl_begin();
}

// Unused shared memory of an FP64 or float-float diagonal tile beside an update:
// at most two per SM, since they share its FP64 pipe (three: 28.4 against 27.7 ms
// per FP64 factor and solve of 32 uneven blocks).
constexpr int kDiagPad = 60000;

// kFF: the matrix is hi + lo (lo null otherwise)
template <bool kFF, typename T>
__global__ void __launch_bounds__(kThreads) pchol_potrf_kernel(T *buf, float *lo,
                                                               const BlkInfo *blk, int k,
                                                               const double *diag0, double tol,
                                                               int *status, double drop,
                                                               const LookAhead la) {
  const BlkInfo bi = blk[blockIdx.x];
  if (!diag_begin(la, k < bi.Tp, status)) return;
  __shared__ double t[NB][NB + 1];
  __shared__ double s_piv[NB], s_inv[NB];
  const int r0 = k * NB;
  const int nr = min(NB, bi.a - r0);
  const int npiv = min(NB, bi.p - r0);
  const long long g0 = bi.base + (long long)r0 * bi.lda + r0;
  {
    const int r = threadIdx.x & (NB - 1), cs = threadIdx.x / NB;
#pragma unroll 8
    for (int c = cs; c < NB; c += kThreads / NB) {
      double v = 0.0;
      if (r < nr && c < nr && r >= c) {
        const long long el = g0 + (long long)c * bi.lda + r;
        if constexpr (kFF) v = (double)buf[el] + (double)lo[el];
        else v = buf[el];
      }
      t[r][c] = v;
    }
  }
  __syncthreads();
  const double cap = kFF ? kDropCapFF : 1e300;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rr = lane & 15, hc = lane >> 4;   // row of 16, column parity
  for (int c0 = 0; c0 < npiv; c0 += kPW) {
    if (warp < 4) {
      const int row = warp * 16 + rr;       // this warp's own rows
      const bool own = warp * 16 > c0;      // below the diagonal block
      double d[8], o[8];                    // columns c0 + 2j + hc
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        d[j] = t[c0 + rr][c0 + 2 * j + hc];
        o[j] = own ? t[row][c0 + 2 * j + hc] : 0.0;
      }
      const double dref = c0 + rr < npiv ? diag0[bi.d0off + r0 + c0 + rr] : 0.0;
      // the pivot must exceed lim: positive doubles compare as their bits
      const double lim = tol * dref;
      const long long limb = max(__double_as_longlong(lim), 0ll);
#pragma unroll
      for (int u = 0; u < kPW; ++u) {
        if (c0 + u < npiv) {   // uniform over the CTA
          const int src = (u & 1) * 16;
          double piv = __shfl_sync(0xffffffffu, d[u >> 1], src + u);
          const long long lb = __shfl_sync(0xffffffffu, limb, u);
          const double v = __shfl_sync(0xffffffffu, d[u >> 1], src + rr);
          const double vo = __shfl_sync(0xffffffffu, o[u >> 1], src + rr);
          const long long pb = __double_as_longlong(piv);
          if (pb <= lb || pb > 0x7ff0000000000000ll) {   // too small, negative or NaN
            const double orig = __shfl_sync(0xffffffffu, dref, u);
            if (threadIdx.x == 0) {
              double q = piv;
              pivot_fix(q, orig, tol, status, bi.tag + (int)blockIdx.x, r0 + c0 + u, drop, cap);
            }
            const double lm = tol * orig;
            piv = drop > 0.0 ? fmin(drop * fmax(orig, 1.0), cap) : lm > 0.0 ? lm : 1.0;
          }
          const double inv = rsqrt_f64(piv);
          if (threadIdx.x == 0) {
            s_piv[c0 + u] = piv;
            s_inv[c0 + u] = inv;
          }
          const double ld = v * inv;   // rows u + 1 .. (the diagonal entry comes later)
          if (hc == (u & 1)) d[u >> 1] = ld;
          double lor = 0.0;
          if (own) {   // uniform over the warp
            lor = vo * inv;
            if (hc == (u & 1)) o[u >> 1] = lor;
          }
#pragma unroll
          for (int j = u >> 1; j < 8; ++j) {   // columns q = 2j + hc > u
            const double lq = __shfl_sync(0xffffffffu, ld, 2 * j + hc);
            if (2 * j + hc > u) {
              d[j] = fma(-ld, lq, d[j]);
              if (own) o[j] = fma(-lor, lq, o[j]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int q = 2 * j + hc;
        if (warp == 0 && q <= rr) t[c0 + rr][c0 + q] = d[j];
        if (own) t[row][c0 + q] = o[j];
      }
    }
    __syncthreads();
    // rank-16 update of the lower triangle right of the panel
    const int q0 = c0 + kPW, cend = min(q0, npiv);
    if (q0 < nr) {
      const int w = nr - q0, ne = w * (w + 1) / 2;
      for (int idx = threadIdx.x; idx < ne; idx += blockDim.x) {
        int ri = (int)((sqrtf(8.0f * (float)idx + 1.0f) - 1.0f) * 0.5f);
        while (ri * (ri + 1) / 2 > idx) --ri;
        while ((ri + 1) * (ri + 2) / 2 <= idx) ++ri;
        const int r = q0 + ri, q = q0 + idx - ri * (ri + 1) / 2;
        double s0 = t[r][q], s1 = 0.0;
        int c = c0;
        for (; c + 1 < cend; c += 2) {
          s0 = fma(-t[r][c], t[q][c], s0);
          s1 = fma(-t[r][c + 1], t[q][c + 1], s1);
        }
        if (c < cend) s0 = fma(-t[r][c], t[q][c], s0);
        t[r][q] = s0 + s1;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x < npiv) {   // sqrt(piv) = piv inv, one correction; an infinite pivot stays
    const double piv = s_piv[threadIdx.x], inv = s_inv[threadIdx.x];
    const double l = piv * inv;
    t[threadIdx.x][threadIdx.x] = isinf(piv) ? piv : fma(fma(-l, l, piv), 0.5 * inv, l);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    const int r = i % NB, c = i / NB;
    if (r < nr && c < nr && r >= c) {
      const long long el = g0 + (long long)c * bi.lda + r;
      if constexpr (kFF) {
        const float h = (float)t[r][c];
        buf[el] = h;
        lo[el] = (float)(t[r][c] - (double)h);
      } else {
        buf[el] = t[r][c];
      }
    }
  }
  diag_end(la);
}

// One 64 x 64 FP64 panel tile as eight FP16 digit planes for the tensor-core
// update (k_dz.cu): row r's exponent E_r is one more than its largest entry's,
// v = round(x 2^(63 - E_r)) is a 64-bit integer below 2^62, and the bytes of
// v + 0x8080...80 less 128 are its balanced digits, most significant first.
// Plane p of the K slice of columns 16 sl .. 16 sl + 15 is a 64 x 16 K-major
// operand of 8-row x 16-byte core matrices, 2 KB at ((8 sl + p) * slots +
// slot): entry (r, c) at (r/8)*128 + ((c%16)/8)*64 + (r%8)*8 + c%8.  Rows past
// the matrix and columns past the pivots are zero.  Rows row0 .. row0 + nrow - 1,
// thread (row row0 + tid / 4, slice tid % 4); x(r, c) returns the entry.  A row
// holding a NaN or an infinity gets the exponent kDzNotFinite and no digits.
template <typename F>
__device__ __forceinline__ void dz_stage_rows(F x, int row0, int nrow, int nri, int npiv,
                                              __half *stage, int *dexp, long long slots,
                                              long long slot) {
  const int r = row0 + (threadIdx.x >> 2), sl = threadIdx.x & 3, c0 = sl * 16;
  const bool mine = r < row0 + nrow;
  const bool row = mine && r < nri;
  int mx = 0;   // largest high word (exponent and leading bits); 1 for a tiny nonzero
#pragma unroll
  for (int j = 0; j < 16; ++j)
    if (row && c0 + j < npiv) {
      const double xv = x(r, c0 + j);
      mx = max(mx, max(__double2hiint(xv) & 0x7fffffff, __double2loint(xv) ? 1 : 0));
    }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  const bool fin = mx < 0x7ff00000;
  const int E = mx ? (mx >> 20) - 1021 : 0;   // |x| < 2^(E - 1); a zero row takes 0
  if (mine && sl == 0) dexp[slot * NB + r] = fin ? E : kDzNotFinite;
  __half *st = stage + ((long long)(sl * kDzQ) * slots + slot) * 1024 + (r >> 3) * 128 + (r & 7) * 8;
#pragma unroll
  for (int h = 0; h < 2; ++h) {   // 8 columns: one 16-byte run per plane
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = c0 + h * 8 + j;
      unsigned long long v = 0;
      if (row && fin && c < npiv) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x(r, c));
        const int be = (int)(b >> 52) & 0x7ff;
        unsigned long long m = b & 0xfffffffffffffull;
        if (be) m |= 1ull << 52;
        // x = m 2^(max(be, 1) - 1075), so v = m 2^(max(be, 1) - 1012 - E)
        const int sh = max(be, 1) - 1012 - E;   // at most 9
        if (sh >= 0) m <<= sh;
        else if (sh > -64) m = (m + (1ull << (-sh - 1))) >> -sh;
        else m = 0;
        v = (b >> 63) ? 0ull - m : m;
      }
      v += 0x8080808080808080ull;
      lo[j] = (uint32_t)v;
      hi[j] = (uint32_t)(v >> 32);
    }
#pragma unroll
    for (int p = 0; p < kDzQ; ++p) {
      const int byte = 3 - (p & 3);
      const uint32_t sel = (uint32_t)(byte | ((byte + 4) << 4));   // that byte of both words
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t a = p < 4 ? hi[2 * q] : lo[2 * q], b = p < 4 ? hi[2 * q + 1] : lo[2 * q + 1];
        // halves 1024 + byte, less 1152
        const uint32_t y = __byte_perm(__byte_perm(a, b, sel), 0x64646464u, 0x4140);
        const __half2 f = __hsub2(*reinterpret_cast<const __half2 *>(&y),
                                  __floats2half2_rn(1152.0f, 1152.0f));
        w[q] = *reinterpret_cast<const uint32_t *>(&f);
      }
      if (mine)
        *reinterpret_cast<uint4 *>(st + (long long)p * slots * 1024 + h * 64) =
            make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// panel tiles below the diagonal tile: X = A_Ik L_kk^-T on the pivot columns,
// and the non-pivot (Schur) columns of the tile updated with the new X.  With
// stage (FP64 factors, tensor-core update) the tile's digits are written too.
//
// Bound by the FP64 pipe: 64^3 / 2 multiply-adds per tile, 34 us of one SM.  So the
// inner loop is nothing but those: a row lives in the registers of G lanes (column
// 4j + g in register j of lane group g, for G = 4), the owner of column c scales
// it, a shuffle hands it to the row's other lanes, and each lane subtracts it from
// its columns right of c, with L_sc broadcast from shared memory; no barrier and no
// shared-memory store.  Every entry's operations and their order are those of
// the plain right-looking loop.  Lanes idle at the diagonal cost 8 % (G = 2), 17 %
// (4) and 35 % (8) more instructions, but a warp's 32 / G rows finish in 37, 20 and
// 12 us, so G grows as the tiles get fewer than the SMs' partitions (trsm_lanes).
constexpr int kTrsmThreads = 128;
constexpr size_t kTrsmSmem = NB * (NB + 1) * sizeof(double);
template <int G>
__global__ void __launch_bounds__(kTrsmThreads, G == 2 ? 3 : 4)
    pchol_trsm_kernel(double *buf, const BlkInfo *blk, int k, __half *stage, int *dexp,
                      long long slots) {
  pdl_begin();
  constexpr int R = 32 / G, kRows = kTrsmThreads / G, kC = NB / G;
  const BlkInfo bi = blk[blockIdx.y];
  if (k >= bi.Tp) return;
  const int I = k + 1 + blockIdx.x / (NB / kRows), row0 = (blockIdx.x % (NB / kRows)) * kRows;
  if (I >= bi.T) return;
  extern __shared__ __align__(16) unsigned char trsm_raw[];
  double *L = reinterpret_cast<double *>(trsm_raw);   // column c at c * NB
  __shared__ double rinv[NB];
  const int r0 = k * NB;
  const int nr = min(NB, bi.a - r0);
  const int npiv = min(NB, bi.p - r0);
  const int ri = I * NB;
  const int nri = min(NB, bi.a - ri);
  const double *gl = buf + bi.base + (long long)r0 * bi.lda + r0;
  double *gx = buf + bi.base + (long long)r0 * bi.lda + ri;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rl = lane % R, g = lane / R, row = row0 + warp * R + rl;
  double x[kC];   // columns G j + g of the row
#pragma unroll
  for (int j = 0; j < kC; ++j) {
    const int s = G * j + g;
    x[j] = (row < nri && s < nr) ? gx[(long long)s * bi.lda + row] : 0.0;
  }
#pragma unroll 8
  for (int i = threadIdx.x; i < NB * NB; i += kTrsmThreads) {
    const int r = i % NB, c = i / NB;
    L[i] = (r < nr && c < nr && r >= c) ? gl[(long long)c * bi.lda + r] : 0.0;
  }
  __syncthreads();
  // one reciprocal per column
  if (threadIdx.x < npiv) rinv[threadIdx.x] = 1.0 / L[threadIdx.x * (NB + 1)];
  __syncthreads();
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    if (c < npiv) {   // uniform
      const int jc = c / G, gc = c % G;
      const double v = x[jc] * rinv[c];
      const double xc = __shfl_sync(0xffffffffu, v, gc * R + rl);
      const double *Lc = L + c * NB + g;
      if (gc < G - 1) {
        const double u = fma(-xc, Lc[G * jc], x[jc]);
        x[jc] = g > gc ? u : g == gc ? v : x[jc];
      } else if (g == gc) {
        x[jc] = v;
      }
#pragma unroll
      for (int j = jc + 1; j < kC; ++j) x[j] = fma(-xc, Lc[G * j], x[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < kC; ++j) {
    const int s = G * j + g;
    if (row < nri && s < nr) gx[(long long)s * bi.lda + row] = x[j];
  }
  if (stage) {   // through shared memory, over L
    __syncthreads();
    double(*X)[NB + 1] = reinterpret_cast<double(*)[NB + 1]>(trsm_raw);
#pragma unroll
    for (int j = 0; j < kC; ++j) X[warp * R + rl][G * j + g] = x[j];
    __syncthreads();
    for (int h = 0; h < kRows; h += 32)
      dz_stage_rows([&](int r, int c) { return X[r - row0][c]; }, row0 + h, min(32, kRows), nri,
                    npiv, stage, dexp, slots, bi.soff + I);
  }
}

// lane groups per row: as many as keep every warp of the step's tiles (2 G per
// tile) on a partition of its own.  One tile: 70 us with a column's updates spread
// over a CTA between two barriers.
constexpr int kSMs = 152;   // chooses layouts of the same arithmetic, nothing else
inline int trsm_lanes(long long tiles) {
  return tiles * 16 <= 4 * kSMs ? 8 : tiles * 8 <= 4 * kSMs ? 4 : 2;
}

// --------------------------------------------------------------------------
// FP32 factors: diagonal tile, then the inverse of its pivot triangle,
// written in the layout the block solves use (inverse on the pivot rows, the
// factor on the non-pivot rows of a block's last pivot tile).  The panel
// below then is a product with that inverse instead of a column-by-column
// substitution.
//
// The 64x64 tile sits in shared memory and is factored in four 16-column
// panels.  Warp 0 factors a panel in registers: lane l holds rows l and
// l + 32 of the panel's 16 columns, the pivot and the scaled column entries
// are broadcast with shuffles, so the sequential path has no shared-memory
// round trip.  All 256 threads then apply the panel to the columns right of
// it (a rank-16 update).  The code of a panel step is small and runs four
// times; a fully unrolled 64-column version was bound by instruction fetch.
// The inverse goes by 16x16 blocks: the diagonal blocks by substitution in
// parallel, each lane's column in registers, then each block row below as two
// small products with the rows above it, so its sequential depth is 16 rows
// rather than 64.  Everything outside the panels' chain of pivots is bound by
// the latency of shared-memory reads, so loops are unrolled and every thread
// works on several entries at once (71.5 k -> 46 k clocks per tile, the same
// roundings).
// --------------------------------------------------------------------------
constexpr int kPotrf32Threads = 256;
__global__ void __launch_bounds__(kPotrf32Threads) pchol_potrf_f32_kernel(
    float *buf, float *tinv, const BlkInfo *blk, int k, const double *diag0, float tol,
    int *status, float drop, const LookAhead la) {
  const BlkInfo bi = blk[blockIdx.x];
  if (!diag_begin(la, k < bi.Tp, status)) return;
  __shared__ float t[NB][NB + 1];
  __shared__ float X[NB][NB + 1];
  __shared__ float Tm[kPW][NB];
  const int r0 = k * NB;
  const int nr = min(NB, bi.a - r0);
  const int npiv = min(NB, bi.p - r0);
  float *g = buf + bi.base + (long long)r0 * bi.lda + r0;
  {
    const int r = threadIdx.x & (NB - 1), cs = threadIdx.x / NB;
#pragma unroll
    for (int u = 0; u < NB / (kPotrf32Threads / NB); ++u) {
      const int c = cs + u * (kPotrf32Threads / NB);
      t[r][c] = (r < nr && c < nr && r >= c) ? g[(long long)c * bi.lda + r] : 0.0f;
      X[r][c] = 0.0f;
    }
  }
  __syncthreads();
  const double *d0 = diag0 + bi.d0off + r0;
  for (int c0 = 0; c0 < npiv; c0 += kPW) {
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      float ra[kPW], rb[kPW];   // rows lane and lane + 32, columns c0 .. c0 + 15
#pragma unroll
      for (int u = 0; u < kPW; ++u) {
        ra[u] = t[lane][c0 + u];
        rb[u] = t[lane + 32][c0 + u];
      }
      const float dref_a = lane < npiv ? (float)d0[lane] : 0.0f;
      const float dref_b = lane + 32 < npiv ? (float)d0[lane + 32] : 0.0f;
#pragma unroll
      for (int u = 0; u < kPW; ++u) {
        const int c = c0 + u;
        if (c < npiv) {   // uniform over the warp
          // values, not array elements, are selected (a select of two
          // array elements would force the arrays into local memory)
          const float va = ra[u], vb = rb[u];
          const bool hi = c >= 32;
          float piv = __shfl_sync(0xffffffffu, hi ? vb : va, c & 31);
          const float dref = __shfl_sync(0xffffffffu, hi ? dref_b : dref_a, c & 31);
          const float lim = tol * dref;
          // the same safeguard as pivot_fix, in FP32
          const float repl = drop > 0.0f ? fminf(drop * fmaxf(dref, 1.0f), (float)kDropCapFP32)
                             : lim > 0.0f ? lim
                                          : 1.0f;
          if (!(piv == piv)) {
            if (lane == 0 && atomicAdd(&status[0], 1) == 0) {
              status[2] = bi.tag + (int)blockIdx.x;
              status[3] = r0 + c;
            }
            piv = repl;
          } else if (!(piv > lim) || !(piv > 0.0f)) {
            if (lane == 0) atomicAdd(&status[1], 1);
            piv = repl;
          }
          const float lcc = sqrtf(piv), inv = 1.0f / lcc;
          const float la = lane == c ? lcc : va * inv;
          const float lb = lane + 32 == c ? lcc : vb * inv;
          ra[u] = la;
          rb[u] = lb;
#pragma unroll
          for (int w = u + 1; w < kPW; ++w) {
            const int q = c0 + w;
            const float lq = __shfl_sync(0xffffffffu, q >= 32 ? lb : la, q & 31);
            ra[w] = fmaf(-la, lq, ra[w]);
            rb[w] = fmaf(-lb, lq, rb[w]);
          }
        }
      }
      // write the panel back (entries above the diagonal stay zero)
#pragma unroll
      for (int u = 0; u < kPW; ++u) {
        const int c = c0 + u;
        if (lane >= c) t[lane][c] = ra[u];
        if (lane + 32 >= c) t[lane + 32][c] = rb[u];
      }
    }
    __syncthreads();
    // rank-16 update of the lower triangle right of the panel:
    // t[r][q] -= sum_c t[r][c] t[q][c], c0 + 16 <= q <= r < nr, c < npiv
    // thread (tx, ty) takes the entries (tx, ty) of the 16x16 blocks (a, b), b <= a,
    // each sum in two chains (even and odd columns of the panel)
    const int q0 = c0 + kPW;
    const int cend = min(c0 + kPW, npiv);
    if (q0 < nr) {
      const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
      const int nbl = (nr - q0 + kPW - 1) / kPW;   // 1..3
      float s0[3][3], s1[3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) s0[a][b] = s1[a][b] = 0.0f;
      if (cend == c0 + kPW) {
#pragma unroll 4
        for (int c = c0; c < c0 + kPW; c += 2) {
          float ra[3], rb[3], qa[3], qb[3];
#pragma unroll
          for (int a = 0; a < 3; ++a)
            if (a < nbl) {
              ra[a] = t[q0 + 16 * a + tx][c];
              rb[a] = t[q0 + 16 * a + tx][c + 1];
              qa[a] = t[q0 + 16 * a + ty][c];
              qb[a] = t[q0 + 16 * a + ty][c + 1];
            }
#pragma unroll
          for (int a = 0; a < 3; ++a)
            if (a < nbl) {
#pragma unroll
              for (int b = 0; b <= a; ++b) {
                s0[a][b] = fmaf(ra[a], qa[b], s0[a][b]);
                s1[a][b] = fmaf(rb[a], qb[b], s1[a][b]);
              }
            }
        }
      } else {
        for (int c = c0; c < cend; ++c)
#pragma unroll
          for (int a = 0; a < 3; ++a)
            if (a < nbl) {
#pragma unroll
              for (int b = 0; b <= a; ++b) {
                const float x = t[q0 + 16 * a + tx][c], y = t[q0 + 16 * b + ty][c];
                if ((c - c0) & 1) s1[a][b] = fmaf(x, y, s1[a][b]);
                else s0[a][b] = fmaf(x, y, s0[a][b]);
              }
            }
      }
#pragma unroll
      for (int a = 0; a < 3; ++a)
        if (a < nbl) {
#pragma unroll
          for (int b = 0; b <= a; ++b) {
            const int r = q0 + 16 * a + tx, q = q0 + 16 * b + ty;
            if (r < nr && q <= r) t[r][q] -= s0[a][b] + s1[a][b];
          }
        }
    }
    __syncthreads();
  }
  // inverse of the pivot triangle by 16x16 blocks: warp w inverts diagonal
  // block w by substitution (lane = column); then block rows 1..3 in turn,
  // X_ij = -X_ii sum_{k=j}^{i-1} L_ik X_kj, all threads on the entries.
  // Rows at or past npiv are zero.
  const int nbk = (npiv + kPW - 1) / kPW;
  {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < 4 && lane < kPW && w * kPW < npiv) {
      // x[i]: rows b0 + i of column b0 + lane; the terms of rows above the
      // column's diagonal are zero, so every lane runs all of them
      const int b0 = w * kPW;
      float x[kPW];
#pragma unroll
      for (int i = 0; i < kPW; ++i) {
        float se = i == lane ? 1.0f : 0.0f, so = 0.0f;   // even and odd rows q
#pragma unroll
        for (int q = 0; q < i; ++q) {
          if (q & 1) so = fmaf(-t[b0 + i][b0 + q], x[q], so);
          else se = fmaf(-t[b0 + i][b0 + q], x[q], se);
        }
        x[i] = (b0 + i < npiv && i >= lane) ? (se + so) / t[b0 + i][b0 + i] : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < kPW; ++i) X[b0 + i][b0 + lane] = x[i];
    }
  }
  __syncthreads();
  for (int bi2 = 1; bi2 < nbk; ++bi2) {
    // block row bi2, columns 0 .. i0-1: thread (row r, column c) of each block
    const int i0 = bi2 * kPW;
    const int r = threadIdx.x % kPW, c = threadIdx.x / kPW;
    float s0[3], s1[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) s0[b] = s1[b] = 0.0f;
#pragma unroll 4
    for (int q = 0; q < i0; q += 2) {   // block b starts at its own row 16 b
      const float ta = t[i0 + r][q], tb = t[i0 + r][q + 1];
#pragma unroll
      for (int b = 0; b < 3; ++b)
        if (b < bi2 && q >= b * kPW) {
          s0[b] = fmaf(ta, X[q][b * kPW + c], s0[b]);
          s1[b] = fmaf(tb, X[q + 1][b * kPW + c], s1[b]);
        }
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
      if (b < bi2) Tm[r][b * kPW + c] = s0[b] + s1[b];
    __syncthreads();
    float s[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int q = 0; q < kPW; ++q) {
      const float xv = X[i0 + r][i0 + q];
      if (q <= r) {
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if (b < bi2) s[b] = fmaf(xv, Tm[q][b * kPW + c], s[b]);
      }
    }
#pragma unroll
    for (int b = 0; b < 3; ++b)
      if (b < bi2) X[i0 + r][b * kPW + c] = i0 + r < npiv ? -s[b] : 0.0f;
    __syncthreads();
  }
  float *out = tinv + bi.ioff + (long long)k * NB * NB;
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    const int r = i % NB, c = i / NB;
    if (r < nr && c < nr && r >= c) g[(long long)c * bi.lda + r] = t[r][c];
    out[i] = r < npiv ? X[r][c] : (c < npiv ? t[r][c] : 0.0f);
  }
  diag_end(la);
}

// Panel tile (I, k) below the diagonal: X = A_Ik L_kk^-T on the pivot columns
// (a 64x64x64 product with the stored inverse), then the non-pivot columns of
// a block's last pivot tile: A_Is -= X L_sk'.
// TF32 rounding (round to nearest, ties away), the value with its low 13
// mantissa bits zero
__device__ __forceinline__ float tf32_round(float x) {
  uint32_t u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
  return __uint_as_float(u);
}

// With pstage (FP32 factors, tensor-core update) the finished panel tile is
// also written to its staging slot as two TF32 words, hi = tf32(x) and
// lo = tf32(x - hi), in the K-major operand layout of tcgen05.mma without
// swizzling: 8-row x 4-column core matrices of 16-byte rows, the 16 core
// matrices of an 8-row group along the pivot columns, then the next group
// (entry (r, c) at (r/8)*512 + (c/4)*32 + (r%8)*4 + c%4; hi in words
// 0..4095, lo in 4096..8191).  Rows past the matrix and columns past the
// pivots are zero.
//
// Bound by the L1 and shared-memory path (83 % of its rate). So both operands are
// copied as they lie in memory, 16 bytes at a time and all requested before the
// first is used, and a thread's 4 x 4 entries of the product take one 16-byte read
// of each operand per pivot column (eight 4-byte reads when a thread's rows lay 16
// apart): 28 -> 22 us per step of an energy model's blocks, 11.5 -> 7.8 us on
// mid-size ones.
__global__ void __launch_bounds__(kThreads, 4)
    pchol_trsm_inv_kernel(float *buf, const float *tinv, const BlkInfo *blk, int k,
                          float *pstage) {
  pdl_begin();
  const BlkInfo bi = blk[blockIdx.y];
  if (k >= bi.Tp) return;
  const int I = k + 1 + blockIdx.x;
  if (I >= bi.T) return;
  __shared__ __align__(16) float A[NB][NB];   // A[c][r]: the tile, column c
  __shared__ __align__(16) float V[NB][NB];   // V[q][c]: inverse (c < npiv) or factor entry (c, q)
  const int r0 = k * NB;
  const int nr = min(NB, bi.a - r0);
  const int npiv = min(NB, bi.p - r0);
  const int ri = I * NB;
  const int nri = min(NB, bi.a - ri);
  float *gx = buf + bi.base + (long long)r0 * bi.lda + ri;   // base, lda: multiples of 8
  const float *ti = tinv + bi.ioff + (long long)k * NB * NB;
  {
    constexpr int kU = NB * NB / 4 / kThreads;
    float4 a[kU], v[kU];
    const int r = (threadIdx.x & 15) * 4;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int c = (threadIdx.x >> 4) + u * (kThreads / 16);
      a[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      // a tile's last rows read into the column's padding (lda >= a, rounded up)
      if (c < nr && r < nri)
        a[u] = *reinterpret_cast<const float4 *>(gx + (long long)c * bi.lda + r);
      v[u] = *reinterpret_cast<const float4 *>(ti + c * NB + r);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int c = (threadIdx.x >> 4) + u * (kThreads / 16);
      if (r + 1 >= nri) a[u].y = 0.0f;
      if (r + 2 >= nri) a[u].z = 0.0f;
      if (r + 3 >= nri) a[u].w = 0.0f;
      *reinterpret_cast<float4 *>(&A[c][r]) = a[u];
      *reinterpret_cast<float4 *>(&V[c][r]) = v[u];
    }
  }
  __syncthreads();
  const int tr = (threadIdx.x & 15) * 4, tc = (threadIdx.x >> 4) * 4;   // 4 x 4 entries
  float acc[4][4];   // [column][row]
#pragma unroll
  for (int b = 0; b < 4; ++b)
#pragma unroll
    for (int a = 0; a < 4; ++a) acc[b][a] = 0.0f;
#pragma unroll 8
  for (int q = 0; q < npiv; ++q) {
    const float4 av = *reinterpret_cast<const float4 *>(&A[q][tr]);
    const float4 bv = *reinterpret_cast<const float4 *>(&V[q][tc]);   // zero for q > column
    const float x[4] = {av.x, av.y, av.z, av.w}, y[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int a = 0; a < 4; ++a) acc[b][a] = fmaf(x[a], y[b], acc[b][a]);
  }
  if (npiv < nr) {   // the last pivot tile's other columns
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (tc + b < npiv) {
#pragma unroll
        for (int a = 0; a < 4; ++a) A[tc + b][tr + a] = acc[b][a];
      }
    __syncthreads();
    const int ns = nr - npiv;
    for (int idx = threadIdx.x; idx < NB * ns; idx += kThreads) {
      const int r = idx % NB, sc = npiv + idx / NB;
      if (r >= nri) continue;
      float u = A[sc][r];
      for (int c = 0; c < npiv; ++c) u = fmaf(-A[c][r], V[c][sc], u);
      gx[(long long)sc * bi.lda + r] = u;
    }
  }
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    if (tc + b >= npiv) continue;
    float *g = gx + (long long)(tc + b) * bi.lda + tr;
    if (tr + 3 < nri) {
      *reinterpret_cast<float4 *>(g) = make_float4(acc[b][0], acc[b][1], acc[b][2], acc[b][3]);
    } else {
#pragma unroll
      for (int a = 0; a < 4; ++a)
        if (tr + a < nri) g[a] = acc[b][a];
    }
  }
  if (pstage) {
    float *st = pstage + (bi.soff + I) * 8192LL + tc * 8;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int r = tr + a;
      float h[4], l[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float v = (r < nri && tc + b < npiv) ? acc[b][a] : 0.0f;
        h[b] = tf32_round(v);
        l[b] = tf32_round(v - h[b]);
      }
      float *o = st + (r >> 3) * 512 + (r & 7) * 4;
      *reinterpret_cast<float4 *>(o) = make_float4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<float4 *>(o + NB * NB) = make_float4(l[0], l[1], l[2], l[3]);
    }
  }
}

// --------------------------------------------------------------------------
// float-float factors (hi + lo, both FP32).  The diagonal tile and the panel
// run in FP64 arithmetic on the converted values (a small share of the work);
// the trailing update -- nearly all the flops -- runs in double-float
// arithmetic on the FP32 pipe: each product by an FMA-based exact product, the
// sum by error-free two-sum, the low parts in FP32, renormalised per chunk.
// The __f*_rn intrinsics keep the compiler from contracting the error-free
// transformations into FMAs.
// --------------------------------------------------------------------------
// (sh, sl) += (ah + al)(bh + bl), al*bl dropped
__device__ __forceinline__ void ff_mac(float &sh, float &sl, float ah, float al, float bh,
                                       float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = fmaf(ah, bh, -p);   // exact rounding error of ah*bh
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  const float t = __fadd_rn(sh, p);
  const float bv = __fsub_rn(t, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bv)), __fsub_rn(p, bv));
  sh = t;
  sl = __fadd_rn(sl, __fadd_rn(err, e));
}

__device__ __forceinline__ void ff_renorm(float &sh, float &sl) {
  const float h = __fadd_rn(sh, sl);
  sl = __fsub_rn(sl, __fsub_rn(h, sh));
  sh = h;
}

// hi + lo -> FP64 copy of the float-float factor, used by the solves; four
// entries per thread and step (16-byte loads of each word, two 16-byte
// stores; the buffers are cudaMalloc-aligned), the last n % 4 one by one
__global__ void ff_expand_kernel(const float *hi, const float *lo,
                                 double *out, long long n) {
  pdl_begin();
  const long long n4 = n / 4;
  const float4 *h4 = reinterpret_cast<const float4 *>(hi);
  const float4 *l4 = reinterpret_cast<const float4 *>(lo);
  double2 *o2 = reinterpret_cast<double2 *>(out);
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
    const float4 h = __ldcs(h4 + i), l = __ldcs(l4 + i);
    __stcs(o2 + 2 * i, make_double2((double)h.x + (double)l.x, (double)h.y + (double)l.y));
    __stcs(o2 + 2 * i + 1, make_double2((double)h.z + (double)l.z, (double)h.w + (double)l.w));
  }
  for (long long i = 4 * n4 + (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += stride)
    out[i] = (double)hi[i] + (double)lo[i];
}

// With dstage (the tensor-core float-float update, k_tc.cu) the finished
// panel tile is also written as exact integer digits: per row r, E_r is the
// exponent with max_c |x_rc| < 2^E_r, and x = 2^E_r sum_s d_s 2^(-9-8s),
// s = 0..5, with |d_0| <= 512 and |d_s| <= 128 (s > 0), each digit an FP16
// integer (49 bits in all).  The digits are taken from the stored pair
// (hi, lo), scaled by a power of two and peeled off in FP32 with every
// remainder kept exactly (a two-word remainder, renormalised by two-sum).
// Digit plane s of the tile is a 64 x 64 FP16 K-major operand without
// swizzling, split into two K halves so that either half is one contiguous
// 4 KB run: entry (r, c) at (c/32)*2048 + (r/8)*256 + ((c%32)/8)*64 +
// (r%8)*8 + c%8; the six planes follow each other (4096 entries each).  Rows
// past the matrix and columns past the pivots are zero.
constexpr int kOzDigits = 6;

__device__ __forceinline__ void two_sum_f(float &a, float &b) {   // (a, b) <- fl(a+b), error
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  a = s;
  b = err;
}

__device__ __forceinline__ void oz_digits(float h, float l, int e, float (&d)[kOzDigits]) {
  h = ldexpf(h, 9 - e);
  l = ldexpf(l, 9 - e);
#pragma unroll
  for (int s = 0; s < kOzDigits; ++s) {
    if (s > 0) {
      h = __fmul_rn(h, 256.0f);
      l = __fmul_rn(l, 256.0f);
    }
    const float q = rintf(h);
    d[s] = q;
    h = __fsub_rn(h, q);   // exact: q is the integer nearest to h
    two_sum_f(h, l);
  }
}

// The panel in double-float arithmetic on the FP32 pipe (FP64 runs at 1/74
// of the FP32 rate on this part): column c of X = A_Ik L_kk^-T is scaled by
// the pivot's reciprocal (taken in FP64 and split into two words), then
// removed from the columns right of it, every product an FMA-based exact
// product and every difference an error-free two-sum.
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float &ph,
                                       float &pl) {
  const float p = __fmul_rn(ah, bh);
  float e = fmaf(ah, bh, -p);
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  ph = __fadd_rn(p, e);
  pl = __fsub_rn(e, __fsub_rn(ph, p));
}

__device__ __forceinline__ void df_sub(float &xh, float &xl, float ph, float pl) {
  const float s = __fsub_rn(xh, ph);
  const float bv = __fsub_rn(s, xh);
  const float err = __fadd_rn(__fsub_rn(xh, __fsub_rn(s, bv)), __fsub_rn(-ph, bv));
  const float el = __fadd_rn(err, __fsub_rn(xl, pl));
  xh = __fadd_rn(s, el);
  xl = __fsub_rn(el, __fsub_rn(xh, s));
}

// Rows of X are independent (X_r = A_r L^-T), so one thread solves one row
// and no step waits for another thread.  A row is taken in chunks of 16
// columns held in registers: first every finished column left of the chunk
// (kept in shared memory) is removed from it, then the chunk's own triangle
// is solved.  Every entry so receives the same operations in the same order
// as in column-by-column substitution (the subtractions of columns
// 0, 1, ..., c - 1, then the scaling), and the same rounding.  Two tiles of
// the same block and step per CTA share the pivot tile.
constexpr int kFFRowTiles = 2;
constexpr int kFFRowThreads = kFFRowTiles * NB;
constexpr int kFFChunk = 16;
constexpr size_t kTrsmFFSmem =
    (2 * NB * NB + 2 * kFFRowTiles * NB * NB + 2 * NB) * sizeof(float);

__global__ void __launch_bounds__(kFFRowThreads) pchol_trsm_ff_kernel(float *hi, float *lo,
                                                                     const BlkInfo *blk, int k,
                                                                     __half *dstage, int *dexp) {
  pdl_begin();
  const BlkInfo bi = blk[blockIdx.y];
  if (k >= bi.Tp) return;
  const int I0 = k + 1 + kFFRowTiles * blockIdx.x;
  if (I0 >= bi.T) return;
  extern __shared__ __align__(16) float trsm_f[];
  float *Lth = trsm_f;                     // [c][sc] = L_kk(sc, c): pivot column c contiguous
  float *Ltl = Lth + NB * NB;
  float *Xsh = Ltl + NB * NB;              // [tile][c][r]: finished columns of the rows
  float *Xsl = Xsh + kFFRowTiles * NB * NB;
  float *s_ih = Xsl + kFFRowTiles * NB * NB;   // pivot reciprocals, split in two words
  float *s_il = s_ih + NB;
  const int r0 = k * NB;
  const int nr = min(NB, bi.a - r0);
  const int npiv = min(NB, bi.p - r0);
  const long long gl = bi.base + (long long)r0 * bi.lda + r0;
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    const int sc = i % NB, c = i / NB;
    const bool lin = sc < nr && c < nr && sc >= c;
    const long long el = gl + (long long)c * bi.lda + sc;
    Lth[c * NB + sc] = lin ? hi[el] : 0.0f;
    Ltl[c * NB + sc] = lin ? lo[el] : 0.0f;
  }
  __syncthreads();
  if (threadIdx.x < npiv) {
    const int c = threadIdx.x;
    const double inv = 1.0 / ((double)Lth[c * NB + c] + (double)Ltl[c * NB + c]);
    s_ih[c] = (float)inv;
    s_il[c] = (float)(inv - (double)s_ih[c]);
  }
  __syncthreads();

  const int t = threadIdx.x / NB, r = threadIdx.x % NB;
  const int I = I0 + t;
  const bool tile_ok = I < bi.T;
  const int ri = I * NB;
  const int nri = tile_ok ? min(NB, bi.a - ri) : 0;
  const bool row_ok = r < nri;
  const long long gx = bi.base + (long long)r0 * bi.lda + ri;
  float *xsh = Xsh + t * NB * NB + r, *xsl = Xsl + t * NB * NB + r;   // column c at [c * NB]
  for (int c0 = 0; c0 < nr; c0 += kFFChunk) {
    float xh[kFFChunk], xl[kFFChunk];
#pragma unroll
    for (int j = 0; j < kFFChunk; ++j) {
      const int c = c0 + j;
      const bool in = row_ok && c < nr;
      xh[j] = in ? hi[gx + (long long)c * bi.lda + r] : 0.0f;
      xl[j] = in ? lo[gx + (long long)c * bi.lda + r] : 0.0f;
    }
    // the finished pivot columns left of the chunk
    const int cend = min(c0, npiv);
    for (int c = 0; c < cend; ++c) {
      const float ah = xsh[c * NB], al = xsl[c * NB];
      const float4 *Lh4 = reinterpret_cast<const float4 *>(Lth + c * NB + c0);
      const float4 *Ll4 = reinterpret_cast<const float4 *>(Ltl + c * NB + c0);
#pragma unroll
      for (int q = 0; q < kFFChunk / 4; ++q) {
        const float4 bh = Lh4[q], bl = Ll4[q];
        const float bhv[4] = {bh.x, bh.y, bh.z, bh.w}, blv[4] = {bl.x, bl.y, bl.z, bl.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float ph, pl;
          df_mul(ah, al, bhv[u], blv[u], ph, pl);
          df_sub(xh[4 * q + u], xl[4 * q + u], ph, pl);
        }
      }
    }
    // the chunk's own triangle
#pragma unroll
    for (int j = 0; j < kFFChunk; ++j) {
      const int c = c0 + j;
      if (c < npiv) {
        df_mul(xh[j], xl[j], s_ih[c], s_il[c], xh[j], xl[j]);
#pragma unroll
        for (int jj = j + 1; jj < kFFChunk; ++jj) {
          float ph, pl;
          df_mul(xh[j], xl[j], Lth[c * NB + c0 + jj], Ltl[c * NB + c0 + jj], ph, pl);
          df_sub(xh[jj], xl[jj], ph, pl);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kFFChunk; ++j) {
      const int c = c0 + j;
      xsh[c * NB] = xh[j];
      xsl[c * NB] = xl[j];
      if (row_ok && c < nr) {
        hi[gx + (long long)c * bi.lda + r] = xh[j];
        lo[gx + (long long)c * bi.lda + r] = xl[j];
      }
    }
  }
  if (dstage && tile_ok) {
    const long long slot = bi.soff + I;
    float mx = 0.0f;
    if (row_ok)
      for (int c = 0; c < npiv; ++c) mx = fmaxf(mx, fabsf(xsh[c * NB]));
    int e = 0;
    if (mx > 0.0f) frexpf(mx, &e);   // mx = f 2^e, f in [0.5, 1)
    dexp[slot * NB + r] = e;
    __half *st = dstage + slot * (kOzDigits * NB * NB) + (r >> 3) * 256 + (r & 7) * 8;
#pragma unroll 1
    for (int cg = 0; cg < NB / 8; ++cg) {   // 8 consecutive columns: one 16-byte run per plane
      __align__(16) __half dv[kOzDigits][8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int c = cg * 8 + u;
        float d[kOzDigits];
        if (row_ok && c < npiv) {
          oz_digits(xsh[c * NB], xsl[c * NB], e, d);
        } else {
#pragma unroll
          for (int q = 0; q < kOzDigits; ++q) d[q] = 0.0f;
        }
#pragma unroll
        for (int q = 0; q < kOzDigits; ++q) dv[q][u] = __float2half_rn(d[q]);
      }
      const int off = (cg >> 2) * 2048 + (cg & 3) * 64;
#pragma unroll
      for (int q = 0; q < kOzDigits; ++q)
        *reinterpret_cast<uint4 *>(st + q * NB * NB + off) =
            *reinterpret_cast<const uint4 *>(dv[q]);
    }
  }
}

// trailing update: C_IJ -= L_Ik L_Jk' over the pivot columns of step k (the
// FP64 factor; FP32 and float-float have their own kernels below).
constexpr int KC = 16;
// S x S CTAs per tile: a tile keeps one SM's FP64 pipe busy for 69 us, so a step
// with fewer tiles than SMs spreads them (79 us at S = 1)
template <typename T, int S>
__global__ void __launch_bounds__(kThreads) pchol_update_kernel(T *buf, const BlkInfo *blk, int k) {
  constexpr int M = NB / S, A = M / 16;
  pdl_begin();
  const BlkInfo bi = blk[blockIdx.y];
  if (k >= bi.Tp) return;
  const long long t = bi.T - k - 1;
  const long long q = blockIdx.x / (S * S);
  const int sub = blockIdx.x % (S * S), sI = sub / S, sJ = sub % S;
  if (q >= t * (t + 1) / 2) return;
  long long ii = (long long)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
  while (ii * (ii + 1) / 2 > q) --ii;
  while ((ii + 1) * (ii + 2) / 2 <= q) ++ii;
  const long long jj = q - ii * (ii + 1) / 2;
  const int I = k + 1 + (int)ii, J = k + 1 + (int)jj;
  const int npiv = min(NB, bi.p - k * NB);
  if (I == J && sI < sJ) return;
  const int rI = I * NB + sI * M, rJ = J * NB + sJ * M;
  const int nrI = min(M, bi.a - rI), nrJ = min(M, bi.a - rJ);   // may be negative
  __shared__ T As[KC][M];
  __shared__ T Bs[KC][M];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  T acc[A][A];
#pragma unroll
  for (int i = 0; i < A; ++i)
#pragma unroll
    for (int j = 0; j < A; ++j) acc[i][j] = T(0);
  const T *colk = buf + bi.base + (long long)(k * NB) * bi.lda;
  for (int kc = 0; kc < npiv; kc += KC) {
    for (int idx = threadIdx.x; idx < KC * M; idx += blockDim.x) {
      const int r = idx % M, kk = idx / M;
      const bool kin = (kc + kk) < npiv;
      const T *col = colk + (long long)(kc + kk) * bi.lda;
      As[kk][r] = (kin && r < nrI) ? col[rI + r] : T(0);
      Bs[kk][r] = (kin && r < nrJ) ? col[rJ + r] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KC; ++kk) {
      T av[A], bv[A];
#pragma unroll
      for (int i = 0; i < A; ++i) av[i] = As[kk][tx + 16 * i];
#pragma unroll
      for (int j = 0; j < A; ++j) bv[j] = Bs[kk][ty + 16 * j];
#pragma unroll
      for (int i = 0; i < A; ++i)
#pragma unroll
        for (int j = 0; j < A; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
  T *gc = buf + bi.base + (long long)rJ * bi.lda + rI;
#pragma unroll
  for (int j = 0; j < A; ++j) {
    const int c = ty + 16 * j;
#pragma unroll
    for (int i = 0; i < A; ++i) {
      const int r = tx + 16 * i;
      if (r < nrI && c < nrJ && (I != J || sI != sJ || r >= c))
        gc[(long long)c * bi.lda + r] -= acc[i][j];
    }
  }
}

// FP32 trailing update.  The FP64 kernel's 4x4-per-thread tile above, run in
// FP32, leaves the FP32 pipe waiting on shared-memory issue (8 scalar loads
// per 16 FMAs); here 64
// threads cover the 64x64 tile with an 8x8 register tile each, reading it
// with four 16-byte shared loads per 64 FMAs.  Rows 4tx..4tx+3 and
// 32+4tx..35+4tx, columns likewise with ty, so that the 16-byte loads of a
// quarter warp cover 128 contiguous bytes.  The whole 64-column panel is
// requested up front with cp.async, in four 16-column groups, and the
// arithmetic on a group starts as soon as it has landed, so the later groups
// arrive behind the arithmetic; ragged rows and columns past the pivots are
// zero-filled by the copy itself.
constexpr int kUpdF32Threads = 64;

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem, int src_bytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem),
               "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__global__ void __launch_bounds__(kUpdF32Threads) pchol_update_f32_kernel(float *buf,
                                                                         const BlkInfo *blk,
                                                                         int k) {
  pdl_begin();
  const BlkInfo bi = blk[blockIdx.y];
  if (k >= bi.Tp) return;
  const long long t = bi.T - k - 1;
  const long long q = blockIdx.x;
  if (q >= t * (t + 1) / 2) return;
  long long ii = (long long)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
  while (ii * (ii + 1) / 2 > q) --ii;
  while ((ii + 1) * (ii + 2) / 2 <= q) ++ii;
  const long long jj = q - ii * (ii + 1) / 2;
  const int I = k + 1 + (int)ii, J = k + 1 + (int)jj;
  const int npiv = min(NB, bi.p - k * NB);
  const int rI = I * NB, rJ = J * NB;
  const int nrI = min(NB, bi.a - rI), nrJ = min(NB, bi.a - rJ);
  __shared__ __align__(16) float As[NB][NB];   // [pivot column][row]
  __shared__ __align__(16) float Bs[NB][NB];
  const int tid = threadIdx.x;
  const int tx = tid & 7, ty = tid >> 3;
  // copies: thread moves float4 number (tid & 15) of columns (tid >> 4) + 4u
  const int lv = (tid & 15) * 4, lk = tid >> 4;
  const float *colk = buf + bi.base + (long long)(k * NB) * bi.lda;
  const int nchunk = (npiv + 15) / 16;
  const int na = 4 * max(0, min(4, nrI - lv)), nb = 4 * max(0, min(4, nrJ - lv));
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    if (ch < nchunk) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int kk = ch * 16 + lk + 4 * u;
        const bool kin = kk < npiv;
        // a zero-byte copy still names a valid address: row rI / rJ of a pivot column
        const float *col = colk + (long long)(kin ? kk : 0) * bi.lda;
        cp_async16(&As[kk][lv], col + rI + (kin && na ? lv : 0), kin ? na : 0);
        cp_async16(&Bs[kk][lv], col + rJ + (kin && nb ? lv : 0), kin ? nb : 0);
      }
    }
    cp_async_commit();
  }
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
  for (int ch = 0; ch < nchunk; ++ch) {
    if (ch == 0) cp_async_wait<3>();
    else if (ch == 1) cp_async_wait<2>();
    else if (ch == 2) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncthreads();
#pragma unroll
    for (int kq = 0; kq < 16; ++kq) {
      const int kk = ch * 16 + kq;
      const float4 a0 = *reinterpret_cast<const float4 *>(&As[kk][4 * tx]);
      const float4 a1 = *reinterpret_cast<const float4 *>(&As[kk][32 + 4 * tx]);
      const float4 b0 = *reinterpret_cast<const float4 *>(&Bs[kk][4 * ty]);
      const float4 b1 = *reinterpret_cast<const float4 *>(&Bs[kk][32 + 4 * ty]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
  float *gc = buf + bi.base + (long long)rJ * bi.lda + rI;
  const bool diag = I == J;
  if (!diag && nrI == NB && nrJ == NB) {
    // interior tile: the eight loads of a row quad are issued before any store
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = h == 0 ? 4 * tx : 32 + 4 * tx;
      float4 cv[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = (j < 4 ? 4 * ty : 32 + 4 * ty) + (j & 3);
        cv[j] = *reinterpret_cast<const float4 *>(gc + (long long)c * bi.lda + r);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = (j < 4 ? 4 * ty : 32 + 4 * ty) + (j & 3);
        cv[j].x -= acc[4 * h][j];
        cv[j].y -= acc[4 * h + 1][j];
        cv[j].z -= acc[4 * h + 2][j];
        cv[j].w -= acc[4 * h + 3][j];
        *reinterpret_cast<float4 *>(gc + (long long)c * bi.lda + r) = cv[j];
      }
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int c = (j < 4 ? 4 * ty : 32 + 4 * ty) + (j & 3);
    if (c >= nrJ) continue;
    float *col = gc + (long long)c * bi.lda;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = (h == 0 ? 4 * tx : 32 + 4 * tx);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (r + e < nrI && (!diag || r + e >= c)) col[r + e] -= acc[4 * h + e][j];
    }
  }
}

// Float-float trailing update with an 8x4 register tile per thread (128
// threads per 64x64 tile): rows 4tx..4tx+3 and 32+4tx..35+4tx, columns
// 4ty..4ty+3, read with six 16-byte shared loads per 32 multiply-adds of 12
// FP32 operations each.  The whole panel (high and low words of both tile
// rows, 64 KB) is requested up front with cp.async in four 16-column groups.
constexpr int kUpdFFThreads = 128;
constexpr size_t kUpdFFSmem = 4 * NB * NB * sizeof(float);

__global__ void __launch_bounds__(kUpdFFThreads) pchol_update_ff8_kernel(float *hi, float *lo,
                                                                        const BlkInfo *blk,
                                                                        int k) {
  pdl_begin();
  const BlkInfo bi = blk[blockIdx.y];
  if (k >= bi.Tp) return;
  const long long t = bi.T - k - 1;
  const long long q = blockIdx.x;
  if (q >= t * (t + 1) / 2) return;
  long long ii = (long long)((sqrt(8.0 * (double)q + 1.0) - 1.0) * 0.5);
  while (ii * (ii + 1) / 2 > q) --ii;
  while ((ii + 1) * (ii + 2) / 2 <= q) ++ii;
  const long long jj = q - ii * (ii + 1) / 2;
  const int I = k + 1 + (int)ii, J = k + 1 + (int)jj;
  const int npiv = min(NB, bi.p - k * NB);
  const int rI = I * NB, rJ = J * NB;
  const int nrI = min(NB, bi.a - rI), nrJ = min(NB, bi.a - rJ);
  extern __shared__ __align__(16) float ffsm[];
  float(*Ah)[NB] = reinterpret_cast<float(*)[NB]>(ffsm);
  float(*Al)[NB] = reinterpret_cast<float(*)[NB]>(ffsm + NB * NB);
  float(*Bh)[NB] = reinterpret_cast<float(*)[NB]>(ffsm + 2 * NB * NB);
  float(*Bl)[NB] = reinterpret_cast<float(*)[NB]>(ffsm + 3 * NB * NB);
  const int tid = threadIdx.x;
  const int tx = tid & 7, ty = tid >> 3;
  // copies: thread moves float4 number (tid & 15) of column (tid >> 4) of a
  // chunk, for both words of both tile rows (8 x 16-byte copies per chunk)
  const int lv = (tid & 15) * 4, lk = tid >> 4;
  const long long colk = bi.base + (long long)(k * NB) * bi.lda;
  const int nchunk = (npiv + 15) / 16;
  const int na = 4 * max(0, min(4, nrI - lv)), nb = 4 * max(0, min(4, nrJ - lv));
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    if (ch < nchunk) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int kk = ch * 16 + lk + 8 * u;
        const bool kin = kk < npiv;
        const long long col = colk + (long long)(kin ? kk : 0) * bi.lda;
        const long long oa = col + rI + (kin && na ? lv : 0);
        const long long ob = col + rJ + (kin && nb ? lv : 0);
        cp_async16(&Ah[kk][lv], hi + oa, kin ? na : 0);
        cp_async16(&Al[kk][lv], lo + oa, kin ? na : 0);
        cp_async16(&Bh[kk][lv], hi + ob, kin ? nb : 0);
        cp_async16(&Bl[kk][lv], lo + ob, kin ? nb : 0);
      }
    }
    cp_async_commit();
  }
  float sh[8][4], sl[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) sh[i][j] = sl[i][j] = 0.0f;
  for (int ch = 0; ch < nchunk; ++ch) {
    if (ch == 0) cp_async_wait<3>();
    else if (ch == 1) cp_async_wait<2>();
    else if (ch == 2) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncthreads();
#pragma unroll 4
    for (int kq = 0; kq < 16; ++kq) {
      const int kk = ch * 16 + kq;
      const float4 h0 = *reinterpret_cast<const float4 *>(&Ah[kk][4 * tx]);
      const float4 h1 = *reinterpret_cast<const float4 *>(&Ah[kk][32 + 4 * tx]);
      const float4 l0 = *reinterpret_cast<const float4 *>(&Al[kk][4 * tx]);
      const float4 l1 = *reinterpret_cast<const float4 *>(&Al[kk][32 + 4 * tx]);
      const float4 bh4 = *reinterpret_cast<const float4 *>(&Bh[kk][4 * ty]);
      const float4 bl4 = *reinterpret_cast<const float4 *>(&Bl[kk][4 * ty]);
      const float ah[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
      const float al[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
      const float bh[4] = {bh4.x, bh4.y, bh4.z, bh4.w};
      const float bl[4] = {bl4.x, bl4.y, bl4.z, bl4.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ff_mac(sh[i][j], sl[i][j], ah[i], al[i], bh[j], bl[j]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) ff_renorm(sh[i][j], sl[i][j]);
  }
  const long long g = bi.base + (long long)rJ * bi.lda + rI;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int c = 4 * ty + j;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = (i < 4 ? 4 * tx : 32 + 4 * tx) + (i & 3);
      if (r < nrI && c < nrJ && (I != J || r >= c)) {
        const long long e = g + (long long)c * bi.lda + r;
        // (ch + cl) - (sh + sl): two-sum of the high parts, low parts added
        const float chv = hi[e], clv = lo[e], s = sh[i][j];
        const float tt = __fsub_rn(chv, s);
        const float bv = __fsub_rn(tt, chv);
        const float err = __fadd_rn(__fsub_rn(chv, __fsub_rn(tt, bv)), __fsub_rn(-s, bv));
        const float el = __fadd_rn(err, __fsub_rn(clv, sl[i][j]));
        const float h = __fadd_rn(tt, el);
        hi[e] = h;
        lo[e] = __fsub_rn(el, __fsub_rn(h, tt));
      }
    }
  }
}

// --------------------------------------------------------------------------
// Wavefront solves with the block partial factors: one CTA per (block, 64-row
// tile), so every block's factor is streamed by many SMs at once.
//
// Each CTA draws a ticket from an atomic counter and takes the job the
// schedule lists under that ticket.  The schedule is in wavefront order (tile
// r of every block before tile r+1 of any block; reversed for the backward
// sweep), so a tile only ever waits for tiles holding smaller tickets, which
// are already running: the waits cannot deadlock.  A CTA prefetches its part
// of the factor before it waits for the entries it needs, solves its diagonal
// tile and publishes its solution rows.  Every wait is bounded: after
// kWaitLimitNs the error word is set, the CTA stops waiting and the host
// reports AHLP_ERR_TIMEOUT.
//
// forward : v <- [L11 0; L21 I]^-1 v     (all a rows; pivot tiles publish)
// backward: v_top <- L11^-T (v_top - L21' v_bottom), v_bottom unchanged
// --------------------------------------------------------------------------
// Inverted diagonal tiles of FP64 factors, one CTA per pivot tile.  The
// non-pivot rows of a block's last pivot tile keep the factor entries, so the
// solves stage one 64x64 tile that covers their whole diagonal step.  By 16x16
// blocks: the diagonal blocks by substitution (a warp each, lane = column),
// then block rows 1..3 in turn, X_ij = -X_ii sum_{k=j}^{i-1} L_ik X_kj, all
// threads on the entries; the FP64 pipe (two lanes per clock) bounds it.  All
// tiles of 32 blocks (1130 tiles): 326 -> 150 us against one thread per column.
constexpr size_t kTinvSmem = (2 * NB * (NB + 1) + 16 * NB + NB) * sizeof(double);

__global__ void __launch_bounds__(kThreads) tinv_kernel(const double *buf,
                                                        double *tinv,
                                                        const BlkInfo *__restrict__ blk,
                                                        const int *__restrict__ sched) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char tinv_raw[];   // kTinvSmem bytes
  double(*Ls)[NB + 1] = reinterpret_cast<double(*)[NB + 1]>(tinv_raw);
  double(*Xs)[NB + 1] = Ls + NB;
  double *Tm = reinterpret_cast<double *>(Xs + NB);   // [16][wc]
  double *rinv = Tm + 16 * NB;
  const int b = sched[2 * blockIdx.x], k = sched[2 * blockIdx.x + 1];
  const BlkInfo bi = blk[b];
  const double *L = buf + bi.base;
  const int r0 = k * NB, nr = min(NB, bi.a - r0), npiv = min(NB, bi.p - r0);
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    const int r = i % NB, c = i / NB;
    Ls[r][c] = (r < nr && c < npiv && r >= c) ? L[(long long)(r0 + c) * bi.lda + r0 + r] : 0.0;
    Xs[r][c] = 0.0;
  }
  __syncthreads();
  if (threadIdx.x < npiv) rinv[threadIdx.x] = 1.0 / Ls[threadIdx.x][threadIdx.x];
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < 4 && lane < 16) {
    const int b0 = w * 16, j = b0 + lane, e = min(b0 + 16, npiv);
    for (int i = b0; i < e; ++i) {   // rows above the column's diagonal come out zero
      double s0 = i == j ? 1.0 : 0.0, s1 = 0.0;
      int q = b0;
      for (; q + 1 < i; q += 2) {
        s0 = fma(-Ls[i][q], Xs[q][j], s0);
        s1 = fma(-Ls[i][q + 1], Xs[q + 1][j], s1);
      }
      if (q < i) s0 = fma(-Ls[i][q], Xs[q][j], s0);
      Xs[i][j] = (s0 + s1) * rinv[i];
    }
  }
  __syncthreads();
  for (int i0 = 16; i0 < npiv; i0 += 16) {
    const int wc = i0;   // columns 0 .. i0 - 1 of this block row
    for (int e = threadIdx.x; e < 16 * wc; e += blockDim.x) {
      const int r = e / wc, c = e - r * wc;
      double s0 = 0.0, s1 = 0.0;
      for (int q = c & ~15; q < i0; q += 2) {
        s0 = fma(Ls[i0 + r][q], Xs[q][c], s0);
        s1 = fma(Ls[i0 + r][q + 1], Xs[q + 1][c], s1);
      }
      Tm[r * wc + c] = s0 + s1;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * wc; e += blockDim.x) {
      const int r = e / wc, c = e - r * wc;
      double s = 0.0;
      for (int q = 0; q <= r; ++q) s = fma(Xs[i0 + r][i0 + q], Tm[q * wc + c], s);
      if (i0 + r < npiv) Xs[i0 + r][c] = -s;
    }
    __syncthreads();
  }
  double *out = tinv + bi.ioff + (long long)k * NB * NB;
  for (int i = threadIdx.x; i < NB * NB; i += blockDim.x) {
    const int r = i % NB, c = i / NB;
    out[i] = r < npiv ? Xs[r][c] : Ls[r][c];
  }
}

// thread = (row rho of a 64-row tile or chunk, column lane q); lane q owns the
// columns q, q + kQL, ... of a 64-column tile.  The next factor tile's entries
// are loaded into registers while this one is used (a shared-memory ring with a
// barrier per tile measured slower), and a warp waits for its own entries of
// the solution alone, so the sweep over a row of tiles has no barrier.  FP32
// forward: 256 threads (sixteen entries each, three CTAs per SM); the others
// 512 threads (eight entries each, two CTAs per SM).  With the factor streamed,
// the chain of tiles is the bound: a link (wait, one tile's product, the
// product with the inverted diagonal tile, publish) took 5.2 us in FP32, and
// 17 us in the FP64 backward sweep, whose eight sums per thread each went
// through five FP64 shuffle steps.
template <typename T, bool Bwd>
struct TrsvCfg {
  static constexpr bool narrow = sizeof(T) == 4 && !Bwd;
  static constexpr int threads = narrow ? 256 : 512;
  static constexpr int min_ctas = narrow ? 3 : 2;   // per SM
  static constexpr int ql = threads / NB;           // column lanes
  static constexpr int jc = NB / ql;                // columns per thread
};

// Sum over a warp of each of a thread's eight values by a transposing exchange
// (the additions of an xor tree, nine per thread instead of forty): the total
// of value warp_sum8_index(lane) is returned.
template <typename T>
__device__ __forceinline__ T warp_sum8(const T (&a)[8], int lane) {
  T h4[4], h2[2];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const T keep = (lane & 16) ? a[u + 4] : a[u], give = (lane & 16) ? a[u] : a[u + 4];
    h4[u] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const T keep = (lane & 8) ? h4[u + 2] : h4[u], give = (lane & 8) ? h4[u] : h4[u + 2];
    h2[u] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
  }
  const T keep = (lane & 4) ? h2[1] : h2[0], give = (lane & 4) ? h2[0] : h2[1];
  T t = keep + __shfl_xor_sync(0xffffffffu, give, 4);
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  return t;
}
__device__ __forceinline__ int warp_sum8_index(int lane) {
  return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
}

// n contiguous entries (a multiple of 16 bytes)
template <typename T>
__device__ __forceinline__ void stage_contiguous(T *dst, const T *src, int n) {
  constexpr int EPC = 16 / sizeof(T);
  for (int i = threadIdx.x * EPC; i < n; i += blockDim.x * EPC) cp_async16(dst + i, src + i, 16);
}

// pub: publication buffer, x on the pivot rows; vec receives every row in FP64
// (the same buffer for FP64 factors)
template <typename T>
__global__ void __launch_bounds__(TrsvCfg<T, false>::threads, TrsvCfg<T, false>::min_ctas)
    trsv_fwd_kernel(const T *buf, const T *tinv,
                    const BlkInfo *__restrict__ blk, const int *__restrict__ sched, int *ticket,
                    int *err, double *vec, T *pub, const double *rhs,
                    const long long *__restrict__ yoff) {
  pdl_begin();
  using P = PubBits<T>;
  constexpr int kQL = TrsvCfg<T, false>::ql, kJC = TrsvCfg<T, false>::jc;
  __shared__ __align__(16) T Xs[NB * NB];      // column-major, Xs[c * NB + r]
  __shared__ T red[kQL][NB];
  __shared__ T u[NB];
  __shared__ T xs[NB];
  __shared__ int s_job;
  if (threadIdx.x == 0) s_job = atomicAdd(ticket, 1);
  __syncthreads();
  const int b = sched[2 * s_job], r = sched[2 * s_job + 1];
  const BlkInfo bi = blk[b];
  const T *L = buf + bi.base;
  const long long lda = bi.lda;
  double *gv = vec + bi.voff;
  T *gp = pub + bi.voff;
  const int r0 = r * NB, nr = min(NB, bi.a - r0);
  const bool pivtile = r < bi.Tp;
  const int npiv = pivtile ? min(NB, bi.p - r0) : 0;
  const int rho = threadIdx.x & (NB - 1), q = threadIdx.x / NB, lane = threadIdx.x & 31;
  const int nct = min(r, bi.Tp);   // pivot column tiles left of this tile
  if (pivtile) stage_contiguous(Xs, tinv + bi.ioff + (long long)r * NB * NB, NB * NB);
  cp_async_commit();
  // the block's rows of the right-hand side; zero in its Schur rows
  const double rhs_r = (threadIdx.x < nr && r0 + (int)threadIdx.x < bi.p)
                           ? rhs[yoff[b] + r0 + threadIdx.x]
                           : 0.0;
  T acc0 = T(0), acc1 = T(0);
  {
    const bool rok = rho < nr;
    const T *Lr = L + r0 + rho;
    T l[kJC], ln[kJC];
    auto load_tile = [&](int k, T(&dst)[kJC]) {
      const int c0 = k * NB, nc = min(NB, bi.p - c0);
#pragma unroll
      for (int j = 0; j < kJC; ++j) {
        const int c = q + kQL * j;
        dst[j] = (rok && c < nc) ? Lr[(long long)(c0 + c) * lda] : T(0);
      }
    };
    // a warp's columns all have its q: lane j holds column q + kQL j's solution
    const int xc = q + kQL * (lane < kJC ? lane : 0);
    auto x_in = [&](int k) { return lane < kJC && k * NB + xc < bi.p; };
    if (nct > 0) load_tile(0, l);
    typename P::U xb = nct > 0 && x_in(0) ? P::ld(gp + xc) : 0;
    for (int k = 0; k < nct; ++k) {
      const int c0 = k * NB, nc = min(NB, bi.p - c0);
      if (k + 1 < nct) load_tile(k + 1, ln);
      wait_published<T>(xb, gp + c0 + xc, x_in(k), err);
      const T xk = P::val(xb);
      if (k + 1 < nct && x_in(k + 1)) xb = P::ld(gp + c0 + NB + xc);
#pragma unroll
      for (int j = 0; j < kJC; ++j) {
        const T xv = __shfl_sync(0xffffffffu, xk, j);
        if (q + kQL * j < nc) {
          if (j & 1)
            acc1 = fma(l[j], xv, acc1);
          else
            acc0 = fma(l[j], xv, acc0);
        }
      }
#pragma unroll
      for (int j = 0; j < kJC; ++j) l[j] = ln[j];
    }
  }
  cp_async_wait<0>();
  auto sum_lanes = [&](int t) {
    if constexpr (sizeof(T) == sizeof(double)) {   // a chain of eight additions is 512 clocks
      static_assert(kQL == 8, "eight column lanes");
      return ((red[0][t] + red[1][t]) + (red[2][t] + red[3][t])) +
             ((red[4][t] + red[5][t]) + (red[6][t] + red[7][t]));
    } else {
      T s = T(0);
#pragma unroll
      for (int i = 0; i < kQL; ++i) s += red[i][t];
      return s;
    }
  };
  red[q][rho] = acc0 + acc1;
  __syncthreads();
  if (threadIdx.x < nr) u[threadIdx.x] = (T)rhs_r - sum_lanes(threadIdx.x);
  __syncthreads();
  if (pivtile) {
    // pivot rows: x = L_rr^-1 u
    T s = T(0);
    if (rho < npiv) {
#pragma unroll
      for (int j = 0; j < kJC; ++j) {
        const int c = q + kQL * j;
        if (c < npiv) s = fma(Xs[c * NB + rho], u[c], s);
      }
    }
    red[q][rho] = s;
    __syncthreads();
    if (threadIdx.x < npiv) {
      const T x = sum_lanes(threadIdx.x);
      P::st(gp + r0 + threadIdx.x, x);
      xs[threadIdx.x] = x;
      if constexpr (sizeof(T) != sizeof(double)) gv[r0 + threadIdx.x] = (double)x;
    }
    if (npiv < nr) {
      // non-pivot rows of the last pivot tile: u -= L(rows, pivots) x
      __syncthreads();
      T s2 = T(0);
      if (rho >= npiv && rho < nr) {
#pragma unroll
        for (int j = 0; j < kJC; ++j) {
          const int c = q + kQL * j;
          if (c < npiv) s2 = fma(Xs[c * NB + rho], xs[c], s2);
        }
      }
      red[q][rho] = s2;
      __syncthreads();
      if (threadIdx.x >= npiv && threadIdx.x < nr)
        gv[r0 + threadIdx.x] = (double)(u[threadIdx.x] - sum_lanes(threadIdx.x));
    }
  } else if (threadIdx.x < nr) {
    gv[r0 + threadIdx.x] = (double)u[threadIdx.x];
  }
}

// the backward solve's ends: the Schur solution it reads (its non-pivot rows
// through the block's index map) and dy = [block rows, link rows, global rows];
// the forward solution of the first `neg` rows counts with its sign changed (the
// border, whose x_0 part is negative definite)
struct TrsvBwdIO {
  const double *svec;
  const int *kmap;
  const long long *kmap_off, *yoff;
  double *dy;
  long long msum;
  int nl, n0, mg, neg;
};

// vec holds the forward solution; pub is the publication buffer (its pivot rows)
template <typename T>
__global__ void __launch_bounds__(TrsvCfg<T, true>::threads, TrsvCfg<T, true>::min_ctas)
    trsv_bwd_kernel(const T *buf, const T *tinv,
                    const BlkInfo *__restrict__ blk, const int *__restrict__ sched, int *ticket,
                    int *err, const double *vec, T *pub, const TrsvBwdIO io) {
  pdl_begin();
  using P = PubBits<T>;
  constexpr int kQL = TrsvCfg<T, true>::ql, kJC = TrsvCfg<T, true>::jc;
  static_assert(kJC == 8, "eight sums per thread");
  __shared__ __align__(16) T Xs[NB * NB];      // column-major, Xs[c * NB + r]
  __shared__ T red[TrsvCfg<T, true>::threads / 32][kJC];
  __shared__ T u[NB];
  __shared__ int s_job;
  if (threadIdx.x == 0) s_job = atomicAdd(ticket, 1);
  __syncthreads();
  const int b = sched[2 * s_job], r = sched[2 * s_job + 1];   // r < Tp
  const BlkInfo bi = blk[b];
  const T *L = buf + bi.base;
  const long long lda = bi.lda;
  T *gp = pub + bi.voff;
  const int r0 = r * NB, nr = min(NB, bi.a - r0), npiv = min(NB, bi.p - r0);
  const int *km = io.kmap + io.kmap_off[b] - bi.p;
  // the link and global rows of dy, shared out over the CTAs
  for (int q = s_job * (int)blockDim.x + threadIdx.x; q < io.nl + io.mg;
       q += (int)gridDim.x * (int)blockDim.x)
    io.dy[io.msum + q] = io.svec[q < io.nl ? q : q + io.n0];
  // lane q dots the tile's columns q, q + kQL, ... with the rows of each chunk
  const int rho = threadIdx.x & (NB - 1), q = threadIdx.x / NB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T *Lc = L + (long long)r0 * lda;
  // chunks of rows below the pivots, bottom first: non-pivot rows are inputs,
  // pivot tiles publish upwards.  Chunk r itself holds the non-pivot rows of
  // the last pivot tile (if any).
  const int kend = npiv < nr ? r : r + 1;
  const int nch = bi.T - kend;   // chunks, taken k = T - 1, T - 2, ..., kend
  stage_contiguous(Xs, tinv + bi.ioff + (long long)r * NB * NB, NB * NB);
  cp_async_commit();
  double fwd_r = threadIdx.x < npiv ? vec[bi.voff + r0 + threadIdx.x] : 0.0;
  if (r0 + (int)threadIdx.x < io.neg) fwd_r = -fwd_r;
  T acc[kJC];
#pragma unroll
  for (int j = 0; j < kJC; ++j) acc[j] = T(0);
  {
    T l[kJC], ln[kJC];
    auto load_chunk = [&](int k, T(&dst)[kJC]) {
      const int row = k * NB + rho;
      const bool ok = row < bi.a && (k > r || rho >= npiv);
#pragma unroll
      for (int j = 0; j < kJC; ++j) {
        const int c = q + kQL * j;
        dst[j] = (ok && c < npiv) ? Lc[(long long)c * lda + row] : T(0);
      }
    };
    // a solved entry: a pivot row another CTA publishes, or a Schur unknown
    auto x_in = [&](int k) { return k > r && k * NB + rho < bi.p; };
    auto x_ld = [&](int k) -> typename P::U {
      const int row = k * NB + rho;
      if (x_in(k)) return P::ld(gp + row);
      typename P::U v = 0;
      if (row >= bi.p && row < bi.a) {
        const T x = (T)io.svec[km[row]];
        memcpy(&v, &x, sizeof v);
      }
      return v;
    };
    typename P::U xb = 0;
    if (nch > 0) {
      load_chunk(bi.T - 1, l);
      xb = x_ld(bi.T - 1);
    }
    for (int k = bi.T - 1; k >= kend; --k) {
      if (k - 1 >= kend) load_chunk(k - 1, ln);
      wait_published<T>(xb, gp + k * NB + rho, x_in(k), err);
      const T xv = P::val(xb);
      if (k - 1 >= kend) xb = x_ld(k - 1);
#pragma unroll
      for (int j = 0; j < kJC; ++j) acc[j] = fma(l[j], xv, acc[j]);
#pragma unroll
      for (int j = 0; j < kJC; ++j) l[j] = ln[j];
    }
  }
  cp_async_wait<0>();
  // column c = q + kQL j is summed over the two warps of lane q
  auto col_sum = [&](int c) {
    const int cq = c % kQL, cj = c / kQL;
    return red[2 * cq][cj] + red[2 * cq + 1][cj];
  };
  const int si = warp_sum8_index(lane);
  {
    const T s = warp_sum8(acc, lane);
    if ((lane & 3) == 0) red[warp][si] = s;
  }
  __syncthreads();
  if (threadIdx.x < npiv) u[threadIdx.x] = (T)fwd_r - col_sum(threadIdx.x);
  __syncthreads();
  // x = L_rr^-T u: column c = q + kQL j collects X(rho, c) u(rho) over the rows
  const T uv = rho < npiv ? u[rho] : T(0);
#pragma unroll
  for (int j = 0; j < kJC; ++j) acc[j] = (rho < npiv) ? Xs[(q + kQL * j) * NB + rho] * uv : T(0);
  {
    const T s = warp_sum8(acc, lane);
    if ((lane & 3) == 0) red[warp][si] = s;
  }
  __syncthreads();
  if (threadIdx.x < npiv) {
    const T x = col_sum(threadIdx.x);
    P::st(gp + r0 + threadIdx.x, x);
    io.dy[io.yoff[b] + r0 + threadIdx.x] = (double)x;
  }
}

void launch_trsm64(int lanes, double *buf, const BlkInfo *info, unsigned panels, int nblk, int k,
                   ahlp_problem *dz, cudaStream_t s) {
  auto *const kern = lanes == 8   ? pchol_trsm_kernel<8>
                     : lanes == 4 ? pchol_trsm_kernel<4>
                                  : pchol_trsm_kernel<2>;
  const unsigned ctas = panels * (NB / (kTrsmThreads / lanes));
  count_launch(), launch_pdl(kern, dim3(ctas, nblk), kTrsmThreads, kTrsmSmem, s, buf, info, k,
                             dz ? dz->dz_stage : nullptr, dz ? dz->dz_exp : nullptr,
                             dz ? dz->stage_slots : 0);
}

template <typename T>
cudaError_t pchol_t(T *buf, T *tinv, const BlkInfo *info, const std::vector<BlkInfo> &h,
                    const double *diag0, double tol, int *status, cudaStream_t s,
                    ahlp_problem *tc = nullptr, ahlp_problem *prof = nullptr,
                    double drop = 0.0, ahlp_problem *dz = nullptr) {
  int nblk = (int)h.size();
  if (nblk == 0) return cudaSuccess;
  int maxTp = 0;
  for (auto &b : h) maxTp = b.Tp > maxTp ? b.Tp : maxTp;
  LookAhead la;   // this step's diagonal tiles, beside the update before
  for (int k = 0; k < maxTp; ++k) {
    LookAhead next;
    long long maxPanel = 0, maxTrail = 0, panels = 0, trails = 0;
    for (auto &b : h) {
      if (k >= b.Tp) continue;
      long long t = b.T - k - 1;
      panels += t;
      trails += t * (t + 1) / 2;
      if (t > maxPanel) maxPanel = t;
      if (t * (t + 1) / 2 > maxTrail) maxTrail = t * (t + 1) / 2;
    }
    if constexpr (sizeof(T) == sizeof(float)) {
      if (prof) kt_mark(prof, 0, s);
      count_launch(), launch_pdl(pchol_potrf_f32_kernel, nblk, kPotrf32Threads, 0, s, buf, tinv,
                                 info, k, diag0, (float)tol, status, (float)drop, la);
      if (prof) kt_mark(prof, 1, s);
      if (maxPanel > 0)
        count_launch(), launch_pdl(pchol_trsm_inv_kernel, dim3((unsigned)maxPanel, nblk),
                                   kThreads, 0, s, buf, tinv, info, k,
                                   tc ? tc->pstage : nullptr);
    } else {
      if (prof) kt_mark(prof, 0, s);
      count_launch(), launch_pdl(pchol_potrf_kernel<false, double>, nblk, kThreads,
                                 la.ready ? kDiagPad : 0, s, buf,
                                 nullptr, info, k, diag0, tol, status, drop, la);
      if (prof) kt_mark(prof, 1, s);
      if (maxPanel > 0)
        launch_trsm64(trsm_lanes(panels), buf, info, (unsigned)maxPanel, nblk, k, dz, s);
    }
    if (prof) kt_mark(prof, 2, s);
    if (maxTrail > 0) {
      if constexpr (sizeof(T) == sizeof(float)) {
        if (tc) {
          cudaError_t e = launch_update_tc(tc, k, s, &next);
          if (e != cudaSuccess) return e;
        } else {
          count_launch(), launch_pdl(pchol_update_f32_kernel, dim3((unsigned)maxTrail, nblk),
                                     kUpdF32Threads, 0, s, buf, info, k);
        }
      } else if (dz) {
        cudaError_t e = launch_update_dz(dz, k, s, &next);
        if (e != cudaSuccess) return e;
      } else {
        auto *const kern = trails <= kSMs / 8 ? pchol_update_kernel<T, 4>
                           : trails <= kSMs   ? pchol_update_kernel<T, 2>
                                              : pchol_update_kernel<T, 1>;
        const unsigned sub = trails <= kSMs / 8 ? 16 : trails <= kSMs ? 4 : 1;
        count_launch(), launch_pdl(kern, dim3((unsigned)maxTrail * sub, nblk), kThreads, 0, s, buf,
                                   info, k);
      }
    }
    if (prof) kt_mark(prof, 3, s);
    la = next;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

// ---------------------------------------------------------------------------
cudaError_t launch_dscale(ahlp_problem *p) {
  count_launch(), launch_pdl(dscale_kernel, (unsigned)((std::max(p->n, 8LL) + 255) / 256), 256, 0,
                             p->stream, p->x, p->z, p->dscale, p->xinv, p->wfin, p->n,
                             p->fac_rho_x, p->fac_rho, p->is_x0, p->status, p->cdiag0,
                             p->cdiag_elems, p->la_ready, p->la_elems);
  return cudaGetLastError();
}

cudaError_t launch_form(ahlp_problem *p, double delta) {
  if (p->ntiles <= 0) return cudaSuccess;
  if (p->fac_prec == kPrecFP32) {
    FormArgs<float> A{nullptr, p->ftiles, p->tile_ent, p->ent_pos, p->ent_cb, p->con_idx,
                      p->con_coef, p->dscale, p->blk, p->aug32, p->diag0, p->cdiag0, delta};
    count_launch(), launch_pdl(form_aug_kernel<float, false>, (unsigned)p->ntiles, kThreads, 0,
                               p->stream, A);
  } else if (p->fac_prec == kPrecFF) {
    FormArgs<float> A{p->aug_lo, p->ftiles, p->tile_ent, p->ent_pos, p->ent_cb, p->con_idx,
                      p->con_coef, p->dscale, p->blk, p->aug32, p->diag0, p->cdiag0, delta};
    count_launch(), launch_pdl(form_aug_kernel<float, true>, (unsigned)p->ntiles, kThreads, 0,
                               p->stream, A);
  } else {
    FormArgs<double> A{nullptr, p->ftiles, p->tile_ent, p->ent_pos, p->ent_cb, p->con_idx,
                       p->con_coef, p->dscale, p->blk, p->aug, p->diag0, p->cdiag0, delta};
    count_launch(), launch_pdl(form_aug_kernel<double, false>, (unsigned)p->ntiles, kThreads, 0,
                               p->stream, A);
  }
  return cudaGetLastError();
}

cudaError_t launch_pchol_ff(float *hi, float *lo, double *out, long long elems,
                            const BlkInfo *info, const std::vector<BlkInfo> &h,
                            const double *diag0, double tol, int *status, cudaStream_t s,
                            ahlp_problem *oz, ahlp_problem *prof, double drop) {
  int nblk = (int)h.size();
  if (nblk == 0) return cudaSuccess;
  int maxTp = 0;
  for (auto &b : h) maxTp = b.Tp > maxTp ? b.Tp : maxTp;
  LookAhead la;   // this step's diagonal tiles, beside the update before
  for (int k = 0; k < maxTp; ++k) {
    LookAhead next;
    long long maxPanel = 0, maxTrail = 0;
    for (auto &b : h) {
      if (k >= b.Tp) continue;
      long long t = b.T - k - 1;
      if (t > maxPanel) maxPanel = t;
      if (t * (t + 1) / 2 > maxTrail) maxTrail = t * (t + 1) / 2;
    }
    if (prof) kt_mark(prof, 0, s);
    count_launch(), launch_pdl(pchol_potrf_kernel<true, float>, nblk, kThreads,
                               la.ready ? kDiagPad : 0, s, hi, lo, info,
                               k, diag0, tol, status, drop, la);
    if (prof) kt_mark(prof, 1, s);
    if (maxPanel > 0)
      count_launch(), launch_pdl(pchol_trsm_ff_kernel,
                                 dim3((unsigned)((maxPanel + kFFRowTiles - 1) / kFFRowTiles), nblk),
                                 kFFRowThreads, kTrsmFFSmem, s, hi, lo, info, k,
                                 oz ? oz->dstage : nullptr, oz ? oz->dexp : nullptr);
    if (prof) kt_mark(prof, 2, s);
    if (maxTrail > 0) {
      if (oz) {
        cudaError_t e = launch_update_oz(oz, k, s, &next);
        if (e != cudaSuccess) return e;
      } else {
        count_launch(), launch_pdl(pchol_update_ff8_kernel, dim3((unsigned)maxTrail, nblk),
                                   kUpdFFThreads, kUpdFFSmem, s, hi, lo, info, k);
      }
    }
    if (prof) kt_mark(prof, 3, s);
    la = next;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (elems > 0)
    count_launch(), launch_pdl(ff_expand_kernel, 152 * 8, 256, 0, s, hi, lo, out, elems);
  return cudaGetLastError();
}

cudaError_t launch_pchol(double *buf, const BlkInfo *info, const std::vector<BlkInfo> &h,
                         const double *diag0, double tol, int *status, cudaStream_t s,
                         ahlp_problem *prof, double drop, ahlp_problem *dz) {
  return pchol_t<double>(buf, nullptr, info, h, diag0, tol, status, s, nullptr, prof, drop, dz);
}

cudaError_t launch_pchol_f32(float *buf, float *tinv, const BlkInfo *info,
                             const std::vector<BlkInfo> &h, const double *diag0, double tol,
                             int *status, cudaStream_t s, ahlp_problem *tc,
                             ahlp_problem *prof, double drop) {
  return pchol_t<float>(buf, tinv, info, h, diag0, tol, status, s, tc, prof, drop);
}

__global__ void schur_dy_kernel(const TrsvBwdIO io) {
  pdl_begin();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < io.nl + io.mg) io.dy[io.msum + q] = io.svec[q < io.nl ? q : q + io.n0];
}

cudaError_t launch_trsv(ahlp_problem *p, bool forward, const double *rhs, double *dy) {
  const int njobs = forward ? p->trsv_nf : p->trsv_nb;
  cudaStream_t s = p->stream;
  int *ticket = p->trsv_ticket + (forward ? 0 : 1);
  const int *sched = forward ? p->trsv_fsched : p->trsv_bsched;
  const TrsvBwdIO io{p->svec, p->kmap, p->kmap_off_d, p->yoff_d, dy, p->msum, p->nl, p->n0, p->mg,
                     0};
  if (njobs == 0) {
    if (!forward && p->nl + p->mg > 0)
      count_launch(), launch_pdl(schur_dy_kernel, (p->nl + p->mg + 255) / 256, 256, 0, s, io);
    return cudaGetLastError();
  }
  if (p->fac_prec == kPrecFP32) {
    float *pubb = reinterpret_cast<float *>(p->vecb);
    if (forward)
      count_launch(), launch_pdl(trsv_fwd_kernel<float>, njobs, TrsvCfg<float, false>::threads, 0,
                                 s, p->aug32, p->tinv32, p->blk, sched, ticket, p->trsv_err,
                                 p->vec, p->vec32, rhs, p->yoff_d);
    else
      count_launch(), launch_pdl(trsv_bwd_kernel<float>, njobs, TrsvCfg<float, true>::threads, 0,
                                 s, p->aug32, p->tinv32, p->blk, sched, ticket, p->trsv_err,
                                 p->vec, pubb, io);
  } else {
    if (forward)
      count_launch(), launch_pdl(trsv_fwd_kernel<double>, njobs, TrsvCfg<double, false>::threads,
                                 0, s, p->aug, p->tinv, p->blk, sched, ticket, p->trsv_err, p->vec,
                                 p->vec, rhs, p->yoff_d);
    else
      count_launch(), launch_pdl(trsv_bwd_kernel<double>, njobs, TrsvCfg<double, true>::threads, 0,
                                 s, p->aug, p->tinv, p->blk, sched, ticket, p->trsv_err, p->vec,
                                 p->vecb, io);
  }
  return cudaGetLastError();
}

// The border solve, in place on svec's border part.  With L the factor of the border
// (x_0 pivots first, then y_g) and J = diag(-I, I), the solution is L^-T J L^-1 b:
// the wavefront sweeps of the blocks on one more factor, a chain of B / 64 tiles on as
// many SMs, 8 us at order 100 and 100 us at 601 for both sweeps (substitution over all
// of L on one SM: 106 and 349 us).  An explicit inverse of L (two matrix-vector products
// over many SMs, 16 us at 601) is not used: its residual was ten times substitution's
// and grew with the order, which cost Krylov steps at ill-conditioned borders (order
// 420, D over 20 decades: 19 steps against 14), and its B^3 / 3 multiply-adds made the
// factor slower than the sweeps' gain from about order 700 on (4096: 54 against 29 ms).
//
// One tile: two products with its inverse X (column-major), t = J X b and x = X' t, one
// warp per entry over several CTAs: 5 us, where the sweeps' kernels take 8.
__global__ void __launch_bounds__(256) border_tile_kernel(const double *X, int B, int n0,
                                                          const double *in, double *out, int fwd) {
  pdl_begin();
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= B) return;
  const int q0 = (fwd ? 0 : i) + lane, q1 = fwd ? i + 1 : B;
  auto x = [&](int q) { return fwd ? X[q * NB + i] : X[i * NB + q]; };
  const double s0 = q0 < q1 ? x(q0) * in[q0] : 0.0;
  const double s1 = q0 + 32 < q1 ? x(q0 + 32) * in[q0 + 32] : 0.0;
  double s = s0 + s1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) out[i] = fwd && i < n0 ? -s : s;
}

cudaError_t launch_border_solve(ahlp_problem *p) {
  const int T = (p->B + NB - 1) / NB;
  double *sb = p->svec + p->nl, *y = p->border_pub, *u = y + p->B;
  if (T == 1) {
    const unsigned ctas = (unsigned)(p->B + 7) / 8;
    count_launch(), launch_pdl(border_tile_kernel, ctas, 256, 0, p->stream, p->border_tinv, p->B,
                               p->n0, sb, y, 1);
    count_launch(), launch_pdl(border_tile_kernel, ctas, 256, 0, p->stream, p->border_tinv, p->B,
                               p->n0, y, sb, 0);
    return cudaGetLastError();
  }
  int *ticket = p->trsv_ticket + 4;
  const TrsvBwdIO io{nullptr, p->kmap, p->bw_zero, p->bw_zero, sb, 0, 0, 0, 0, p->n0};
  count_launch(), launch_pdl(trsv_fwd_kernel<double>, T, TrsvCfg<double, false>::threads, 0,
                             p->stream, p->border, p->border_tinv, p->bw_info, p->bw_sched, ticket,
                             p->trsv_err, y, y, sb, p->bw_zero);
  count_launch(), launch_pdl(trsv_bwd_kernel<double>, T, TrsvCfg<double, true>::threads, 0,
                             p->stream, p->border, p->border_tinv, p->bw_info,
                             p->bw_sched + 2 * T, ticket + 1, p->trsv_err, y, u, io);
  return cudaGetLastError();
}

cudaError_t launch_tinv(ahlp_problem *p) {
  // FP32 factors write their inverse tiles in pchol_potrf_f32_kernel; FP64 and
  // float-float factors (through their FP64 copy) get them here
  if (p->trsv_nb == 0 || p->fac_prec == kPrecFP32) return cudaSuccess;
  count_launch(), launch_pdl(tinv_kernel, p->trsv_nb, kThreads, kTinvSmem, p->stream, p->aug,
                             p->tinv, p->blk, p->trsv_bsched);
  return cudaGetLastError();
}

cudaError_t launch_tile_inverses(const double *buf, double *tinv, const BlkInfo *info,
                                 const int *sched, int njobs, cudaStream_t s) {
  if (njobs > 0)
    count_launch(), launch_pdl(tinv_kernel, njobs, kThreads, kTinvSmem, s, buf, tinv, info, sched);
  return cudaGetLastError();
}

cudaError_t set_dense_smem_limits() {
  cudaError_t e = cudaFuncSetAttribute(pchol_potrf_kernel<false, double>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kDiagPad);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(pchol_potrf_kernel<true, float>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, kDiagPad);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(tinv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kTinvSmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(pchol_update_ff8_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kUpdFFSmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(pchol_trsm_ff_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kTrsmFFSmem);
  if (e != cudaSuccess) return e;
  return e;
}

}  // namespace ahlp
