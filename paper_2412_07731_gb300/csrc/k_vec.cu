// Vector kernels of the IPM: sparse mat-vecs, deterministic reductions and
// elementwise updates.  All bandwidth-bound FP64.
#include <algorithm>

#include "ahlp_internal.h"

namespace ahlp {

namespace {

constexpr int kRedBlocks = 304;   // 2 x 152 SMs, fixed so sums are reproducible
constexpr int kRedThreads = 256;
constexpr int kMdotBlocks = kMdotParts;   // 4 x 152 SMs
constexpr int kMaxpyBlocks = 2432;        // 16 x 152 SMs (partial sums fit red_part)
static_assert(kMaxpyBlocks <= kRedSetMax * kRedBlocks, "partial sums");

struct RedArgs {
  int op;
  const double *a, *b, *c, *d;
  double s1, s2;
  long long len;
};

__device__ __forceinline__ double red_identity(int op) {
  return (op == RED_MAXABS) ? 0.0 : ((op == RED_MINSTEP || op == RED_MIN) ? 1e300 : 0.0);
}

__device__ __forceinline__ double red_combine(int op, double u, double v) {
  switch (op) {
    case RED_MAXABS: return fmax(u, v);
    case RED_MINSTEP:
    case RED_MIN: return fmin(u, v);
    default: return u + v;
  }
}

template <int OP>
__device__ __forceinline__ double red_elem(const RedArgs &r, long long i) {
  if constexpr (OP == RED_DOT) return r.a[i] * r.b[i];
  if constexpr (OP == RED_MAXABS) return fabs(r.a[i]);
  if constexpr (OP == RED_MINSTEP) {   // largest step keeping a + t b >= 0
    const double bi = r.b[i];
    return bi < 0.0 ? -r.a[i] / bi : 1e300;
  }
  if constexpr (OP == RED_STEP) return (r.a[i] + r.s1 * r.b[i]) * (r.c[i] + r.s2 * r.d[i]);
  return r.a[i];
}

template <int OP>
__device__ __forceinline__ double red_range(const RedArgs &r, long long i0, long long stride) {
  double acc = red_identity(OP);
#pragma unroll 4
  for (long long i = i0; i < r.len; i += stride) acc = red_combine(OP, acc, red_elem<OP>(r, i));
  return acc;
}

// sum (or min, max) over a CTA of kRedThreads, valid in thread 0
__device__ __forceinline__ double cta_reduce(int op, double v, double *sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = red_combine(op, v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = sh[threadIdx.x & (kRedThreads / 32 - 1)];
#pragma unroll
    for (int o = kRedThreads / 64; o > 0; o >>= 1)
      v = red_combine(op, v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}

// CTAs of a reduction over len entries, one entry per thread up to cap: a
// function of len alone, so that sums are reproducible; a short vector takes
// one CTA and no second phase
inline int red_blocks(long long len, int cap) {
  return (int)std::max<long long>(
      1, std::min<long long>((len + kRedThreads - 1) / kRedThreads, cap));
}

// true in every thread of the CTA that arrives last of n at *cnt (reset for the
// next use); what the others wrote before is visible to it
__device__ __forceinline__ bool last_cta(int *cnt, int n) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const int t = atomicAdd(cnt, 1);
    s_last = t == n - 1;
    if (t == n - 1) *cnt = 0;
    __threadfence();
  }
  __syncthreads();
  return s_last != 0;
}

// Several reductions in one launch (blockIdx.y), each finished by its last CTA
// in a fixed order.  A reduction is a few microseconds of latency whatever its
// length, so one launch for all the norms of a step, and no second launch to
// add the partial sums, is what counts here.
struct RedSet {
  RedArgs r[kRedSetMax];
  double *out[kRedSetMax];
  int nb[kRedSetMax];
};

__global__ void __launch_bounds__(kRedThreads) reduce_set_kernel(const RedSet S, double *part,
                                                                 int *cnt) {
  pdl_begin();
  __shared__ double sh[kRedThreads / 32];
  const RedArgs &r = S.r[blockIdx.y];
  const int nb = S.nb[blockIdx.y];
  if ((int)blockIdx.x >= nb) return;
  const long long stride = (long long)nb * blockDim.x;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  double acc = r.op == RED_DOT       ? red_range<RED_DOT>(r, i0, stride)
               : r.op == RED_MAXABS  ? red_range<RED_MAXABS>(r, i0, stride)
               : r.op == RED_MINSTEP ? red_range<RED_MINSTEP>(r, i0, stride)
               : r.op == RED_MIN     ? red_range<RED_MIN>(r, i0, stride)
               : r.op == RED_SUM     ? red_range<RED_SUM>(r, i0, stride)
                                     : red_range<RED_STEP>(r, i0, stride);
  double v = cta_reduce(r.op, acc, sh);
  if (nb > 1) {
    double *pp = part + (long long)blockIdx.y * kRedBlocks;
    if (threadIdx.x == 0) pp[blockIdx.x] = v;
    if (!last_cta(cnt + blockIdx.y, nb)) return;
    acc = red_identity(r.op);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc = red_combine(r.op, acc, __ldcg(pp + i));
    v = cta_reduce(r.op, acc, sh);
  }
  if (threadIdx.x == 0) *S.out[blockIdx.y] = v;
}

// --------------------------------------------------------------------------
// sparse products y[r] = yadd[r] + alpha * sum_k v[k] x[ci[k]]
//
// Rows of up to kShortRow entries: a warp takes 32 rows, eight lanes per row
// and four rows at a time.  The first eight entries of all 32 rows are
// requested before any is used, and the eight partial sums a lane ends up with
// (its share of the rows 8g .. 8g+7 of its group g) are added across the group
// by a transposing exchange: 7 FP64 additions per 32 rows instead of 24, and
// lane l is left with row l, so what follows a row (the direction's dx and dz,
// the residual) runs on full warps.  FP64 instructions bound the product at
// size (one warp instruction in 19 clocks per SM): 23.8 -> 12 us for 192 k rows
// of nine entries.  Longer rows (the linking variables) take one CTA each, in
// the same launch.
// --------------------------------------------------------------------------
constexpr int kRowLanes = 8;
constexpr int kSpThreads = 256;

struct SpSeg {
  const int *rp, *ci;
  const double *v;
  long long rows;
  const int *long_rows;
  int n_long;
  const double *x, *yadd;   // yadd may be null
  double *y;
  double alpha;
};

// what is done with row i's value (yadd + alpha * sum)
enum SpTail { SP_STORE = 0, SP_FINISH = 1, SP_RESID = 2 };
struct SpTailArgs {
  // SP_FINISH: dx, dz of the direction from val = (A'dy)_i, and with wx / wc
  // the Newton product's first and third parts of (dx, dy, dz)
  const double *f, *w, *xinv, *z, *x, *rc;
  double *dx, *dz, *wx, *wc;
  // SP_RESID: e_c and the dz term of e_d (val = r_d - A'dy)
  const double *ddx, *ddz;
  double *e_c;
  int adjoint;
};

template <int TAIL>
__device__ __forceinline__ void sp_tail(const SpSeg &S, const SpTailArgs &T, long long i,
                                        double val) {
  if constexpr (TAIL == SP_FINISH) {
    // dx = (A'dy - f) / (D^-1 + rho on the linking variables), dz from dx; w
    // and xinv are those quotients' reciprocals, taken once per factor point
    const double zi = T.z[i], rci = T.rc[i], xi = T.xinv[i];
    const double dxi = (val - T.f[i]) * T.w[i];
    const double dzi = T.adjoint ? (rci - dxi) * xi : (rci - zi * dxi) * xi;
    T.dx[i] = dxi;
    T.dz[i] = dzi;
    if (T.wx) {   // J (dx, dy, dz) = (A'dy + dz, ., z dx + x dz), J' likewise
      const double xx = T.x[i];
      T.wx[i] = T.adjoint ? val + zi * dzi : val + dzi;
      T.wc[i] = T.adjoint ? dxi + xx * dzi : zi * dxi + xx * dzi;
    }
  } else if constexpr (TAIL == SP_RESID) {
    const double dzi = T.ddz[i], dxi = T.ddx[i], zi = T.z[i], xx = T.x[i];
    S.y[i] = T.adjoint ? val - zi * dzi : val - dzi;
    T.e_c[i] = T.adjoint ? T.rc[i] - dxi - xx * dzi : T.rc[i] - zi * dxi - xx * dzi;
  } else {
    S.y[i] = val;
  }
}

// one CTA per long row, fixed-order tree reduction
template <int TAIL>
__device__ __forceinline__ void sp_long(const SpSeg &S, const SpTailArgs &T, int which,
                                        double *part) {
  const int row = S.long_rows[which];
  const int k0 = S.rp[row], k1 = S.rp[row + 1];
  double s0 = 0.0, s1 = 0.0;
  int k = k0 + threadIdx.x;
#pragma unroll 4
  for (; k + 256 < k1; k += 512) {
    s0 = fma(S.v[k], S.x[S.ci[k]], s0);
    s1 = fma(S.v[k + 256], S.x[S.ci[k + 256]], s1);
  }
  if (k < k1) s0 = fma(S.v[k], S.x[S.ci[k]], s0);
  double s = s0 + s1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += part[w];
    sp_tail<TAIL>(S, T, row, (S.yadd ? S.yadd[row] : 0.0) + S.alpha * t);
  }
}

template <int TAIL>
__device__ __forceinline__ void sp_short(const SpSeg &S, const SpTailArgs &T, long long cta) {
  const int lane = threadIdx.x & 31, g8 = lane & ~7, l8 = lane & 7;
  const long long base = cta * kSpThreads + (threadIdx.x & ~31);
  if (base >= S.rows) return;   // whole warps leave together
  const long long row = base + lane;
  int a0 = 0, a1 = 0;
  if (row < S.rows) {
    a0 = S.rp[row];
    a1 = S.rp[row + 1];
  }
  const bool mine = row < S.rows && a1 - a0 <= kShortRow;
  if (!mine) a1 = a0;   // a long row: its own CTA
  int kk[8], ke[8];
  double s[8];
#pragma unroll
  for (int it = 0; it < 8; ++it) {   // row base + g8 + it
    kk[it] = __shfl_sync(0xffffffffu, a0, g8 + it) + l8;
    ke[it] = __shfl_sync(0xffffffffu, a1, g8 + it);
    s[it] = 0.0;
  }
  // eight entries of each of the 32 rows per round, all requested together
  const int rounds = (__reduce_max_sync(0xffffffffu, a1 - a0) + kRowLanes - 1) / kRowLanes;
  for (int rd = 0; rd < rounds; ++rd) {
    int cc[8];
    double vv[8];
#pragma unroll
    for (int it = 0; it < 8; ++it) {
      const bool in = kk[it] < ke[it];
      cc[it] = in ? S.ci[kk[it]] : -1;
      vv[it] = in ? S.v[kk[it]] : 0.0;
      kk[it] += kRowLanes;
    }
#pragma unroll
    for (int it = 0; it < 8; ++it) {
      // rows of the warp that have ended skip the FP64 instruction
      const double xv = cc[it] >= 0 ? S.x[cc[it]] : 0.0;
      if (__any_sync(0xffffffffu, cc[it] >= 0)) s[it] = fma(vv[it], xv, s[it]);
    }
  }
  // transposing sum over the group's eight lanes
  double h4[4], h2[2];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const double keep = (l8 & 4) ? s[u + 4] : s[u], give = (l8 & 4) ? s[u] : s[u + 4];
    h4[u] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const double keep = (l8 & 2) ? h4[u + 2] : h4[u], give = (l8 & 2) ? h4[u] : h4[u + 2];
    h2[u] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
  }
  const double keep = (l8 & 1) ? h2[1] : h2[0], give = (l8 & 1) ? h2[0] : h2[1];
  const double sum = keep + __shfl_xor_sync(0xffffffffu, give, 1);
  if (mine) sp_tail<TAIL>(S, T, row, (S.yadd ? S.yadd[row] : 0.0) + S.alpha * sum);
}

// product with one matrix (its rows' values through TAIL) and, with b.rows > 0,
// a second one stored plainly: CTAs [a's long rows | a's short | b's long | b's short]
template <int TAIL>
__global__ void __launch_bounds__(kSpThreads) spmv_kernel(const SpSeg a, const SpSeg b,
                                                          const SpTailArgs T) {
  pdl_begin();
  __shared__ double part[8];
  long long c = blockIdx.x;
  const long long na = (a.rows + kSpThreads - 1) / kSpThreads;
  if (c < a.n_long) return sp_long<TAIL>(a, T, (int)c, part);
  c -= a.n_long;
  if (c < na) return sp_short<TAIL>(a, T, c);
  c -= na;
  if (c < b.n_long) return sp_long<SP_STORE>(b, T, (int)c, part);
  sp_short<SP_STORE>(b, T, c - b.n_long);
}

__global__ void axpby_k(double *y, const double *x, double a, double b, long long n) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = a * x[i] + b * y[i];
}

__global__ void fill_k(double *y, double v, long long n) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = v;
}

__global__ void mul_k(double *y, const double *a, const double *b, double sc, long long n) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = sc * a[i] * b[i];
}

// r_c = sigma_mu - x z - dxa dza
__global__ void ipm_rc_k(double *rc, const double *x, const double *z, const double *dxa,
                         const double *dza, double smu, long long n) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) rc[i] = smu - x[i] * z[i] - (dxa ? dxa[i] * dza[i] : 0.0);
}

__global__ void centrality_rc_k(double *rc2, const double *rc, const double *x, const double *dx,
                                double ap, const double *z, const double *dz, double ad,
                                double lo, double hi, long long n) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = (x[i] + ap * dx[i]) * (z[i] + ad * dz[i]);
  double t = v < lo ? lo - v : (v > hi ? hi - v : 0.0);
  if (t < -hi) t = -hi;
  rc2[i] = rc[i] + t;
}

__global__ void add_scalar_k(double *y, const double *x, double s, long long n) {
  pdl_begin();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = x[i] + s;
}

// out[i] = <V_i, w> for i < k (vectors of length len, stride ld), eight vectors
// at a time: w is read once per eight, and the eight per-thread sums are added
// across a warp by a transposing exchange (9 FP64 additions instead of 40).
// The last CTA adds the partial sums in a fixed order.
__global__ void __launch_bounds__(kRedThreads) mdot_kernel(const double *V,
                                                           long long ld, int k,
                                                           const double *w,
                                                           long long len, double *part,
                                                           double *out, int *cnt) {
  pdl_begin();
  __shared__ double sh[8][kRedThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (int i0 = 0; i0 < k; i0 += 8) {
    double a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) a[u] = 0.0;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += stride) {
      const double we = w[e];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u < k) a[u] = fma(V[(long long)(i0 + u) * ld + e], we, a[u]);
    }
    double h4[4], h2[2];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const double keep = (lane & 16) ? a[u + 4] : a[u], give = (lane & 16) ? a[u] : a[u + 4];
      h4[u] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const double keep = (lane & 8) ? h4[u + 2] : h4[u], give = (lane & 8) ? h4[u] : h4[u + 2];
      h2[u] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
    const double keep = (lane & 4) ? h2[1] : h2[0], give = (lane & 4) ? h2[0] : h2[1];
    double t = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    // lanes with (lane & 3) == 0 hold vector 4 (lane>>4 & 1) + 2 (lane>>3 & 1) + (lane>>2 & 1)
    if ((lane & 3) == 0) sh[((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)][warp] = t;
    __syncthreads();
    if (threadIdx.x < 8 && i0 + (int)threadIdx.x < k) {
      double v = sh[threadIdx.x][0];
#pragma unroll
      for (int q = 1; q < kRedThreads / 32; ++q) v += sh[threadIdx.x][q];
      part[(long long)(i0 + threadIdx.x) * gridDim.x + blockIdx.x] = v;
    }
    __syncthreads();
  }
  if (!last_cta(cnt, gridDim.x)) return;
  for (int i = warp; i < k; i += kRedThreads / 32) {
    double v = 0.0;
    for (int q = lane; q < (int)gridDim.x; q += 32) v += __ldcg(part + (long long)i * gridDim.x + q);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) out[i] = v;
  }
}

// w[e] += sum_i coef[i] V_i[e], fixed order over i, for vectors in up to three
// pieces (w0, w1, w2 of lengths n0, n1 and the rest; V_i contiguous); the
// coefficients come from the device (coef, times sc) or by value.  With
// nrm2 the last CTA also leaves nrm2[0] = <w, w> and nrm2[1] = 1 / |w| (1 when
// <w, w> is not positive).
struct HostCoefs {
  double c[kMaxKrylov];
};

__global__ void __launch_bounds__(kRedThreads) maxpy_kernel(const double *V, long long ld, int k,
                                                            const double *coef, double sc,
                                                            const HostCoefs hc, double *w0,
                                                            long long n0, double *w1,
                                                            long long n1, double *w2,
                                                            long long len, double *part,
                                                            double *nrm2, int *cnt) {
  pdl_begin();
  __shared__ double cs[kMaxKrylov + 1];
  __shared__ double sh[kRedThreads / 32];
  for (int i = threadIdx.x; i < k; i += blockDim.x) cs[i] = coef ? sc * coef[i] : hc.c[i];
  __syncthreads();
  const long long stride = (long long)gridDim.x * blockDim.x;
  double q = 0.0;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += stride) {
    double *w = e < n0 ? w0 + e : e < n0 + n1 ? w1 + (e - n0) : w2 + (e - n0 - n1);
    double acc = *w;
#pragma unroll 8
    for (int i = 0; i < k; ++i) acc = fma(cs[i], V[(long long)i * ld + e], acc);
    *w = acc;
    if (nrm2) q = fma(acc, acc, q);
  }
  if (!nrm2) return;
  double v = cta_reduce(RED_DOT, q, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = v;
  if (!last_cta(cnt, gridDim.x)) return;
  double a = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) a += __ldcg(part + i);
  v = cta_reduce(RED_DOT, a, sh);
  if (threadIdx.x == 0) {
    nrm2[0] = v;
    nrm2[1] = v > 0.0 ? 1.0 / sqrt(v) : 1.0;
  }
}

__global__ void publish_k(const unsigned *src, unsigned *dst, int n, const unsigned *src2,
                          unsigned *dst2, int n2, unsigned *seq, unsigned val) {
  pdl_begin();
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
  for (int i = threadIdx.x; i < n2; i += blockDim.x) dst2[i] = src2[i];
  __threadfence_system();
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence_system();
    *reinterpret_cast<volatile unsigned *>(seq) = val;
  }
}

__global__ void copies_k(const CopySet c) {
  pdl_begin();
  const double *src = c.src[blockIdx.y];
  double *dst = c.dst[blockIdx.y];
  const long long n = c.n[blockIdx.y], stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    dst[i] = src[i];
}

// y = a x, a on the device (da) or not
__global__ void scale_k(double *y, const double *x, const double *da, double a, long long n) {
  pdl_begin();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = (da ? *da : a) * x[i];
}

inline unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_mdot(ahlp_problem *p, const double *V, long long ld, int k, const double *w,
                        long long len, double *out) {
  if (k <= 0) return cudaSuccess;
  count_launch(), launch_pdl(mdot_kernel, red_blocks(len, kMdotBlocks), kRedThreads, 0, p->stream,
                             V, ld, k, w, len, p->mdot_part, out, p->red_cnt + kRedSetMax);
  return cudaGetLastError();
}

cudaError_t launch_maxpy(ahlp_problem *p, const double *V, long long ld, int k, const double *coef,
                         double *w, long long len, double sign, double *nrm2) {
  if (k <= 0 || len <= 0) return cudaSuccess;
  count_launch(), launch_pdl(maxpy_kernel, red_blocks(len, kMaxpyBlocks), kRedThreads, 0,
                             p->stream, V, ld, k, coef, sign, HostCoefs{}, w, len, w, 0, w, len,
                             p->red_part, nrm2, p->red_cnt + kRedSetMax + 1);
  return cudaGetLastError();
}

cudaError_t launch_maxpy3(ahlp_problem *p, const double *V, long long ld, int k,
                          const double *coef, double *w0, long long n0, double *w1, long long n1,
                          double *w2, long long len) {
  if (k <= 0 || len <= 0) return cudaSuccess;
  HostCoefs hc{};
  for (int i = 0; i < k; ++i) hc.c[i] = coef[i];
  count_launch(), launch_pdl(maxpy_kernel, red_blocks(len, kMaxpyBlocks), kRedThreads, 0,
                             p->stream, V, ld, k, nullptr, 1.0, hc, w0, n0, w1, n1, w2, len,
                             p->red_part, nullptr, p->red_cnt + kRedSetMax + 1);
  return cudaGetLastError();
}

cudaError_t launch_publish(const unsigned *src, unsigned *dst, int n, const unsigned *src2,
                           unsigned *dst2, int n2, unsigned *seq, unsigned val, cudaStream_t s) {
  count_launch(), launch_pdl(publish_k, 1, 64, 0, s, src, dst, n, src2, dst2, n2, seq, val);
  return cudaGetLastError();
}

cudaError_t launch_copies(const CopySet &c, cudaStream_t s) {
  const long long n = std::max(std::max(c.n[0], c.n[1]), std::max(c.n[2], c.n[3]));
  if (n <= 0) return cudaSuccess;
  const unsigned g = (unsigned)std::min<long long>((n + 255) / 256, 1216);
  count_launch(), launch_pdl(copies_k, dim3(g, 4), 256, 0, s, c);
  return cudaGetLastError();
}

cudaError_t launch_scale(double *y, const double *x, const double *da, double a, long long len,
                         cudaStream_t s) {
  if (len <= 0) return cudaSuccess;
  count_launch(), launch_pdl(scale_k, blocks_for(len, 256), 256, 0, s, y, x, da, a, len);
  return cudaGetLastError();
}

cudaError_t launch_add_scalar(double *y, const double *x, double s, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launch(), launch_pdl(add_scalar_k, blocks_for(n, 256), 256, 0, st, y, x, s, n);
  return cudaGetLastError();
}

cudaError_t launch_reduce_set(ahlp_problem *p, const RedOne *ops, int n) {
  for (int i0 = 0; i0 < n; i0 += kRedSetMax) {
    const int c = std::min(kRedSetMax, n - i0);
    RedSet S{};
    int nb = 1;
    for (int i = 0; i < c; ++i) {
      const RedOne &o = ops[i0 + i];
      S.r[i] = RedArgs{o.op, o.a, o.b, o.c, o.d, o.s1, o.s2, o.len};
      S.out[i] = o.out;
      S.nb[i] = red_blocks(o.len, kRedBlocks);
      nb = std::max(nb, S.nb[i]);
    }
    count_launch(), launch_pdl(reduce_set_kernel, dim3(nb, c), kRedThreads, 0, p->stream, S,
                               p->red_part, p->red_cnt);
  }
  return cudaGetLastError();
}

cudaError_t launch_reduce(ahlp_problem *p, int op, const double *a, const double *b,
                          long long len, double *out) {
  const RedOne o{op, a, b, len, out};
  return launch_reduce_set(p, &o, 1);
}

cudaError_t launch_step_dot(ahlp_problem *p, const double *x, const double *dx, double ap,
                            const double *z, const double *dz, double ad, long long n,
                            double *out) {
  const RedOne o{RED_STEP, x, dx, n, out, z, dz, ap, ad};
  return launch_reduce_set(p, &o, 1);
}

static SpSeg sp_seg(const SpMat &A, const double *x, double *y, double alpha, const double *yadd) {
  return SpSeg{A.rp, A.ci, A.v, A.rows, A.long_rows, A.n_long, x, yadd, y, alpha};
}

static unsigned sp_ctas(const SpSeg &a) {
  return (unsigned)(a.n_long + (a.rows + kSpThreads - 1) / kSpThreads);
}

cudaError_t launch_spmv(const SpMat &A, const double *x, double *y, double alpha,
                        const double *yadd, cudaStream_t s) {
  if (A.rows <= 0) return cudaSuccess;
  const SpSeg a = sp_seg(A, x, y, alpha, yadd);
  count_launch(), launch_pdl(spmv_kernel<SP_STORE>, sp_ctas(a), kSpThreads, 0, s, a, SpSeg{},
                             SpTailArgs{});
  return cudaGetLastError();
}

cudaError_t launch_finish(ahlp_problem *p, const double *dy, const double *rc, double *dx,
                          double *dz, bool adjoint, double *wx, double *wc) {
  if (p->n <= 0) return cudaSuccess;
  const SpSeg a = sp_seg(p->ATmat, dy, nullptr, 1.0, nullptr);
  SpTailArgs T{};
  T.f = p->f;
  T.w = p->wfin;
  T.xinv = p->xinv;
  T.z = p->z;
  T.x = p->x;
  T.rc = rc;
  T.dx = dx;
  T.dz = dz;
  T.wx = wx;
  T.wc = wc;
  T.adjoint = adjoint ? 1 : 0;
  count_launch(), launch_pdl(spmv_kernel<SP_FINISH>, sp_ctas(a), kSpThreads, 0, p->stream, a,
                             SpSeg{}, T);
  return cudaGetLastError();
}

cudaError_t launch_residual(ahlp_problem *p, const double *r_d, const double *r_p,
                            const double *r_c, const double *dx, const double *dy,
                            const double *dz, double *e_d, double *e_p, double *e_c,
                            bool adjoint) {
  const SpSeg a = sp_seg(p->ATmat, dy, e_d, -1.0, r_d), b = sp_seg(p->Amat, dx, e_p, -1.0, r_p);
  if (sp_ctas(a) + sp_ctas(b) == 0) return cudaSuccess;
  SpTailArgs T{};
  T.ddx = dx;
  T.ddz = dz;
  T.z = p->z;
  T.x = p->x;
  T.rc = r_c;
  T.e_c = e_c;
  T.adjoint = adjoint ? 1 : 0;
  count_launch(), launch_pdl(spmv_kernel<SP_RESID>, sp_ctas(a) + sp_ctas(b), kSpThreads, 0,
                             p->stream, a, b, T);
  return cudaGetLastError();
}

cudaError_t launch_axpby(double *y, const double *x, double a, double b, long long n,
                         cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  count_launch(), launch_pdl(axpby_k, blocks_for(n, 256), 256, 0, s, y, x, a, b, n);
  return cudaGetLastError();
}

cudaError_t launch_fill(double *y, double v, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  count_launch(), launch_pdl(fill_k, blocks_for(n, 256), 256, 0, s, y, v, n);
  return cudaGetLastError();
}

cudaError_t launch_mul(double *y, const double *a, const double *b, double scale, long long n,
                       cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  count_launch(), launch_pdl(mul_k, blocks_for(n, 256), 256, 0, s, y, a, b, scale, n);
  return cudaGetLastError();
}

cudaError_t launch_ipm_rc(double *rc, const double *x, const double *z, const double *dxa,
                          const double *dza, double sigma_mu, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  count_launch(), launch_pdl(ipm_rc_k, blocks_for(n, 256), 256, 0, s, rc, x, z, dxa, dza, sigma_mu,
                             n);
  return cudaGetLastError();
}

cudaError_t launch_centrality_rc(double *rc2, const double *rc, const double *x,
                                 const double *dx, double ap, const double *z, const double *dz,
                                 double ad, double lo, double hi, long long n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  count_launch(), launch_pdl(centrality_rc_k, blocks_for(n, 256), 256, 0, s, rc2, rc, x, dx, ap, z,
                             dz, ad, lo, hi, n);
  return cudaGetLastError();
}

}  // namespace ahlp
