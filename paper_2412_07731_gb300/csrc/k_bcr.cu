// Block cyclic reduction of the link chain (the block-tridiagonal part T of
// the Schur complement, App. A), its border coupling Z = L^-1 E' and its
// solves.
//
// In a chain segment of n link pairs, position i is eliminated at level
// ctz(i + 1): level 0 takes every other pair, level 1 every other remaining
// one, and so on, so a segment of n pairs needs ceil(log2(n + 1)) levels and
// the positions of one level are independent of each other.  At level v the
// remaining neighbours of position j are a = j - 2^v and b = j + 2^v (when
// inside the segment).  Eliminating j (all FP64):
//   T_j  -= sum over the earlier levels v' of  GR_m' GR_m  (m = j - 2^v')
//                                          and GL_m' GL_m  (m = j + 2^v');
//   L_j L_j' = T_j;  Linv_j = L_j^-1;
//   GL_j = Linv_j C(j, a),  GR_j = Linv_j C(b, j)'   (couplings to a and b);
//   E_j' -= the same earlier-level terms applied to their Z, Z_j = Linv_j E_j'.
// The coupling C(b, a) that appears between j's neighbours is -GR_j' GL_j,
// built on demand one level later by whoever needs it (at level 0 the
// couplings are the assembled H blocks).  In elimination order the factor's
// off-diagonal blocks are GL_j' (row a) and GR_j' (row b), so
//   forward:  u_j = Linv_j (r_j - sum_m GR_m' u_m (m left of j) - sum_m GL_m' u_m (m right)),
//   backward: x_j = Linv_j' (u_j - GL_j x_a - GR_j x_b),
// level by level upwards and downwards.  Z' Z over all rows equals
// E T^-1 E' for any elimination order, so the border factor and its solves
// are unchanged.  The sequential depth is the number of levels, not the
// number of pairs.
#include <algorithm>

#include "ahlp_internal.h"
#include "publish.h"

namespace ahlp {

namespace {

constexpr int kBcrThreads = 128;
constexpr int kBcrSmallL = 32;   // link blocks up to this size: one-warp Cholesky

struct BArgs {
  const int *l;                        // [N-1] link rows per pair
  const long long *td_off, *h_off, *link_off;
  const int *order;                    // pairs of the current level
  const int *info;                     // [N-1][4]: level, segment first pair, segment end, -
  int lmax;
  double *Td;                          // in: assembled T_j; out: L_j (lower)
  const double *Hd;                    // assembled H_j (l_{j+1} x l_j, ld l_{j+1})
  double *Linv;                        // L_j^-1 (layout of T_j)
  double *GL, *GR;                     // [N-1][lmax^2], ld l_j
  double *Et;                          // [B][nl]: E' in, Z out
  const double *Td_diag0;
  double tol;
  int *status;
  int B, nl;
};

__device__ __forceinline__ void pair_info(const BArgs &A, int j, int &lv, int &jb, int &je) {
  lv = A.info[4 * j];
  jb = A.info[4 * j + 1];
  je = A.info[4 * j + 2];
}

// dst (rows x cols, ld rows) -= G' H for G (k x rows, ld k), H (k x cols, ld k)
__device__ void sub_gtg(double *dst, int rows, int cols, const double *G, const double *H, int k,
                        int tid, int bd) {
  for (int i = tid; i < rows * cols; i += bd) {
    const int r = i % rows, c = i / rows;
    double a0 = 0.0, a1 = 0.0;
    int q = 0;
    for (; q + 1 < k; q += 2) {
      a0 = fma(G[q + (long long)r * k], H[q + (long long)c * k], a0);
      a1 = fma(G[q + 1 + (long long)r * k], H[q + 1 + (long long)c * k], a1);
    }
    if (q < k) a0 = fma(G[q + (long long)r * k], H[q + (long long)c * k], a0);
    dst[i] -= a0 + a1;
  }
}

// Factor of the pairs of one level: earlier-level updates of T_j, its
// Cholesky and inverse, and GL_j, GR_j.  One CTA per pair.
__global__ void __launch_bounds__(kBcrThreads) bcr_factor_kernel(BArgs A) {
  pdl_begin();
  extern __shared__ double sm[];
  const int lm = A.lmax;
  double *T = sm, *Li = sm + lm * lm, *C = sm + 2 * lm * lm;
  __shared__ double Tinv[96];
  const int tid = threadIdx.x, bd = blockDim.x;
  const int j = A.order[blockIdx.x];
  int lv, jb, je;
  pair_info(A, j, lv, jb, je);
  const int lj = A.l[j];
  double *Tg = A.Td + A.td_off[j];
  for (int i = tid; i < lj * lj; i += bd) T[i] = Tg[i];
  __syncthreads();
  // T_j -= GR_m' GR_m (m = j - 2^v') and GL_m' GL_m (m = j + 2^v'), v' < lv
  for (int v = 0; v < lv; ++v) {
    const int ml = j - (1 << v), mr = j + (1 << v);
    if (ml >= jb) sub_gtg(T, lj, lj, A.GR + (long long)ml * lm * lm,
                          A.GR + (long long)ml * lm * lm, A.l[ml], tid, bd);
    __syncthreads();
    if (mr < je) sub_gtg(T, lj, lj, A.GL + (long long)mr * lm * lm,
                         A.GL + (long long)mr * lm * lm, A.l[mr], tid, bd);
    __syncthreads();
  }
  // Cholesky of T_j (pivot safeguard against the link rows' full diagonal)
  if (lj <= kBcrSmallL) {
    if (tid < 32) {
      const int lane = tid;
      for (int c = 0; c < lj; ++c) {
        double piv = T[c + c * lj];
        const double orig = A.Td_diag0[A.link_off[j] + c];
        const double lim = A.tol * orig, floor_v = lim > 0.0 ? lim : 1.0;
        if (!(piv == piv)) {
          if (lane == 0 && atomicAdd(&A.status[0], 1) == 0) {
            A.status[2] = -1 - j;
            A.status[3] = c;
          }
          piv = floor_v;
        } else if (!(piv > lim) || !(piv > 0.0)) {
          if (lane == 0) atomicAdd(&A.status[1], 1);
          piv = floor_v;
        }
        const double inv = rsqrt(piv);
        __syncwarp();
        if (lane == c) {
          T[c + c * lj] = piv * inv;
          Tinv[c] = inv;
        } else if (lane > c && lane < lj) {
          T[lane + c * lj] *= inv;
        }
        __syncwarp();
        if (lane > c && lane < lj) {
          const double lr = T[lane + c * lj];
          for (int q = c + 1; q <= lane; ++q) T[lane + q * lj] = fma(-lr, T[q + c * lj], T[lane + q * lj]);
        }
        __syncwarp();
      }
    }
  } else {
    for (int c = 0; c < lj; ++c) {
      if (tid == 0) {
        double piv = T[c + c * lj];
        pivot_fix(piv, A.Td_diag0[A.link_off[j] + c], A.tol, A.status, -1 - j, c);
        const double lcc = sqrt(piv);
        T[c + c * lj] = lcc;
        Tinv[c] = 1.0 / lcc;
      }
      __syncthreads();
      const double inv = Tinv[c];
      for (int r = c + 1 + tid; r < lj; r += bd) T[r + c * lj] *= inv;
      __syncthreads();
      const int m = lj - c - 1;
      for (int i = tid; i < m * m; i += bd) {
        const int rr = i % m, ss = i / m;
        if (rr >= ss)
          T[(c + 1 + rr) + (c + 1 + ss) * lj] -= T[(c + 1 + rr) + c * lj] * T[(c + 1 + ss) + c * lj];
      }
      __syncthreads();
    }
  }
  __syncthreads();
  // Linv_j: column c by forward substitution (one thread per column)
  for (int c = tid; c < lj; c += bd) {
    for (int r = 0; r < c; ++r) Li[r + c * lj] = 0.0;
    Li[c + c * lj] = Tinv[c];
    for (int r = c + 1; r < lj; ++r) {
      double acc = 0.0;
      for (int q = c; q < r; ++q) acc = fma(T[r + q * lj], Li[q + c * lj], acc);
      Li[r + c * lj] = -acc * Tinv[r];
    }
  }
  __syncthreads();
  for (int i = tid; i < lj * lj; i += bd) {
    const int r = i % lj, s = i / lj;
    Tg[i] = r >= s ? T[i] : 0.0;
    A.Linv[A.td_off[j] + i] = Li[i];
  }
  // GL_j = Linv_j C(j, a), a = j - 2^lv
  const int a = j - (1 << lv), b = j + (1 << lv);
  for (int side = 0; side < 2; ++side) {
    const int nb = side == 0 ? a : b;
    if (side == 0 ? nb < jb : nb >= je) continue;
    const int ln = A.l[nb];
    // C = the coupling as (l_j x l_nb): C(j, a) for the left side, C(b, j)'
    // for the right side
    if (lv == 0) {
      if (side == 0) {   // H_{j-1}: l_j x l_{j-1}, ld l_j
        const double *H = A.Hd + A.h_off[j - 1];
        for (int i = tid; i < lj * ln; i += bd) C[i] = H[i];
      } else {           // H_j: l_{j+1} x l_j, ld l_{j+1}; transposed
        const double *H = A.Hd + A.h_off[j];
        for (int i = tid; i < lj * ln; i += bd) {
          const int r = i % lj, c = i / lj;
          C[i] = H[c + (long long)r * ln];
        }
      }
    } else {
      // the coupling created by the position m between j and its neighbour:
      // C(j, a) = -GR_m' GL_m (m = j - 2^(lv-1)); C(b, j) = -GR_m' GL_m
      // (m = j + 2^(lv-1)), so C(b, j)' = -GL_m' GR_m
      const int m = side == 0 ? j - (1 << (lv - 1)) : j + (1 << (lv - 1));
      const int lmm = A.l[m];
      const double *G1 = (side == 0 ? A.GR : A.GL) + (long long)m * lm * lm;   // l_m x l_j
      const double *G2 = (side == 0 ? A.GL : A.GR) + (long long)m * lm * lm;   // l_m x l_nb
      for (int i = tid; i < lj * ln; i += bd) C[i] = 0.0;
      __syncthreads();
      sub_gtg(C, lj, ln, G1, G2, lmm, tid, bd);
    }
    __syncthreads();
    double *G = (side == 0 ? A.GL : A.GR) + (long long)j * lm * lm;
    for (int i = tid; i < lj * ln; i += bd) {
      const int r = i % lj, c = i / lj;
      double acc = 0.0;
      for (int q = 0; q <= r; ++q) acc = fma(Li[r + q * lj], C[q + c * lj], acc);
      G[i] = acc;
    }
    __syncthreads();
  }
}

// Z_j = Linv_j (E_j' - earlier-level terms), thread (row, column) over 32 x 4,
// blockIdx.y over groups of four border columns
__global__ void __launch_bounds__(kBcrThreads) bcr_z_kernel(BArgs A) {
  pdl_begin();
  const int j = A.order[blockIdx.x];
  int lv, jb, je;
  pair_info(A, j, lv, jb, je);
  const int lj = A.l[j], lm = A.lmax;
  const int cl = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rb = blockIdx.y * 4 + cl;
  __shared__ double e[4][96];
  const bool col = rb < A.B;
  double *ez = A.Et + (long long)(col ? rb : 0) * A.nl;
  for (int r = lane; r < lj; r += 32) {
    double v = col ? ez[A.link_off[j] + r] : 0.0;
    for (int w = 0; w < lv && col; ++w) {
      const int ml = j - (1 << w), mr = j + (1 << w);
      if (ml >= jb) {   // GR_ml' Z_ml
        const double *G = A.GR + (long long)ml * lm * lm;
        const int k = A.l[ml];
        const double *z = ez + A.link_off[ml];
        for (int q = 0; q < k; ++q) v = fma(-G[q + (long long)r * k], z[q], v);
      }
      if (mr < je) {    // GL_mr' Z_mr
        const double *G = A.GL + (long long)mr * lm * lm;
        const int k = A.l[mr];
        const double *z = ez + A.link_off[mr];
        for (int q = 0; q < k; ++q) v = fma(-G[q + (long long)r * k], z[q], v);
      }
    }
    e[cl][r] = v;
  }
  __syncwarp();
  if (!col) return;
  const double *Li = A.Linv + A.td_off[j];
  for (int r = lane; r < lj; r += 32) {
    double a0 = 0.0, a1 = 0.0;
    int q = 0;
    for (; q + 1 <= r; q += 2) {
      a0 = fma(Li[r + q * lj], e[cl][q], a0);
      a1 = fma(Li[r + (q + 1) * lj], e[cl][q + 1], a1);
    }
    if (q <= r) a0 = fma(Li[r + q * lj], e[cl][q], a0);
    ez[A.link_off[j] + r] = a0 + a1;
  }
}

// The solves.  A pair needs a few thousand multiply-adds and then the solutions
// of its neighbours, so they are bound by latency.  One launch per sweep, a CTA
// per pair: CTAs take the pairs in elimination order by ticket (the backward
// sweep in reverse), so a pair only waits for pairs whose CTAs already run, and
// a pair's solution is published entry by entry (publish.h).  While it waits, a
// CTA reads its coupling blocks once, which brings them into its L1.  Eight
// lanes share a row; left and right terms go to the two halves of the CTA.  A
// launch per level took 8.4 us (forward) and 6.8 us (backward) at 64 pairs of 20
// rows, 91 us for both sweeps' six levels; a thread per row had taken 18.6 and
// 15.1 us per level.
constexpr int kBcrLanes = 8;
constexpr int kBcrSolveThreads = 512;   // 32 rows at a time, left and right terms apart
constexpr int kBcrMaxTerms = 64;        // earlier-level terms of a pair, both sides

__device__ __forceinline__ double bcr_lanes_sum(double v) {
#pragma unroll
  for (int o = kBcrLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// s += sum_q G[q] z[q], q = q0, q0 + 8, ... < k
__device__ __forceinline__ void bcr_dot(const double *G, const double *z, int k, int stride,
                                        int q0, double &s) {
#pragma unroll 4
  for (int q = q0; q < k; q += kBcrLanes) s = fma(G[(long long)q * stride], z[q], s);
}

// the same entries of G read and dropped
__device__ __forceinline__ void bcr_touch(const double *G, int k, int stride, int q0) {
#pragma unroll 4
  for (int q = q0; q < k; q += kBcrLanes) {
    const double v = G[(long long)q * stride];
    asm volatile("" ::"d"(v));
  }
}

// zs[i] = the published entry pub[at[i / lm] + i % lm], i % lm < cnt[i / lm]
__device__ __forceinline__ void bcr_collect(double *zs, const double *pub, const int *cnt,
                                            const long long *at, int nterm, int lm, int *err) {
  const int total = nterm * lm;
  for (int i0 = threadIdx.x & ~31; i0 < total; i0 += blockDim.x) {   // whole warps
    const int i = i0 + (threadIdx.x & 31);
    const int t = i < total ? i / lm : 0, q = i - t * lm;
    const bool in = i < total && q < cnt[t];
    const double *p = pub + (in ? at[t] + q : 0);
    PubBits<double>::U bits = in ? PubBits<double>::ld(p) : 0;
    wait_published<double>(bits, p, in, err);
    if (in) zs[i] = PubBits<double>::val(bits);
  }
}

// forward: u_j = Linv_j (r_j - earlier-level terms); r in svec's link part, u
// published in pub
__global__ void __launch_bounds__(kBcrSolveThreads) bcr_fwd_kernel(BArgs A, const double *svec,
                                                                   double *pub, int *ticket,
                                                                   int *err) {
  pdl_begin();
  extern __shared__ double zs[];   // [terms][lmax]
  __shared__ double r[kMaxLinks], part[2][kMaxLinks];
  __shared__ int cnt[kBcrMaxTerms];         // term 2w + side: rows, 0: none
  __shared__ long long at[kBcrMaxTerms];    // and where its solution starts
  __shared__ int s_job;
  if (threadIdx.x == 0) s_job = atomicAdd(ticket, 1);
  __syncthreads();
  const int j = A.order[s_job];
  int lv, jb, je;
  pair_info(A, j, lv, jb, je);
  const int lj = A.l[j], lm = A.lmax;
  const long long off = A.link_off[j];
  const int side = threadIdx.x / (kBcrSolveThreads / 2);
  const int lane = threadIdx.x & (kBcrLanes - 1);
  const int row0 = (threadIdx.x % (kBcrSolveThreads / 2)) / kBcrLanes;
  constexpr int rows = kBcrSolveThreads / 2 / kBcrLanes;
  if (threadIdx.x < 2 * lv) {
    const int w = threadIdx.x >> 1, m = (threadIdx.x & 1) ? j + (1 << w) : j - (1 << w);
    const bool in = (threadIdx.x & 1) ? m < je : m >= jb;
    cnt[threadIdx.x] = in ? A.l[m] : 0;
    at[threadIdx.x] = in ? A.link_off[m] : 0;
  }
  __syncthreads();
  const double *Gs = side ? A.GL : A.GR;
  const double *Li = A.Linv + A.td_off[j];
  for (int i = row0; i < lj; i += rows) {
    for (int w = 0; w < lv; ++w) {
      const int k = cnt[2 * w + side];
      const long long m = side ? j + (1 << w) : j - (1 << w);
      bcr_touch(Gs + m * lm * lm + (long long)i * k, k, 1, lane);
    }
    if (side == 0) bcr_touch(Li + i, i + 1, lj, lane);
  }
  bcr_collect(zs, pub, cnt, at, 2 * lv, lm, err);
  __syncthreads();
  for (int i0 = 0; i0 < lj; i0 += rows) {
    const int i = i0 + row0;
    double s = 0.0;
    if (i < lj)
      for (int w = 0; w < lv; ++w) {
        const int k = cnt[2 * w + side];
        const long long m = side ? j + (1 << w) : j - (1 << w);
        bcr_dot(Gs + m * lm * lm + (long long)i * k, zs + (2 * w + side) * lm, k, 1, lane, s);
      }
    s = bcr_lanes_sum(s);
    if (lane == 0 && i < lj) part[side][i] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < lj; i += kBcrSolveThreads)
    r[i] = svec[off + i] - (part[0][i] + part[1][i]);
  __syncthreads();
  for (int i0 = 0; i0 < lj; i0 += 2 * rows) {
    const int i = i0 + threadIdx.x / kBcrLanes;
    double s = 0.0;
    if (i < lj) bcr_dot(Li + i, r, i + 1, lj, lane, s);
    s = bcr_lanes_sum(s);
    if (lane == 0 && i < lj) PubBits<double>::st(pub + off + i, s);
  }
}

// backward: x_j = Linv_j' (v_j - GL_j x_a - GR_j x_b); x goes to svec's link part
// (which may be v) and is published in pub
__global__ void __launch_bounds__(kBcrSolveThreads) bcr_bwd_kernel(BArgs A, int npairs,
                                                                   const double *v, double *svec,
                                                                   double *pub,
                                                                   int *ticket, int *err) {
  pdl_begin();
  extern __shared__ double zs[];   // [2][lmax]
  __shared__ double r[kMaxLinks], part[2][kMaxLinks];
  __shared__ int cnt[2];
  __shared__ long long at[2];
  __shared__ int s_job;
  if (threadIdx.x == 0) s_job = atomicAdd(ticket, 1);
  __syncthreads();
  const int j = A.order[npairs - 1 - s_job];
  int lv, jb, je;
  pair_info(A, j, lv, jb, je);
  const int lj = A.l[j], lm = A.lmax;
  const long long off = A.link_off[j];
  const int side = threadIdx.x / (kBcrSolveThreads / 2);
  const int lane = threadIdx.x & (kBcrLanes - 1);
  const int row0 = (threadIdx.x % (kBcrSolveThreads / 2)) / kBcrLanes;
  constexpr int rows = kBcrSolveThreads / 2 / kBcrLanes;
  if (threadIdx.x < 2) {
    const int m = threadIdx.x ? j + (1 << lv) : j - (1 << lv);
    const bool in = threadIdx.x ? m < je : m >= jb;
    cnt[threadIdx.x] = in ? A.l[m] : 0;
    at[threadIdx.x] = in ? A.link_off[m] : 0;
  }
  __syncthreads();
  const double *G = (side ? A.GR : A.GL) + (long long)j * lm * lm;   // l_j x l_neighbour
  const double *Li = A.Linv + A.td_off[j];
  const int k = cnt[side];
  for (int i = row0; i < lj; i += rows) {
    bcr_touch(G + i, k, lj, lane);
    if (side == 0) bcr_touch(Li + (long long)i * lj + i, lj - i, 1, lane);
  }
  bcr_collect(zs, pub, cnt, at, 2, lm, err);
  __syncthreads();
  for (int i0 = 0; i0 < lj; i0 += rows) {
    const int i = i0 + row0;
    double s = 0.0;
    if (i < lj) bcr_dot(G + i, zs + side * lm, k, lj, lane, s);
    s = bcr_lanes_sum(s);
    if (lane == 0 && i < lj) part[side][i] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < lj; i += kBcrSolveThreads)
    r[i] = v[off + i] - (part[0][i] + part[1][i]);
  __syncthreads();
  for (int i0 = 0; i0 < lj; i0 += 2 * rows) {
    const int i = i0 + threadIdx.x / kBcrLanes;
    double s = 0.0;
    // entries i .. lj - 1 of column i
    if (i < lj) bcr_dot(Li + (long long)i * lj + i, r + i, lj - i, 1, lane, s);
    s = bcr_lanes_sum(s);
    if (lane == 0 && i < lj) {
      PubBits<double>::st(pub + off + i, s);
      svec[off + i] = s;
    }
  }
}

BArgs bargs(ahlp_problem *p) {
  BArgs A{};
  A.l = p->l_d;
  A.td_off = p->td_off_d;
  A.h_off = p->h_off_d;
  A.link_off = p->link_off_d;
  A.order = p->bcr_order;
  A.info = p->bcr_info;
  A.lmax = p->bcr_lmax;
  A.Td = p->Td;
  A.Hd = p->Hd;
  A.Linv = p->Linv;
  A.GL = p->bcr_GL;
  A.GR = p->bcr_GR;
  A.Et = p->Et;
  A.Td_diag0 = p->Td_diag0;
  A.tol = p->fac_pivot_tol;
  A.status = p->status;
  A.B = p->B;
  A.nl = p->nl;
  return A;
}

}  // namespace

cudaError_t launch_bcr_factor(ahlp_problem *p) {
  cudaStream_t s = p->stream;
  const int nlev = (int)p->bcr_loff.size() - 1;
  const size_t smem = (size_t)3 * p->bcr_lmax * p->bcr_lmax * sizeof(double);
  for (int v = 0; v < nlev; ++v) {
    const int n = p->bcr_loff[v + 1] - p->bcr_loff[v];
    if (n == 0) continue;
    BArgs A = bargs(p);
    A.order = p->bcr_order + p->bcr_loff[v];
    count_launch(), launch_pdl(bcr_factor_kernel, n, kBcrThreads, smem, s, A);
    if (p->B > 0)
      count_launch(), launch_pdl(bcr_z_kernel, dim3(n, (p->B + 3) / 4), kBcrThreads, 0, s, A);
  }
  return cudaGetLastError();
}

cudaError_t launch_bcr_solve(ahlp_problem *p, bool forward) {
  const int n = p->bcr_loff.back(), nlev = (int)p->bcr_loff.size() - 1;
  if (n == 0) return cudaSuccess;
  const BArgs A = bargs(p);
  const size_t row = (size_t)p->bcr_lmax * sizeof(double);
  if (forward)
    count_launch(), launch_pdl(bcr_fwd_kernel, n, kBcrSolveThreads, 2 * (nlev - 1) * row,
                               p->stream, A, p->svec, p->bcr_pub, p->trsv_ticket + 2, p->trsv_err);
  else
    count_launch(), launch_pdl(bcr_bwd_kernel, n, kBcrSolveThreads, 2 * row, p->stream, A, n,
                               p->B > 0 ? p->svec : p->bcr_pub, p->svec, p->bcr_pub + p->nl,
                               p->trsv_ticket + 3, p->trsv_err);
  return cudaGetLastError();
}

// The limits belong to the functions, not to a handle: they cover every accepted
// size, so that no handle lowers another's.
cudaError_t set_bcr_smem_limits() {
  constexpr int row = kMaxLinks * (int)sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(bcr_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kBcrMaxTerms * row);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(bcr_factor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              3 * kMaxLinks * row);
}

}  // namespace ahlp
