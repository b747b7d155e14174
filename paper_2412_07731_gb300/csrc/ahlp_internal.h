// Internal declarations shared by the host runtime and the kernels.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <utility>
#include <vector>

#include "../../include/ahlp.h"

namespace ahlp {

constexpr int NB = 64;            // tile edge of the dense kernels
constexpr int kPrecFP64 = 0;      // factor storage of the block matrices
constexpr int kPrecFP32 = 1;
// float-float: value = hi + lo with two FP32 arrays (aug32 = hi, aug_lo = lo);
// the factorisation runs in double-float arithmetic on the FP32 pipe (about
// 46 significant bits); the finished factor is expanded into the FP64 buffer,
// which the Schur assembly and the solves read as for an FP64 factor
constexpr int kPrecFF = 2;
constexpr double kFp32PivotTol = 1e-6;    // smallest clamp threshold for FP32 pivots
constexpr double kFFPivotTol = 1e-12;     // smallest clamp threshold for float-float pivots
// pivot_mode 1: a failing pivot becomes scale * max(its starting diagonal, 1),
// capped so that its square root and reciprocal stay normal in the factor's
// storage words
constexpr double kDropFP64 = 1e32, kDropFF = 1e16, kDropFP32 = 1e16;
constexpr double kDropCapFF = 1e60, kDropCapFP32 = 1e30;
constexpr int kMaxBorder = 20480;   // linking variables and global rows, at most
constexpr int kTickets = 6;         // ticket counters of a solve
constexpr int kMaxLinks = 96;     // local link rows of a block pair, at most
constexpr int kThreads = 256;     // threads per CTA of the dense kernels
// FP64 factors on the tensor cores (k_dz.cu): digits per entry, and the row
// exponent that marks a row holding a NaN or an infinity
constexpr int kDzQ = 8;
constexpr int kDzNotFinite = 1 << 20;

// One dense lower-triangular "partial Cholesky" problem: an a x a matrix
// (column-major, leading dimension lda, element offset base) whose first p
// pivots are eliminated.  After the factorisation the (p..a) x (p..a) corner
// holds the Schur complement of the leading p x p block.
// CSR matrix on the device with its rows binned by length: rows up to
// kShortRow nonzeros go to 8-lane groups, the rest (the dense linking-variable
// rows of A') to one CTA each.
constexpr int kShortRow = 256;
struct SpMat {
  const int *rp = nullptr, *ci = nullptr;
  const double *v = nullptr;
  long long rows = 0;
  const int *long_rows = nullptr;   // [n_long] rows with more than kShortRow nonzeros
  int n_long = 0;
};

struct BlkInfo {
  long long base;    // offset of element (0,0) in its buffer
  long long voff;    // offset of this problem's vector segment in solve vectors
  long long d0off;   // offset of its original diagonal in the diag0 array
  int lda, a, p;
  int T, Tp;         // tiles of a, tiles holding pivots
  int tag;           // added to the problem index in pivot reports (kTag*)
  long long cdoff;   // offset of the corner (non-pivot) diagonal in cdiag0
  long long ioff;    // offset of its Tp inverted diagonal tiles (block solves)
  long long soff;    // first staging slot of its panel tiles (tensor-core update)
};
constexpr int kTagBorderX = 1 << 20;   // pivot reports of the border x_0 factor
constexpr int kTagBorderG = 2 << 20;   // pivot reports of the border y_g factor

#ifdef __CUDACC__
// Every device wait of the library gives up after this long; the host then reports
// AHLP_ERR_TIMEOUT.
constexpr unsigned long long kWaitLimitNs = 1000000000ull;   // 1 s

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// First statement of nearly every kernel that launch_pdl starts: returns when the
// kernels before this one are complete and their writes are visible; from then
// on the next kernel of the stream may be scheduled (it waits in turn).
// pdl_wait leaves that to the kernel's end: for kernels that fill the GPU, whose
// successors would only hold shared memory and registers.  Pointers to data that
// other kernels write are not marked __restrict__ here: such loads count as
// invariant and could be moved above the wait.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_begin() {
  pdl_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch with programmatic stream serialisation: the kernel's launch and the
// scheduling of its CTAs overlap the tail of the kernel before it.  Dependent
// kernels of a few CTAs follow each other in 1.5 us instead of 4.1 us, and most
// of a solve's kernels are that small.  Only for kernels in which every thread passes
// griddepcontrol.wait before it touches what earlier kernels wrote: with pdl_begin or
// pdl_wait first, or, in diagonal factorisations beside an update, after the wait for
// that update's counts (diag_begin), with griddepcontrol.wait at the end (diag_end).
template <typename... P, typename... A>
inline void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       A &&...args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Pivot safeguard shared by every Cholesky in the library.  A pivot that is
// not above tol * (the diagonal entry it started from) has lost all its
// significant digits to cancellation.  It is clamped to that threshold, which
// keeps the factor nonsingular (the Krylov refinement of kkt_solve then
// corrects the solve against the exact Newton matrix); or, with drop > 0, it
// becomes drop * max(orig, 1) (at most cap), which leaves the row out of the
// factor: its column below the pivot and its solution entry come out ~0, the
// treatment of nearly dependent rows of A D A' in interior-point codes.  NaN
// pivots are counted in status[0] with the first location, failing pivots in
// status[1].
__device__ __forceinline__ void pivot_fix(double &piv, double orig, double tol, int *status,
                                          int where, int row, double drop = 0.0,
                                          double cap = 1e300) {
  const double floor_v = tol * orig > 0.0 ? tol * orig : 1.0;
  const double repl = drop > 0.0 ? fmin(drop * fmax(orig, 1.0), cap) : floor_v;
  if (!(piv == piv)) {
    if (atomicAdd(&status[0], 1) == 0) {
      status[2] = where;
      status[3] = row;
    }
    piv = repl;
  } else if (!(piv > tol * orig) || !(piv > 0.0)) {
    atomicAdd(&status[1], 1);
    piv = repl;
  }
}
#endif

// One formation tile: block, tile row, tile column.
struct FormTile {
  int blk, I, J, pad;
};

// Per-block layout of the local Schur columns k_i = n0 + lprev + lnext + mg.
struct SchurBlk {
  int m;       // pivots (rows of A_i)
  int k;       // local Schur columns: [x_0 slice | links i-1 | links i | global-row slice]
  int lprev, lnext;
  int link_prev_off, link_next_off;   // offsets of pairs i-1 and i in the link block
  int x0lo, x0n;   // the block's slice of the linking variables (all of them for one LP;
  int glo, gn;     // its LP's ones in a batch) and of the global rows
};

// A sparse matrix assembled column by column (host), and the equality-form
// description of an LP given in the full statement (general.cpp), with the
// map back to its original variables.
struct StdCsc {
  using Entry = std::pair<int, double>;   // (row, value)
  using Col = std::vector<Entry>;
  int m = 0;
  std::vector<int32_t> cp{0}, ri;
  std::vector<double> v;
  void push(const Col &c) {
    for (auto &e : c) {
      ri.push_back(e.first);
      v.push_back(e.second);
    }
    cp.push_back((int32_t)ri.size());
  }
  int n() const { return (int)cp.size() - 1; }
  ahlp_csc csc() const {
    return ahlp_csc{m, n(), cp.data(), ri.empty() ? nullptr : ri.data(),
                    v.empty() ? nullptr : v.data()};
  }
};

struct StdDesc {
  // original variable `orig` of block blk (-1: of x_0) = shift + sign x'_k
  // (- x'_k2 when k2 >= 0), k and k2 indices among its block's (x_0's)
  // standard-form columns
  struct Recov {
    int blk, orig;
    double shift;
    int k;
    double sign;
    int k2;
  };
  int N = 0;
  std::vector<StdCsc> A, W, Fg, FL, FR, F0;
  StdCsc Fg0;
  std::vector<std::vector<double>> b, c, blink;
  std::vector<double> bg, c0;
  std::vector<int32_t> l;
  std::vector<ahlp_csc> Ac, Wc, Fgc, FLc, FRc, F0c;
  ahlp_csc Fg0c{};
  std::vector<const double *> bp, cp, blp;
  ahlp_desc d{};
  std::vector<Recov> recov;
  double const_obj = 0.0;
  std::vector<int> n_orig;
  int n0_orig = 0;
};

// true when the description uses bounds or inequality rows
bool desc_is_general(const ahlp_desc &d);
// the equality form with x >= 0 of a description in the full statement
// (throws Fail on invalid input)
void standardize(const ahlp_desc &d, StdDesc &S);

struct DeviceBuf {
  void *ptr = nullptr;
  size_t bytes = 0;
};

}  // namespace ahlp

struct ahlp_problem {
  // ---- sizes -------------------------------------------------------------
  int N = 0, n0 = 0, mg = 0, B = 0, nl = 0, nS = 0;
  // batch > 1: the direct sum of independent LPs; per LP its first block and
  // the offsets of its slices of x_0 and of the global rows
  int batch = 1;
  std::vector<long long> lp_blk0, lp_x0off, lp_goff;
  struct LpRange {   // index ranges of one LP of a batch in the global vectors
    long long xb0, xb1, x00, x01;            // x: its blocks, its linking variables
    long long yb0, yb1, yl0, yl1, yg0, yg1;  // y: block rows, link rows, global rows
    double bnorm, cnorm;                      // its ||b||_inf and ||c||_inf
  };
  std::vector<LpRange> lp_rng;
  // LPs given in the full statement: per LP its map back to the original
  // variables (empty: the LP was already in equality form with x >= 0)
  struct LpRecov {
    std::vector<ahlp::StdDesc::Recov> recov;
    std::vector<int> n_orig;
    int n0_orig = 0;
    double const_obj = 0.0;
  };
  std::vector<LpRecov> lp_recov;
  long long n = 0, m = 0, msum = 0;   // n_total, m_total, sum of m_i
  std::vector<int> mi, ni, ki, lprev, lnext;
  std::vector<long long> xoff, yoff, link_off;   // link_off has N entries (pairs + 1)
  ahlp_options opt{};
  cudaStream_t stream = nullptr;
  std::string err;
  double bnorm_inf = 0, cnorm_inf = 0;
  int device = 0;

  // ---- LP data on the device ----------------------------------------------
  double *b = nullptr, *c = nullptr;               // global rhs, cost
  int *A_rp = nullptr, *A_ci = nullptr;            // CSR of A (m x n)
  double *A_v = nullptr;
  int *AT_rp = nullptr, *AT_ci = nullptr;          // CSR of A' (n x m)
  double *AT_v = nullptr;
  unsigned char *is_x0 = nullptr;                  // [n] 1 for x_0 columns
  ahlp::SpMat Amat, ATmat;                         // A and A' with their long-row lists

  // ---- factor storage -----------------------------------------------------
  double *aug = nullptr;            // all augmented matrices, FP64 (allocated when first used)
  float *aug32 = nullptr;           // the same layout in FP32 (mixed mode; hi part of FF)
  float *aug_lo = nullptr;          // lo part of float-float factors
  long long aug_elems = 0;
  // per pivot tile of every block, a 64x64 column-major tile: the inverse of
  // the pivot triangle on its pivot rows, the factor itself on the non-pivot
  // rows of a block's last pivot tile, zeros elsewhere
  double *tinv = nullptr;
  float *tinv32 = nullptr;
  long long tinv_elems = 0;
  int fac_prec = 0;                 // precision of the current factor (kPrec*)
  ahlp::BlkInfo *blk = nullptr;     // [N]
  std::vector<ahlp::BlkInfo> h_blk;
  ahlp::SchurBlk *sblk = nullptr;   // [N]
  std::vector<ahlp::SchurBlk> h_sblk;
  double *diag0 = nullptr;          // original diagonals (blocks)
  double *cdiag0 = nullptr;         // corner diagonals before elimination ([U;Fg] D [U;Fg]')
  double *sb_ref = nullptr;         // reference diagonal of the border pivots
  long long cdiag_elems = 0;
  long long vec_elems = 0;          // sum of a_i
  int maxT = 0, maxTp = 0;
  // tensor-core trailing update of FP32 factors (k_tc.cu): each panel tile
  // of the current step staged as TF32 hi / lo words in the MMA operand
  // layout (one 8192-word slot per tile of every block), the update jobs of
  // every step as prefix offsets over the blocks, and one tensor map per
  // block over its FP32 augmented matrix
  float *pstage = nullptr;
  long long stage_slots = 0;
  int *tc_joff = nullptr;            // [maxTp][2 N + 2] (StepJobs::joff)
  // diagonal tiles of the next step, counted off by an update's CTAs: [maxTp][N],
  // cleared by launch_dscale; blocks a step's jobs do not touch; blocks per step
  int *la_ready = nullptr, *la_miss = nullptr;
  long long la_elems = 0;
  std::vector<long long> la_miss_off;
  std::vector<int> la_pot;
  std::vector<long long> tc_jobs;    // [maxTp]
  // FP64 factors on the tensor cores: each panel tile of the current step as
  // eight FP16 digit planes, one exponent per row, and the CUtensorMaps of the
  // A and B operand copies
  __half *dz_stage = nullptr;
  int *dz_exp = nullptr;
  unsigned char dz_map[2][128] = {};
  bool fac_dz = false;      // the last FP64 factor's updates ran on the tensor cores
  // FP64 factors keep to the FP64 pipe: set when a digit factor broke down (a NaN
  // pivot or a stalled direction), for the rest of a solve
  bool fp64_pipe = false;
  void *tc_tmap = nullptr;           // [N] CUtensorMap
  bool tc_ready = false;
  // float-float factors on the tensor cores: each panel tile as six FP16
  // digit planes (6 x 4096 halves per slot) and one exponent per row
  __half *dstage = nullptr;
  int *dexp = nullptr;
  bool oz_ready = false;
  void *oz_tmap = nullptr;           // [2N] CUtensorMap: each block's hi, then lo matrix
  int ff_update = 0;                 // trailing update of float-float factors: 1 FP32 pipe, 2 tensor
                                     // cores (one CTA per job), 3 tensor cores (persistent)
  // per block, T x T: lower tile (I, J) of the formed augmented matrix has entries
  std::vector<std::vector<unsigned char>> tile_nz;
  // tile-sparse update jobs (option tile_sparse): per step, the kept jobs of the
  // dense enumeration as {block, I0, J, has_i1}; nullptr = the dense triangle
  int4 *tc_jtab = nullptr;
  std::vector<long long> tc_jtab_off;
  long long tc_jobs_dense = 0, tc_jobs_kept = 0;
  int fp32_update = 0;               // trailing update of FP32 factors: 1 SIMT, 2 tensor
                                     // cores (one CTA per job), 3 tensor cores (persistent
                                     // warp-specialised pipeline), 0 either, by the jobs of a step
  int num_sms = 1;
  double fac_flops = 0;   // algorithmic flops of one batched partial Cholesky
  double tri_elems = 0;   // lower-triangle entries of all augmented matrices

  // ---- formation pattern --------------------------------------------------
  ahlp::FormTile *ftiles = nullptr;
  long long *tile_ent = nullptr;    // [ntiles+1]
  int *ent_pos = nullptr;           // [nent]
  long long *ent_cb = nullptr;      // [nent+1]
  int *con_idx = nullptr;           // [ncon]
  double *con_coef = nullptr;       // [ncon]
  long long ntiles = 0, nent = 0, ncon = 0;

  // ---- Schur complement ---------------------------------------------------
  std::vector<long long> td_off, h_off;   // offsets of T_j (l_j^2) and H_j (l_{j+1} l_j)
  long long td_elems = 0, h_elems = 0;
  double *Td = nullptr, *Hd = nullptr, *Et = nullptr, *SB = nullptr;
  double *Td_asm = nullptr, *Hd_asm = nullptr, *Et_asm = nullptr, *SB_asm = nullptr;
  double *Td_diag0 = nullptr;        // assembled diagonal of T (pivot test)
  double *Linv = nullptr;            // L_j^-1 per pair (layout of Td)
  double *Yf = nullptr, *Yb = nullptr;   // chain coupling operators (layout of Hd)
  double *chain_tmp = nullptr;       // [nl] chain-solve scratch
  long long *td_off_d = nullptr, *h_off_d = nullptr;
  int *l_d = nullptr;                // [N-1]
  long long *link_off_d = nullptr;   // [N]
  int *kmap = nullptr;               // local Schur index -> global S index
  int *link_pair_d = nullptr;        // [nl] pair of each link row
  int *chain_seg = nullptr;          // [2 nchain_seg] pair ranges with link rows throughout
  int nchain_seg = 0;
  int *zlo = nullptr, *zhi = nullptr;   // [B] link rows a border column of Z can touch
  // cyclic reduction of the link chain (k_bcr.cu): pairs in level order,
  // per pair (level, segment first pair, segment end, -), the level offsets
  // into the order, and per pair its couplings GL_j, GR_j (lmax^2 each)
  int *bcr_order = nullptr, *bcr_info = nullptr;
  std::vector<int> bcr_loff;
  int bcr_lmax = 0;
  double *bcr_GL = nullptr, *bcr_GR = nullptr;
  double *bcr_pub = nullptr;   // [2 nl] published forward, then backward chain solution
  bool fac_bcr = false;   // the current Schur factor's chain is the cyclic-reduction one
  long long *yoff_d = nullptr;       // [N] start of y_i
  long long *kmap_off_d = nullptr;   // [N]
  std::vector<long long> kmap_off;
  long long *f0_idx = nullptr; double *f0_val = nullptr; long long nf0 = 0;   // Et constants
  long long *fg0_idx = nullptr; double *fg0_val = nullptr; long long nfg0 = 0; // SB constants
  // border (quasi-definite) factor
  double *border = nullptr; int Bld = 0;
  ahlp::BlkInfo *bx_info = nullptr, *bp_info = nullptr;
  ahlp::BlkInfo h_bx{}, h_bp{};
  double *border_diag0 = nullptr;
  // the border solves: the whole border factor (x_0 and y_g parts) as one more block of
  // the wavefront sweeps, its inverted diagonal tiles, the jobs of the forward and then
  // the backward sweep, and the two sweeps' published solutions
  ahlp::BlkInfo *bw_info = nullptr;
  int *bw_sched = nullptr;
  long long *bw_zero = nullptr;      // [1] the block's offset: 0
  double *border_tinv = nullptr;
  double *border_pub = nullptr;      // [2 B]

  // ---- vectors ------------------------------------------------------------
  double *x = nullptr, *z = nullptr, *dscale = nullptr;   // current point, d = x/z
  double *xinv = nullptr, *wfin = nullptr;   // 1 / x, 1 / (1 / d + rho on x_0)
  double *vec = nullptr;      // block solve segments [sum a_i]
  double *vecb = nullptr;     // backward solution as published (FP32 words with FP32 factors)
  float *vec32 = nullptr;     // forward solution as published with FP32 factors
  double *svec = nullptr;     // Schur vector [nS]
  double *f = nullptr, *g = nullptr, *rhat = nullptr;      // solve scratch
  double *stg[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};  // staging for host I/O
  double *res[3] = {nullptr, nullptr, nullptr};            // refinement residual
  double *best[3] = {nullptr, nullptr, nullptr};           // a direction while its factor is redone
  double *ipmv[19] = {};      // IPM work vectors (the last three: a batch's balanced rhs)
  double *red_part = nullptr; // reduction partials
  int *red_cnt = nullptr;     // arrivals at the reductions' last CTAs (0 between launches)
  double *mdot_part = nullptr;  // multi-dot partials [kMaxKrylov+1][304]
  double *gm_V = nullptr, *gm_Z = nullptr;   // Krylov bases, allocated on first use
  double *gm_h = nullptr;       // Arnoldi column on the device: both Gram-Schmidt passes and |w|^2
  int gm_cap = 0;               // vectors allocated in gm_Z (gm_V has one more)
  double *scal = nullptr;     // device scalars
  double *h_scal = nullptr;   // pinned host scalars; [511] holds the sequence word below
  unsigned read_seq = 0;      // value the device writes there when a read-back has arrived
  int *status = nullptr;      // device status words [4]
  // wavefront block solves: (block, row tile) jobs in ticket order, and the
  // ticket counters of the forward and backward block, chain and border solves (zeroed by
  // the first kernel of a solve, which also fills the publication buffers)
  int *trsv_fsched = nullptr, *trsv_bsched = nullptr;   // [2 * jobs]
  int *trsv_ticket = nullptr;     // [kTickets]
  int *trsv_err = nullptr;        // set when a wait timed out
  int trsv_nf = 0, trsv_nb = 0;
  int tiny_pivots = 0;
  bool factored = false;
  bool assembled = false;     // the Schur complement of the last kkt_factor exists
  double fac_delta = 0, fac_rho = 0, fac_pivot_tol = 0;
  double fac_rho_x = 0;   // primal regularisation of the preconditioner's D (ipm_solve's last safeguard)

  // ---- host <-> device traffic since create (ahlp_transfer_bytes) ----------
  long long bytes_h2d = 0, bytes_d2h = 0;

  // ---- timing -------------------------------------------------------------
  cudaEvent_t ev[8] = {};
  std::vector<cudaEvent_t> kt_pool;     // kernel-class timer: events, and per
  std::vector<int> kt_cls;              // recorded event the class it opens
  double kt_ms[3] = {0, 0, 0};          // last factor: diagonal tiles, panels, updates
  long long kt_n[3] = {0, 0, 0};        // and their launch groups
  float stage_ms[4] = {0, 0, 0, 0};

  std::vector<ahlp::DeviceBuf> allocs;
};

namespace ahlp {

// Every kernel launch of the library is written `count_launch(), launch_pdl(k, ...)`
// so the number of launches can be reported (arrowhead_lp_launch_count).
void count_launch();
long long launch_count();

// ---- kernels (launch wrappers) --------------------------------------------
// All wrappers enqueue on p->stream and return the cudaError_t of the launch.
// What a diagonal factorisation that runs beside the step before it waits for:
// ready[b] >= target (ready == nullptr: for that whole kernel, as usual).
struct LookAhead {
  int *ready = nullptr;
  int target = 0;
};
cudaError_t launch_dscale(ahlp_problem *p);   // dscale = x / (z + fac_rho_x x)
cudaError_t launch_form(ahlp_problem *p, double delta);
// prof (nullable): a handle whose kernel-class timer records the launches
// (kt_mark); classes 0 diagonal tiles, 1 panels, 2 trailing updates
// with dz (a handle set up by dz_setup) the trailing updates run on the tensor
// cores (k_dz.cu), else on the FP64 pipe
cudaError_t launch_pchol(double *buf, const BlkInfo *info, const std::vector<BlkInfo> &h,
                         const double *diag0, double tol, int *status, cudaStream_t s,
                         ahlp_problem *prof = nullptr, double drop = 0.0,
                         ahlp_problem *dz = nullptr);
// float-float (hi = aug32, lo): diagonal tiles and panels in FP64 arithmetic,
// trailing updates in double-float; then hi + lo is expanded into out (the
// FP64 factor buffer, elems entries), which the Schur assembly and the solves use
// with oz (a handle set up by oz_setup) the trailing updates run on the
// tensor cores as exact FP16 digit products (k_tc.cu)
cudaError_t launch_pchol_ff(float *hi, float *lo, double *out, long long elems,
                            const BlkInfo *info, const std::vector<BlkInfo> &h,
                            const double *diag0, double tol, int *status, cudaStream_t s,
                            ahlp_problem *oz = nullptr, ahlp_problem *prof = nullptr,
                            double drop = 0.0);
// FP32: also writes the inverted diagonal tiles into tinv (see launch_tinv);
// with tc (a handle set up by tc_setup) the trailing updates run on the
// tensor cores (k_tc.cu), else on the FP32 pipe
cudaError_t launch_pchol_f32(float *buf, float *tinv, const BlkInfo *info,
                             const std::vector<BlkInfo> &h, const double *diag0, double tol,
                             int *status, cudaStream_t s, ahlp_problem *tc = nullptr,
                             ahlp_problem *prof = nullptr, double drop = 0.0);
// inverted 64 x 64 diagonal tiles of an FP64 factor: (problem, tile) jobs of sched
cudaError_t launch_tile_inverses(const double *buf, double *tinv, const BlkInfo *info,
                                 const int *sched, int njobs, cudaStream_t s);
// inverted diagonal tiles of the current block factors (p->tinv / tinv32)
cudaError_t launch_tinv(ahlp_problem *p);
// forward wavefront solve of rhs (ordered like y) with all block factors into
// p->vec, or the backward one from p->vec and the Schur solution p->svec, which
// also writes dy; wait timeouts set p->trsv_err
cudaError_t launch_trsv(ahlp_problem *p, bool forward, const double *rhs, double *dy);
// the border system on p->svec's border part, in place
cudaError_t launch_border_solve(ahlp_problem *p);
cudaError_t launch_schur_assemble(ahlp_problem *p, double delta, double rho);
cudaError_t launch_schur_factor(ahlp_problem *p);
// cyclic reduction of the link chain: factor (T_j, Linv_j, GL_j, GR_j, and Z
// into Et); forward solve of svec's link part into bcr_pub, backward solve in
// place on svec's link part
cudaError_t launch_bcr_factor(ahlp_problem *p);
cudaError_t launch_bcr_solve(ahlp_problem *p, bool forward);
cudaError_t launch_solve(ahlp_problem *p, const double *r_d, const double *r_p,
                         const double *r_c, double *dx, double *dy, double *dz, bool adjoint,
                         double *wx = nullptr, double *wc = nullptr);
cudaError_t launch_residual(ahlp_problem *p, const double *r_d, const double *r_p,
                            const double *r_c, const double *dx, const double *dy,
                            const double *dz, double *e_d, double *e_p, double *e_c,
                            bool adjoint);

// ---- vector utilities ------------------------------------------------------
enum RedOp { RED_DOT = 0, RED_MAXABS = 1, RED_MINSTEP = 2, RED_MIN = 3, RED_SUM = 4, RED_STEP = 5 };
// one reduction of a set: out <- reduce(op, a, b [, c, d, s1, s2]) over len entries
struct RedOne {
  int op;
  const double *a, *b;
  long long len;
  double *out;
  const double *c = nullptr, *d = nullptr;
  double s1 = 0.0, s2 = 0.0;
};
constexpr int kRedSetMax = 12;   // reductions per launch
constexpr int kMdotParts = 608;  // CTAs of a multi-dot, at most
cudaError_t launch_reduce_set(ahlp_problem *p, const RedOne *ops, int n);
// out <- reduce(op, a, b) over len entries, deterministic order; out is a
// device scalar.
cudaError_t launch_reduce(ahlp_problem *p, int op, const double *a, const double *b,
                          long long len, double *out);
cudaError_t launch_spmv(const SpMat &A, const double *x, double *y, double alpha,
                        const double *yadd, cudaStream_t s);   // y = yadd + alpha A x (yadd may be null)
cudaError_t launch_axpby(double *y, const double *x, double a, double b, long long n,
                         cudaStream_t s);  // y = a x + b y
// generic elementwise kernels for the IPM
cudaError_t launch_ipm_rc(double *rc, const double *x, const double *z, const double *dxa,
                          const double *dza, double sigma_mu, long long n, cudaStream_t s);
cudaError_t launch_fill(double *y, double v, long long n, cudaStream_t s);
cudaError_t launch_add_scalar(double *y, const double *x, double s, long long n,
                              cudaStream_t st);   // y = x + s
constexpr int kMaxKrylov = 64;   // cap on GMRES iterations per solve
// out[i] = <V_i, w>, i < k (V_i = V + i*ld), deterministic
cudaError_t launch_mdot(ahlp_problem *p, const double *V, long long ld, int k, const double *w,
                        long long len, double *out);
// w += sign * sum_i coef[i] V_i (coef on the device, fixed order over i); with
// nrm2 also nrm2[0] = <w, w> and nrm2[1] = 1 / |w| (1 when <w, w> is not positive)
cudaError_t launch_maxpy(ahlp_problem *p, const double *V, long long ld, int k, const double *coef,
                         double *w, long long len, double sign = 1.0, double *nrm2 = nullptr);
// w += sum_i coef[i] V_i, coefficients from the host, for w in three pieces of
// lengths n0, n1 and len - n0 - n1
cudaError_t launch_maxpy3(ahlp_problem *p, const double *V, long long ld, int k,
                          const double *coef, double *w0, long long n0, double *w1, long long n1,
                          double *w2, long long len);
// y = a x, the factor on the device when da is not null
cudaError_t launch_scale(double *y, const double *x, const double *da, double a, long long len,
                         cudaStream_t s);
// dx, dz of a direction from dy (and the right-hand side's f, r_c); with wx, wc
// also the first and third parts of J (dx, dy, dz) (adjoint: J')
cudaError_t launch_finish(ahlp_problem *p, const double *dy, const double *rc, double *dx,
                          double *dz, bool adjoint, double *wx, double *wc);
// dst <- src over n 32-bit words, two pieces, then *seq = val, all in host memory
cudaError_t launch_publish(const unsigned *src, unsigned *dst, int n, const unsigned *src2,
                           unsigned *dst2, int n2, unsigned *seq, unsigned val, cudaStream_t s);
// up to four copies of doubles in one launch
struct CopySet {
  const double *src[4];
  double *dst[4];
  long long n[4];
};
cudaError_t launch_copies(const CopySet &c, cudaStream_t s);
cudaError_t launch_mul(double *y, const double *a, const double *b, double scale, long long n,
                       cudaStream_t s);   // y = scale * a .* b
// centrality corrector right-hand side: rc2 = rc + t, where v = (x + ap dx) .* (z + ad dz)
// is projected onto [lo, hi] and t = proj(v) - v, bounded below by -hi
cudaError_t launch_centrality_rc(double *rc2, const double *rc, const double *x,
                                 const double *dx, double ap, const double *z, const double *dz,
                                 double ad, double lo, double hi, long long n, cudaStream_t s);
cudaError_t launch_step_dot(ahlp_problem *p, const double *x, const double *dx, double ap,
                            const double *z, const double *dz, double ad, long long n,
                            double *out);  // (x+ap dx)'(z+ad dz)

// ---- tensor-core trailing update (k_tc.cu) -----------------------------------
// staging, job offsets and tensor maps for the FP32 factors (needs aug32);
// false when the driver has no tensor-map encoder
bool tc_setup(ahlp_problem *p);
cudaError_t launch_update_tc(ahlp_problem *p, int k, cudaStream_t s, LookAhead *la);
// the same for float-float factors: FP16 digit staging and job offsets
bool oz_setup(ahlp_problem *p);
cudaError_t launch_update_oz(ahlp_problem *p, int k, cudaStream_t s, LookAhead *la);

// the same for FP64 factors: eight-digit staging, job offsets, tensor maps
bool dz_setup(ahlp_problem *p);
cudaError_t launch_update_dz(ahlp_problem *p, int k, cudaStream_t s, LookAhead *la);
// update jobs of every step (called by the three set-ups)
void jobs_setup(ahlp_problem *p);

// ---- kernel-class timer (option profile_kernels) -----------------------------
// kt_mark records an event on s that ends the previous mark's interval and
// opens one of class cls (0 diagonal tiles, 1 panels, 2 trailing updates,
// 3 closes without opening); kt_collect, after the stream has synchronised,
// sums the intervals per class into kt_ms and their counts into kt_n
void kt_mark(ahlp_problem *p, int cls, cudaStream_t s);
void kt_collect(ahlp_problem *p);

// ---- host runtime helpers (api.cpp) -------------------------------------------
// device allocations owned by the handle (freed at destroy); throw Fail
void *dalloc_bytes(ahlp_problem *p, size_t bytes);
void *dupload_bytes(ahlp_problem *p, const void *h, size_t bytes);
bool is_device_ptr(const void *ptr);
const double *stage_in(ahlp_problem *p, const double *v, long long n, double *staging);
int set_err(ahlp_problem *p, int code, const std::string &msg);
void read_scalars(ahlp_problem *p, int k);
// Read up to two pieces of device memory (32-bit words) back into pinned host
// memory: a kernel writes them there, then a sequence word the host polls.
// Everything launched on the stream before it is complete on return.  A memcpy
// and a stream synchronisation cost about 9 us more, and a solve reads back once
// per Krylov step and twice besides.
void read_back(ahlp_problem *p, const void *src, void *dst, int words, const void *src2 = nullptr,
               void *dst2 = nullptr, int words2 = 0);
// ff_nan_up: a NaN pivot of a float-float factor refactors in FP64 (else the
// call returns AHLP_ERR_NOT_SPD and the caller picks the next safeguard)
int factor_impl(ahlp_problem *p, double delta, double rho, double pivot_tol,
                bool ff_nan_up = true);
// tol_override > 0 replaces refine_tol as the FGMRES target
int solve_impl(ahlp_problem *p, const double *rd, const double *rp, const double *rc, double *dx,
               double *dy, double *dz, bool adjoint, ahlp_solve_info *info,
               double tol_override = 0.0);
void ck(cudaError_t e, const char *what);   // throws on error

struct Fail {
  int code;
  std::string msg;
};

// Device memory that a handle takes while a scope is open is given back at its
// end unless the scope is kept: a set-up whose later allocation fails leaves
// nothing behind.  Pointers go to the handle once everything has succeeded.
struct AllocScope {
  explicit AllocScope(ahlp_problem *q) : p(q), mark(q->allocs.size()) {}
  ~AllocScope();
  ahlp_problem *p;
  size_t mark;
  bool keep = false;
};

}  // namespace ahlp
