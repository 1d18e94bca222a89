// rh_kernels.h -- device data layout and kernel launchers of librh.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "batch_plan.h"

namespace rh {

// Phases of the direction kernel (one bit each, executed in this order).
enum : unsigned {
    PH_WLOAD = 1u << 0,    // W (or identity columns) -> rows n_x.. of V; zero row
    PH_SPMUL = 1u << 1,    // V[x rows] = -J_p W                          (Alg. 2 SpMul)
    PH_L = 1u << 2,        // V <- L^{-1} V                                (BatchSparseSolve 1)
    PH_U = 1u << 3,        // V <- U^{-1} V
    PH_TPROJ = 1u << 4,    // T[x rows] = -y_x, T[p rows] = y_p            (BatchTensorProjection)
    PH_UT = 1u << 5,       // T <- U^{-T} T                                (BatchSparseSolve 2)
    PH_LT = 1u << 6,       // T <- L^{-T} T
    PH_MULADD = 1u << 7,   // HW = y_p + J_p^T psi                         (SpMulAdd)
};

// A bus-level schedule: level l holds the bus blocks slots[ptr[l] .. ptr[l+1]),
// maxext[l] = their longest row part.  Slots are packed descriptors
//   forward  {q, n, rp, rpv}: theta row q, n columns left of the bus (or left of
//            the dense tail for the tail's external phase), row parts at rp / rpv
//            (rpv = -1 for a PV bus);
//   backward {q, n, ue0, ue1}: U parts right of the bus at ue0 / ue1 (-1: PV).
struct LevelSet {
    int n_lev;
    const int *ptr;
    const int4 *slots;
    const int *maxext;
};

// Read-only grid data used by the direction kernel, all device pointers.
struct DirGrid {
    int n_x, n_p;
    int nnz;                                   // positions of the pattern of A (index checks)
    int zero_row;                              // n_x + n_p: a row of zeros in V
    // columns of the filled matrix A = L + U (CSR) and 1/diagonal
    const int *col;
    const double *invdiag;
    LevelSet lf, lb;                           // full forward / backward schedules
    LevelSet sf, sb, ef;                       // sparse part only, and the tail's external phase
    LevelSet sbr;                              // sb restricted to the rows of J_p and their ancestors
    int t0, T;                                 // dense trailing block [t0, t0 + T)
    // Unit-diagonal factors used by k_dirs (J_x = D L'' U', D = diag(U)): values of
    // L'' and U' in A's pattern and transposed, the dense tail's triangles of L'',
    // U', U'^T, L''^T, and D^-1 J_p by p index (jptvd)
    const double *Ad, *Atd;
    const double *triLd, *triUd, *triUtd, *triLtd;
    const double *jptvd;
    // bus structure by theta row: theta row of the bus owning row q; the bus's
    // elimination-tree parent as 2 * (its theta row) + (1 if it has a v row), or -1
    // for a root or a parent in the dense tail
    const int *qtheta, *bparent;
    // J_p by internal rows and by p index; rows with and without entries
    const int *jp_ptr, *jp_col;
    const double *jpv;
    int n_jp_rows, n_jp_zero;
    const int *jp_rows, *jp_zero_rows;
    const int *jpt_ptr, *jpt_row;
    const double *jptv;
    // narrow-level k-split cap of the sweeps: lanes per row at most (1, 2, 4, ..., 32)
    int ks_cap;
    // projection data (per bus, original ids); rows are V/Y row indices
    int n_bus;
    const int *tp_bus;                         // bus processing order (internal order, slack last)
    const int *uth, *uv;                       // rows of theta_b (zero row at the slack) and v_b
    const int *tp_l0;                          // position of (v, theta) in Atd for a PQ bus of forward level 0, else -1
    const int *inc_ptr, *inc_uth, *inc_uv;     // incident branches: rows of the other end
    const double4_32a *inc_coef;               // (K, -a, b, -c) per incidence (state dependent)
    const double *d2, *asum, *csum;            // per-bus coefficients (state dependent)
    const uint8_t *has_gref;
    const double *gref_th, *gref_v;            // grad P_slack at the rows of bus b
    int n_gref;
    const int *gref_row;
    const double *gref_val;
    const double *c2ref;                       // device scalar c''_slack
    const int *pg_row;                         // per bus: row of Pg (or -1)
    const double *pg_curv;                     // per bus: c''_k
};

struct DirLaunch {
    int N;                     // directions in this launch
    int n_cta;                 // CTAs; CTA c owns directions [c*N/n_cta, (c+1)*N/n_cta)
    // Layout of V and T: element (row r, direction c0 + d) of CTA c is at
    //   cta_stride > 0 (panel-major): c * cta_stride + r * ld + d   (each CTA's panel contiguous)
    //   cta_stride = 0 (interleaved):  r * ld + c0 + d              (ld >= N)
    int64_t ld;
    int64_t cta_stride;
    double *V, *T;             // tangent buffer; buffer of the transposed sweeps / projection
    const double *W;           // n_p x N column-major (ldw), or NULL for identity columns
    int64_t ldw;
    int col0;                  // identity columns start at col0
    double *HW;                // n_p x N column-major (ldhw)
    int64_t ldhw;
    unsigned phases;
    int64_t ws_elems;          // doubles of V and of T each (0: not stated; index checks of the bounds build)
    int use_tail;              // dense tail in shared memory (needs T * ceil(N / n_cta) <= 4096)
    int use_reach;             // identity W: forward L sweep only over the reach of B's nonzeros (needs use_tail,
                               // and phases L and U in the same launch)
    // identity W: direction j is column colmap[col0 + j] of the identity and writes that
    // column of HW (relative to HW: colmap[col0 + j] - col0); NULL: column col0 + j
    const int* colmap;
    // identity W with use_reach: each CTA's reach precomputed on the host (NULL: found at
    // run time, a bit mask grown level by level)
    const struct ReachSched* reach;
};

// The reach of every CTA of one identity-W launch (N directions on n_cta CTAs, columns
// through colmap): for CTA c, the sparse buses its J_p columns can make nonzero in the
// forward L sweep (those columns' buses and their ancestors), as forward-sweep slots
// grouped by level (only the CTA's nonempty levels), and the bit mask of their rows.
struct ReachSched {
    int n_cta, words;          // CTAs; 32-bit words of a row mask ((n_x + 31) / 32)
    const int* nlev;           // [n_cta] levels of CTA c
    const int* lev0;           // [n_cta] CTA c's first entry in ptr / maxext
    const int* ptr;            // per CTA nlev + 1 offsets into slots
    const int* maxext;         // per CTA and level: longest row part
    const int4* slots;         // forward slots {q, n, rp, rpv} of the reach buses
    const unsigned* masks;     // [n_cta * words] rows of the reach
};

// Up to kMaxBatch (grid, W block) items of one batched launch, passed by value as
// the kernel parameter (about 16 KB).
struct DirBatch {
    int n_items;
    int cta_ptr[kMaxBatch + 1];
    DirGrid g[kMaxBatch];
    DirLaunch l[kMaxBatch];
};
// threads: one of the compiled CTA shapes (dirs_batch_shape_ok)
// beside: started with the launch before it on `st` (launch_dir1_batch) instead of after it
cudaError_t launch_dirs_batch(const DirBatch& B, int threads, bool beside, cudaStream_t st);
bool dirs_batch_shape_ok(int threads);
int dirs_batch_ctas_per_sm(int threads);   // resident CTAs per SM of a shape (0: not compiled)
int dirs_batch_slots(int threads);         // resident CTAs of a shape on the current device

// Grid-wide power-flow evaluation data (per bus, original ids).
struct PfGrid {
    int n_bus, n_x, ref;
    int nnz_a, nnz_jp;                 // slots of A and of J_p (index checks)
    const int *yp, *yj, *ydiag;
    const double *G, *B;
    const int *qth, *qv, *ip_v, *ip_pg;
    const int *jac_dst;
    const int *pg_slot;
    double base_mva;
    const double *c2, *c1;
    // the warp-per-entry evaluation: bus of every admittance entry, and the buses
    // [pf_wb[w], pf_wb[w + 1]) of warp w (n_pfw = 0: one thread per bus instead)
    const int *yrow, *pf_wb;
    int n_pfw;
};

struct PfState {
    double *vm, *va, *pg, *pd, *qd;  // per bus
    double *P, *Q;                   // injections (output)
    double *sc;                      // per bus: sin, cos of the angle (launch_pf_prep; NULL: not kept)
};

// ---- programmatic dependent launch --------------------------------------------
// The long chains of dependent launches (refactorisation levels, dense-tail and
// Cholesky tile columns, the triangular solves) use programmatic stream
// serialisation: the next launch is scheduled as the current one's CTAs exit
// instead of after its completion is signalled, hiding part of the launch
// latency.  Every kernel launched this way calls pdl_wait() before it touches
// memory that an earlier kernel of its chain writes (what no kernel of the chain
// writes it may read before), which returns once the previous kernel in the stream
// has completed and its writes are visible; without a previous kernel it returns
// at once.
// The first kernel of a chain is launched without the attribute (pdl = false),
// so it is fully ordered after whatever precedes it (copies, event waits).
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's CTAs start (up to their own pdl_wait) once every CTA of this one
// is here; without it they start as this kernel's CTAs exit.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- division-free elimination of dense tiles -----------------------------------
// The diagonal tiles of the dense factorisations (the refactorisation's dense
// tail LU, the tracking step's Cholesky) are eliminated by cross-multiplied steps
// a_rc <- 2^-e (d a_rc - a_rj a_jc), d the current pivot, instead of a reciprocal of
// every pivot on the critical path.  e is 0 while d lies within 2^+-64 and otherwise the
// power of two that brings |d| into [1, 2): most steps do not carry the exponent update (12
// dependent integer instructions) in their chain.  A 16 x 16 tile of the tail's LU: 8300
// cycles with the update, the own entry and its indexes in every step, 6000 without.
//
// The trailing block after j steps is s_j times the ordinary one, s_0 = 1 and s_{j+1} =
// s_j d_j 2^-e with d_j = s_j u_j, u_j the ordinary pivot.  A rescaled step takes |s| up by
// less than a factor 2; any other leaves |s_{j+1}| = d_j^2 / |u_j| between 2^-128 / max|u|
// and 2^130 / min|u|.  So |s| < 2^(130 + TB) max(1, 1 / min|u|) in a tile of TB columns, and
// no product of a step overflows while the entries a of the tile and its Schur complements
// have max|a| < 2^350 min(1, min|u|) (TB = 32).  An equilibrated Cholesky tile has |a| < 4:
// pivots down to 2^-348.  The tail's LU tiles are not equilibrated: its pivots are at least
// 1e-14 max|J_x|, or the factorisation is reported singular, which leaves its entries a
// growth of 2^300 over a max|J_x| of up to 1.
// e for a pivot d: 0 also where d is zero, subnormal, infinite or NaN and the
// factorisation has failed (|e| <= 1022, so 2^-e is normal).
__device__ __forceinline__ int pivot_shift(double d) {
    const int f = (__double2hiint(d) >> 20) & 0x7ff, e = f - 1023;
    return ((unsigned)(e + 64) > 128u && f != 0 && f != 0x7ff) ? min(e, 1022) : 0;
}

// v * 2^-sh for |sh| <= 1022 by an integer update of the exponent field, with
// the bits of the IEEE multiplication whenever v and the result are normal
// numbers; zero, subnormal, infinite and NaN v are returned as they are, a
// result below the normal range is flushed to a signed zero and one above it
// becomes a signed infinity.  Selects only, no branch: the update sits on the
// critical path of every elimination step.
__device__ __forceinline__ double scale_pow2(double v, int sh) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long sign = b & 0x8000000000000000ull;
    const int f = (int)((b >> 52) & 0x7ffu);
    const int nf = f - sh;
    unsigned long long r = b - ((unsigned long long)(long long)sh << 52);
    r = nf < 1 ? sign : r;
    r = nf > 0x7fe ? (sign | 0x7ff0000000000000ull) : r;
    r = (f == 0 || f == 0x7ff) ? b : r;
    return __longlong_as_double((long long)r);
}
#endif
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(bool pdl, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// ---- launchers (all asynchronous on `st`) ----------------------------------
void launch_injections(const PfGrid& g, const PfState& s, cudaStream_t st);
// residual (internal order) and/or Jacobian values; gmax / jmax receive
// max |g| and max |J_x| as ordered bit patterns (zeroed by the caller).
// `chained`, here and below: the operation before it on `st` is a kernel, and the launch is
// scheduled with it (see above); launch_pf_eval and launch_line_values always follow one.
// Before launch_pf_eval: sin and cos of every bus angle into s.sc and, with zero,
// A (nnz_a slots), the two maxima and *err (if given) cleared.
void launch_pf_prep(const PfGrid& g, const PfState& s, double* A, unsigned long long* umax, int* err, bool zero,
                    bool chained, cudaStream_t st);
void launch_pf_eval(const PfGrid& g, const PfState& s, double* gres, double* A, double* jpv,
                    unsigned long long* gmax, unsigned long long* jmax, bool want_jac, cudaStream_t st);
void launch_newton_update(const PfGrid& g, const PfState& s, const double* dx, bool chained, cudaStream_t st);
// Coloured forward-mode Jacobian (section 4.2.2): the injections evaluated on
// dual numbers whose tangents are the seed colours (col_th, col_v, col_pg per
// bus), in chunks of tangents; writes the J_x slots of A (and max |J_x| into
// jmax) and the J_p values.  The residual comes from launch_pf_eval.
cudaError_t launch_jac_ad(const PfGrid& g, const PfState& s, const int* col_th, const int* col_v, const int* col_pg,
                          int n_colors, double* A, double* jpv, unsigned long long* jmax, cudaStream_t st);
// Fixed-pattern LU refactorisation data (device pointers).
struct RfGrid {
    int n_x, t0, T;                    // dense trailing block [t0, n_x), T = n_x - t0
    int nnz;                           // positions of A (index checks)
    double* tailD;                     // T x T row-major scratch of the tiled dense LU
    const int* tail_pos;               // (i, j) of the trailing block -> position in A, -1 if structurally zero
    const int *rf_lev_bus, *q0;
    const uint8_t *nv;
    const int *rowptr, *col, *diagpos, *tpos;
    const int *tgt_pos;                // update targets (positions in A; -1: empty lane), grouped by level
    // 3 int2 per group: {dt (first level) or bus k (later levels), dv}, {a_it, a_tj},
    // {a_iv, a_vj} positions; grp: each target's first group (all -1: none), xgrp:
    // its further groups [xptr[t], xptr[t + 1])
    const int2 *grp, *xgrp;
    const int64_t *xptr;
    const int4 *lev;                   // per level: first target, targets, first pivot job, pivot jobs
    // pivot quantities per sparse bus (1/u_tt, l_vt, 1/u_vv, u_tv), written by the
    // pivot jobs (bus piv_bus[q], block positions piv_pos[4 q ..]; see launch_refactor)
    double4_32a *piv;
    int n_piv;
    const int *piv_bus, *piv_pos;
    // pivot steps by entry (k_rf_pivot): bus and positions {a_tj, a_vj, a_jt, a_jv}
    int64_t n_pe;
    const int *pe_bus;
    const int4 *pe_pos;
    double *A, *invdiag;
    double *triLd, *triUd, *triUtd, *triLtd;   // the tail's triangles, written with it when tail_in_one(T)
    const unsigned long long *jmax;
    int *err;
};
// Whether launch_refactor factors the dense tail in one CTA and writes its triangles too
// (launch_build_tail and launch_tail_tri_batch then do nothing).
constexpr int kTailOne = 64;
inline bool tail_in_one(int T) { return T > 0 && T <= kTailOne; }
// L2 prefetch of up to 8 read-only device arrays (16-byte aligned; the bytes of
// each are rounded down to a multiple of 16); `first` is filled by the launcher.
struct PrefetchList {
    int n;
    const char* p[8];
    unsigned long long bytes[8];
    unsigned long long first[9];
};
void launch_prefetch_l2(const PrefetchList& L, cudaStream_t st);
// One update launch per level (its pivot jobs [piv_lev_ptr[l], piv_lev_ptr[l + 1])
// at the front), the pivot steps of every sparse bus, then the dense tail's LU.
cudaError_t launch_refactor(const RfGrid& g, const int* lev_ptr_host, const int64_t* tgt_lev_ptr_host,
                            const int* piv_lev_ptr_host, int n_lev, cudaStream_t st);
// Ad / Atd (the unit-diagonal factors L'', U' of J_x = D L'' U' and their transpose), jptv
// (J_p by p index) and jptvd (D^-1 J_p by p index)
void launch_transpose_values(int nnz, const int* tpos, const int* arow, const int* col, const int* diagpos,
                             const double* A, const double* invdiag, double* Ad, double* Atd, int nnz_jp,
                             const int* jpt_src, const int* jpt_row, const double* jpv, double* jptv, double* jptvd,
                             cudaStream_t st);
void launch_dirs(const DirGrid& g, const DirLaunch& L, cudaStream_t st);
// raise the dynamic shared-memory limits of the kernels that need it (once per grid)
cudaError_t prepare_kernels();
bool dirs_tail_fits(int T, int N, int n_cta);
int dirs_tail_cap();       // dense-tail rows x directions a CTA can hold
// dense tail triangles of the current factors (pos: T*T map to A, -1 where structurally zero)
// x[r][c] *= s[r] for r < n, c < N
void launch_scale_rows(int n, int N, const double* s, double* x, int64_t ld, cudaStream_t st);
void launch_build_tail(int T, int t0, const int* pos, const double* A, const double* invdiag, double* triLd,
                       double* triUd, double* triUtd, double* triLtd, cudaStream_t st);
// One right-hand side in one CTA with x in shared memory: mode 2 also keeps the
// dense tail triangle there (needs the tail triangles built), 1 without it,
// 0 when x does not fit (use the direction kernel instead).
int solve1_mode(int n_x, int T);
// Its schedule: steps of line_threads(n_x) descriptors {q, base, b, w} each, built by
// line_steps from the level lists (kernels.cu explains the descriptor).
constexpr int kLineRegs = 512;        // threads an SM holds at 128 registers
constexpr int kLinePre = 8;           // entries a lane holds ahead
// LineBits, the fields of a descriptor's w: the warp's entries per lane, log2(G), the warp's
// largest log2(G), and the flags
constexpr int kLineCntMask = 0xff, kLineLg = 8, kLineWlg = 11;
constexpr int kLineExt = 1 << 26;     // rows of the dense tail, subtract only
constexpr int kLineSync = 1 << 27;    // barrier after the step (its level ends)
constexpr int kLineSplit = 1 << 28;   // a bus of two rows: a group of lanes for each, side by side
constexpr int kLineActive = 1 << 30;  // the warp has a bus in this step
struct LineSched {
    int n, n_ent, n_vt;               // steps, entries and buses' own entries of the line arrays
    const int4* steps;
    const int* col;                   // line arrays: column of each entry (n_x: a pad),
    const double* val;                //   its value negated (0: a pad), and each bus's own
    const double* vt;                 //   off-diagonal entry negated
};
struct LineGrid {
    int n_x, t0, T, nnz;              // nnz: positions of the pattern of A (index checks)
    LineSched up, down, tup, tdown;   // with L'', U', and with U'^T, L''^T
    int n_line;                       // entries of the line arrays [up | down | up's vt | down's vt]
    const int *map, *arow, *col, *tpos, *diagpos;   // their positions in A (-1: a pad); A's rows, columns, ...
    double *line, *tline;             // their values, of the factors and of their transpose
    const double *A, *invdiag;
    const double *triLd, *triUd, *triUtd, *triLtd;
};
void launch_line_values(const LineGrid& g, bool transposed_too, cudaStream_t st);
// The direction kernel's unit-diagonal factors from the line values and the tail's triangles
struct LineCopies {
    const int* tail_pos;
    double *Ad, *Atd, *triLd, *triUd, *triUtd, *triLtd;
};
cudaError_t launch_copies_from_lines(const LineGrid& g, const LineCopies& o, bool use_tail, cudaStream_t st);
int line_threads(int n_x);
cudaError_t launch_solve1(const LineGrid& g, const double* x, double* out, bool trans, bool use_tail, bool chained,
                          cudaStream_t st);          // out may be x
// Directions of a launch with one direction per CTA and x in shared memory (L.N CTAs;
// direction c's rows at V + c * (zero_row + 1) and T likewise): SpMul to the U sweep, the
// projection to SpMulAdd, or both.  Needs solve1_mode() > 0 and its schedule.
cudaError_t launch_dir1(const DirGrid& g, const LineGrid& s, const DirLaunch& L, bool use_tail, cudaStream_t st);

// Several items with one direction per CTA; all of line_threads(n_x) == 512.
struct Dir1Batch {
    int n_items;
    int cta_ptr[kMaxBatch + 1];
    DirGrid g[kMaxBatch];
    LineGrid s[kMaxBatch];
    DirLaunch l[kMaxBatch];
};
static_assert(sizeof(Dir1Batch) <= 32764, "kernel parameters");
cudaError_t launch_dir1_batch(const Dir1Batch& B, cudaStream_t st);

// Dense Cholesky of the tracking step (dense.cu).  A, L, B, work, y and info
// are device pointers; column-major.  info receives 0 or the 1-based column of
// the first pivot that is not positive.  launch_potrf with y != NULL also runs
// the forward solve L y = b in place on the vector y (b on entry).
// launch_potrs: work holds n * nrhs doubles; with forward = false it only runs
// the backward sweep L^T X = work, writing X into B.
// ---- Newton power flow over several grids of one topology (load scenarios) ----
// Every batched launch takes item i from blockIdx.y (blockIdx.x for the solve):
// the grids share their symbolic data, so every level range is the same for all.
constexpr int kMaxPfBatch = 32;
struct PfBatchItem {
    PfGrid g;
    PfState s;
    double *A, *jpv;            // J_x values (in A's slots), J_p values
    double* x;                  // residual in, Newton step out (internal order)
    unsigned long long* umax;   // max |g|, max |J_x| as ordered bits
    int* err;                   // pivot flag of the refactorisation
};
struct PfBatch {
    int n, max_bus;
    PfBatchItem it[kMaxPfBatch];
};
struct RfBatch {
    int n;
    RfGrid g[kMaxPfBatch];
};
struct TriBatch {
    int n, T, t0;
    const int* pos[kMaxPfBatch];
    const double *A[kMaxPfBatch], *invdiag[kMaxPfBatch];
    double *triLd[kMaxPfBatch], *triUd[kMaxPfBatch];
};
struct Solve1Batch {
    int n;
    LineGrid g[kMaxPfBatch];
    double* x[kMaxPfBatch];
};
// residual and Jacobian of every item (after launch_pf_prep_batch)
void launch_pf_eval_batch(const PfBatch& B, cudaStream_t st);
// every item's sin/cos per bus, A and the maxima cleared (not the pivot flag)
void launch_pf_prep_batch(const PfBatch& B, cudaStream_t st);
// out[2 i] = max |g| of item i, out[2 i + 1] = its pivot flag
void launch_batch_status(const PfBatch& B, double* out, cudaStream_t st);
cudaError_t launch_refactor_batch(const RfBatch& B, const int* lev_ptr_host, const int64_t* tgt_lev_ptr_host,
                                  const int* piv_lev_ptr_host, int n_lev, cudaStream_t st);
// the dense tail's triangles of the single solves (L'' and U')
void launch_tail_tri_batch(const TriBatch& B, cudaStream_t st);
cudaError_t launch_solve1_batch(const Solve1Batch& B, bool use_tail, int n_x, int T, cudaStream_t st);
void launch_newton_update_batch(const PfBatch& B, bool chained, cudaStream_t st);

int dense_tile(int n);
cudaError_t launch_potrf(int n, double* A, int64_t lda, int* info, double* y, cudaStream_t s);
cudaError_t launch_potrs(int n, const double* L, int64_t ldl, double* B, int64_t ldb, int nrhs, double* work,
                         bool forward, cudaStream_t s);
int dirs_default_ctas(int N);
// CTA slots of the direction kernel on a device of n_sm SMs, and the CTAs a launch of
// N directions takes there
int dirs_cta_slots_for(int n_sm);
int dirs_ctas_for(int N, int slots);
// CTAs of k_dirs the device holds at once (CTAs per SM x SMs)
int dirs_cta_slots();
int num_sms();             // SMs of the current device (1 if the query fails)

// adjoint helpers
struct AdjData {
    double *rhs;          // n_rhs >= n_x, internal order (output: -grad_x f, zero beyond)
    int n_rhs;
    double *cref, *c2ref; // device scalars c'_slack, c''_slack
    double *F;            // device scalar
    double *gref_th, *gref_v;   // per bus
    int *gref_row;        // up to n_gref_max entries
    double *gref_val;
    int n_gref;           // number of entries (static: slack + its neighbours)
    const int *uth, *uv;  // combined rows per bus
};
void launch_adjoint_rhs(const PfGrid& g, const PfState& s, const AdjData& a, cudaStream_t st);
// Once lambda is there: the projection's coefficients and grad F
struct CoefData {
    const double *lam, *cref, *gref_v;
    const int* inc_ptr;
    double4_32a* coef;          // per incidence
    double *d2, *asum, *csum, *pg_curv;
    const int *jpt_ptr, *jpt_row;
    const double* jptv;
    double* grad;
};
void launch_adjoint_coef(const PfGrid& g, const PfState& s, const CoefData& c, bool chained, cudaStream_t st);

// permutation helpers between external (x, p) order and the internal rows
void launch_gather_rows(int n_rows, int N, const int* map, const double* src, int64_t lds, double* dst,
                        int64_t ldd, double scale_x, int n_x, cudaStream_t st);
void launch_scatter_rows(int n_rows, int N, const int* map, const double* src, int64_t lds, double* dst,
                         int64_t ldd, double scale_x, int n_x, cudaStream_t st);

}  // namespace rh
