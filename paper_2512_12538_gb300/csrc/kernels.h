// kernels.h -- host-side launchers of the libhh CUDA kernels (internal header).
#pragma once
#include <cuda_runtime.h>
#include "hh_core.cuh"

namespace hh {

// Counts kernel launches made by this library (process-wide); see hh_launch_count().
void note_launch();

// ---- field kernels (k_field.cu) ----------------------------------------------------
// y = (v ? v : 0) - sgn * A~ x  on a band (b rows, Sx cols, nc columns per point).
// With `v` null and sgn = -1 this is y = A~ x.  If `part` is non-null each block writes
// its partial sum of |y|^2 to part[blockIdx.x] (nblk_out receives the block count).
template <typename TX, typename TV, typename TY>
void launch_apply(const cplx<TX>* x, const cplx<TV>* v, cplx<TY>* y, OpGeom g, int nc, double sgn,
                  double* part, int* nblk_out, cudaStream_t s);

// y = v - A x (FP64, one column) with per-block |y|^2 partials, and yt = y rounded to T.
// gate (may be null): when the device word is nonzero at launch, nothing is done.
template <typename T>
void launch_residual_cast(const c128* x, const c128* v, c128* y, cplx<T>* yt, OpGeom g, double* part, int* nblk_out,
                          cudaStream_t s, const int* gate = nullptr);

// Residuals of up to RB_MAX_JOBS problems in one launch: per job yt = v - A x (FP64) rounded
// to T and *norm = ||v - A x||^2 (fixed-order sums).  part: scratch of part_cap doubles.
constexpr int RB_MAX_JOBS = 32;
struct ResidJob {
    const c128* x;
    const c128* v;
    void* yt;
    double* norm;
    OpGeom g;
    unsigned blk0, nblk;   // set by the launcher
};
struct ResidBatch {
    ResidJob job[RB_MAX_JOBS];
    int njobs;
};
template <typename T>
void launch_residual_batch(ResidBatch bt, double* part, int part_cap, cudaStream_t s);

// out = sum of n doubles (deterministic single-block reduction)
void launch_sum(const double* part, int n, double* out, cudaStream_t s);
// launch_residual_cast with the stopping test of the stationary iteration kept on the
// device, in the same launch.  Unless ctl[0] is already set (then nothing is done):
// y (may be null: not stored), yt and the partials as launch_residual_cast, then
// nrm[0] = ||y||^2 (launch_sum's order), ctl[1] += 1, and with rel = sqrt(nrm[0] / nrm[2]) (0 when nrm[2] is 0)
// ctl[0] = 2 if rel is not finite, 1 if rel < tol.  ctl[0] is the gate of the next
// step's launches; ticket is a device counter that is zero between launches.
template <typename T>
void launch_residual_stop(const c128* x, const c128* v, c128* y, cplx<T>* yt, OpGeom g, double* part, double* nrm,
                          int* ctl, unsigned* ticket, double tol, cudaStream_t s);

// b = h^2 w_i w_j f + h (w_j gx + w_i gy) for the global problem (q1: the bilinear
// elements' load vector, h^2 M_y F M_x^T + h (edge masses) g).
// the right-hand side b with |b|^2 into *b2, and as wanted (not null) u = 0, the residual b in the
// leaf precision and in FP64, its squared norm, the stop words; nclear ints from clear are zeroed;
// part: a double a block (608 at most), ticket: zero between launches
template <typename T> struct StartOut {
    c128* u = nullptr;
    cplx<T>* rt = nullptr;
    c128* res = nullptr;
    double *b2 = nullptr, *r2 = nullptr;
    int* ctl = nullptr;
    int* clear = nullptr;
    int nclear = 0;
};
template <typename T>
void launch_start(const c128* f, const c128* g, c128* b, const StartOut<T>& o, int dim, int S, double h, int q1,
                  double* part, unsigned* ticket, double tol, cudaStream_t s);

// dst[i] (+)= (TD) src[i], i < n
template <typename TS, typename TD>
void launch_copy(const cplx<TS>* src, cplx<TD>* dst, size_t n, bool accumulate, bool conjugate,
                 cudaStream_t s);

// Y[x][c] = boundary row of A~_s applied to u: u_if = row on the sibling's artificial
// boundary, u_in = the next row inward (both rows of the child's solution).
template <typename T>
void launch_robin_trace(const cplx<T>* u_if, const cplx<T>* u_in, cplx<T>* Y, int b_s, int Sx, int nc,
                        double kh, const double* khr_row, cudaStream_t s, int q1 = 0);

// v_if/v_in = rows of A~_s B_s^T conj(Q) (the adjoint trace, conjugated for the
// conj o solve o conj adjoint); other rows untouched.
template <typename T>
void launch_adjoint_place(const cplx<T>* Q, cplx<T>* v_if, cplx<T>* v_in, int b_s, int Sx, int nc,
                          double kh, const double* khr_row, cudaStream_t s, int q1 = 0);

// Omega[x][j] (Sx x m) for child `node`: SplitMix64 + Box-Muller, re/im ~ N(0,1/2).
template <typename T>
void launch_sketch(cplx<T>* Om, int Sx, int m, int node, unsigned long long seed, cudaStream_t s);

// W[n][c] += sum_j C[n][j] y[j][c]   (n < npts, j < p, c < nc), y FP64 [p][nc]
template <typename TC, typename TW>
void launch_coarse_update(const cplx<TC>* C, const c128* y, cplx<TW>* W, size_t npts, int p, int nc,
                          cudaStream_t s);

// ---- coarse correction with a column-major basis C[j * N + pt] (k_coarse.cu) --------
template <typename T>
void launch_build_basis(const cplx<T>* src, size_t src0, int r, cplx<T>* C, size_t ldc, int coff, size_t dst0,
                        size_t n, cudaStream_t s);
// One-column coarse corrections of up to CB_MAX_JOBS nodes in one cooperative launch
// (k_coarse.cu).  Per job: basis C [p][N] (TC), right-hand side v (TV), iterate w_in
// (TW, may be null), output out (TO) for the rows [r0, r1) of the node:
//   out[pt - r0 Sx] = (acc_out ? out : 0) + (add_w ? w_in[pt] : 0) + (C y)[pt],
//   y = Minv C^H (v - A~ w_in)  (Minv in TC; y also stored in FP64 when non-null).
// partial: (total blocks) x p scratch entries of TC; bar: two zeroed words (grid
// barrier); err: the device status word (DEV_TIMEOUT if the barrier wait gives up).
constexpr int CB_MAX_JOBS = 16;
constexpr int CB_COLS = 16;   // basis columns one block of k_coarse_batch projects on (p <= 64)
struct CoarseJob {
    const void* C;
    const void* v;
    const void* w_in;
    void* out;
    const void* Minv;
    c128* y;
    OpGeom g;
    int r0, r1;
    int acc_out, add_w;
    int split;             // >= 0: columns [0, p/2) vanish on rows >= split, [p/2, p) on rows
                           // below (each child's basis lives on its owned rows); -1: dense
    unsigned blk0, nblk;   // set by the launcher
    void* dout;            // may be null: also receives the correction added to out (without
                           // out's old value), in the basis precision, at out's index
    int ngrp;              // set by the launcher: column groups per half (p/2 / CB_COLS, rounded up)
    unsigned sb[5];        // set by the launcher: blocks of set s are [sb[s], sb[s + 1])
};
struct CoarseBatch {
    CoarseJob job[CB_MAX_JOBS];
    int njobs;
    const int* gate;       // may be null: when the word is nonzero at launch, nothing is done
    long long wait_polls;  // polls of the grid barrier's wait before it gives up (set by the launcher)
    float keep;            // set by the launcher: < 1 when the launch's basis exceeds the L2 (see the kernel)
};

// Polls a bounded device-side wait makes before giving up with DEV_TIMEOUT: the
// cooperative grid barrier of the coarse corrections and the tensor-core transforms'
// waits for their operands and MMAs.  Negative: each wait's default (about a second).
// Read when a kernel is launched (a captured graph keeps the value of its capture).
// The drains after a wait gave up always use the default.
void set_wait_polls(long long polls);
long long wait_polls(long long dflt);
template <typename TC, typename TV, typename TW, typename TO>
void launch_coarse_batch(CoarseBatch bt, int p, void* partial, unsigned* bar, int* err, cudaStream_t s);
// W[pt][c] += sum_j C[j ldc + pt] y[j][c] for N points (nc columns); split_pt as
// launch_ip_partial_colA (it may be negative or past the end: one child's columns only)
template <typename TC, typename TW>
void launch_coarse_updn(const cplx<TC>* C, size_t ldc, const c128* y, cplx<TW>* W, size_t N, int p, int nc,
                        cudaStream_t s, long long split_pt);
// tiled inner products with a column-major A (p x N); split_pt >= 0: A's first p/2
// columns vanish from point split_pt on and the others before it (a node's coarse basis)
template <typename TA, typename TB, typename ACC>
int launch_ip_partial_colA(const cplx<TA>* A, const cplx<TB>* B, int ldb, size_t N, int p, int q, c128* partial,
                           int max_blocks, cudaStream_t s, long long split_pt = -1);

// Krylov bases, point-major B[n * ld + j]:
void launch_col_load(const c128* B, int ld, int col, c128* dst, size_t n, cudaStream_t s);
void launch_col_store_normalised(c128* B, int ld, int col, const c128* src, const c128* nrm2, size_t n,
                                 cudaStream_t s);
// w += sgn * B[:, :j] c   (c = conj(coef) if cj), coef on the device, j <= 128
void launch_basis_combine(const c128* B, int ld, int j, const c128* coef, bool cj, double sgn, c128* w, size_t n,
                          cudaStream_t s);

// Flexible GMRES's least-squares problem on the device (one thread): the Hessenberg
// matrix H (entry (i, j) at H[i * mk + j], mk + 1 rows), the Givens rotations (cs, sn) and
// the rotated right-hand side g of one restart cycle.
struct GmresState {
    int stop;      // 1 once the estimate is below tol / 2, the new column vanished, or not finite
    int jstop;     // columns of the cycle when it stopped
    int bad;       // 1: the estimate was not finite
    int steps;     // columns done
    double est;    // |g[steps]| / ||b||, the residual estimate
    double pad;
};
struct GmresLs {
    c128* H;       // [(mk + 1) * mk]
    double* cs;    // [mk]
    c128* sn;      // [mk]
    c128* g;       // [mk + 1]
    GmresState* st;
    int mk;
};
// start a cycle: g = (beta, 0, ...), state cleared
void launch_gmres_init(GmresLs ls, double beta, cudaStream_t s);
// column j from the dot products of the two Gram-Schmidt passes (d1, d2: conj(h_ij)) and
// ||w||^2 (dn.re): rotations, g, the estimate and the stop test; does nothing once stopped
void launch_gmres_rotate(GmresLs ls, const c128* d1, const c128* d2, const c128* dn, int j, double nbv, double tol,
                         cudaStream_t s);
// y = R^{-1} g over the first jn columns (R the rotated H)
void launch_gmres_solve(GmresLs ls, int jn, c128* y, cudaStream_t s);

// ---- dense kernels (k_dense.cu) ----------------------------------------------------
// partial[blk][i][j] = sum_{n in blk} conj(A[n*lda+i]) * B[n*ldb+j]; returns nblk.
// ACC is the accumulation precision (double, or float for complex64 working data).
template <typename TA, typename TB, typename ACC = double>
int launch_ip_partial(const cplx<TA>* A, int lda, const cplx<TB>* B, int ldb, size_t N, int p, int q,
                      c128* partial, int max_blocks, cudaStream_t s);
// out[i][j] = sum_blk partial; if Minv != null, out2 = Minv (p x p) * out  (p x q).
void launch_ip_reduce(const c128* partial, int nblk, int p, int q, c128* out, const c128* Minv,
                      c128* out2, cudaStream_t s);
// Galerkin partials: partial[blk][a][l] = sum_pts conj(C[a][pt]) (A~ C)[l][pt]  (p = 2r,
// C column-major).
// split_row >= 0: columns [0, p/2) of C vanish on rows >= split_row and [p/2, p) below it.
// Galerkin partial sums of A_c = C^H A~ C: basis stored in TI, stencil and products in T
// Returns the number of partial blocks written (partial holds max_blocks + 1 blocks of p x p).
// *herm set: the partials are in the Hermitian-packed form (FP64 products of the 5-point
// rows), and launch_herm_fill completes the summed matrix.
template <typename TI, typename T>
int launch_galerkin_partial(const cplx<TI>* C, OpGeom g, int p, int split_row, c128* partial, int max_blocks,
                            cudaStream_t s, bool* herm = nullptr);
// A[j][i] = conj(A[i][j]) + A[j][i] for i < j (p x p, row-major)
void launch_herm_fill(c128* A, int p, cudaStream_t s);
// In-place QR (classical Gram-Schmidt, two passes) of nq independent Sx x m blocks.
template <typename T>
void launch_qr(cplx<T>* const* Y, int nq, int Sx, int m, cplx<T>** dev_ptr_scratch, cudaStream_t s);
// Hermitian eigenproblems of nq m x m FP64 matrices (m <= 64): all eigenvalues
// descending in lam, the r leading eigenvectors in columns 0..r-1 of U (m x m).  Each G
// holds m^2 + 4m complex entries; the matrix is destroyed (used as workspace).
void launch_heig(c128* const* G, c128* const* U, double* const* lam, int nq, int m, int r,
                 void** dev_ptr_scratch, cudaStream_t s);
// V[x][j] = sum_k Z[x][k] U[k][j] / sqrt(lam_j)  for j < r
template <typename T>
void launch_form_v(const cplx<T>* Z, const c128* U, const double* lam, cplx<T>* V, int Sx, int m, int r,
                   cudaStream_t s);
// In-place Gauss-Jordan inverses with partial pivoting of `count` n x n FP64 matrices
// A[0..count) (count <= GJ_MAX_BATCH), one launch.
constexpr int GJ_MAX_BATCH = 32;
struct GjBatch {
    c128* A[GJ_MAX_BATCH];
    void* AT[GJ_MAX_BATCH];   // complex64 copies of the inverses (entries may be NULL)
    int n;
    int* err;
    uint32_t wait;            // polls of a wait before it gives up (set by the launcher)
};
// fp32: eliminate in FP32 (the complex64 form), else FP64.
void launch_gj_inverse(GjBatch bt, int count, bool fp32, cudaStream_t s);

// ---- leaf kernels (k_leaf.cu) ------------------------------------------------------
struct LeafTask {
    void* X;          // factor store: Sx steps of b x ldx blocks (2D) or b diagonal inverses (1D)
    const void* F;    // right-hand sides [b][Sx][nrhs]
    void* W;          // solutions [b][Sx][nrhs]
    int b;
    int ldx;
    const double* khr;   // k h per row of the band (layered media) or null: the launch's kh
};
template <typename T>
void launch_factor(const LeafTask* d_tasks, int ntasks, int b_max, int Sx, double kh, int* err,
                   cudaStream_t s);
template <typename T>
void launch_sweep(const LeafTask* d_tasks, int ntasks, int b_max, int Sx, int nrhs, int* err,
                  cudaStream_t s);
int leaf_ldx(int b, int elem_bytes);
// tallest band the explicit-inverse path factors (shared-memory bound of k_factor2d)
int leaf_block_bmax(int elem_bytes);

// ---- eigenbasis leaf path (k_eig.cu) -------------------------------------------------
struct EigTask {
    void* V;          // [b][b] generalised eigenvectors of the column pencil (V^T W V = I)
    void* xi;         // [Sx][b] scalar Schur recursion coefficients
    void* lam;        // [b] eigenvalues (complex128)
    const void* F;    // right-hand sides [b][Sx][nrhs]
    void* Fh;         // transformed right-hand sides / solutions [b][Sx][nrhs]
    void* W;          // solutions [b][Sx][nrhs]
    int b;
    int Sx;           // columns of the leaf's problem (tasks of several problems may share a launch)
    int w0, w1;       // the sweep writes local rows [w0, w1) only, row a to W + (a - w0) Sx nrhs
                      // (all rows: w0 = 0, w1 = b)
    const void* vt_emb;   // complex64 form: V^T and V as the tensor-core transforms' B operand
    const void* vn_emb;   // (tc_prepare_v layout; null where the transforms run on CUDA cores)
    void* sc;             // bilinear elements: [b] per-mode scale of the recursions' input
                          // (null: the 5-point rows, scale 1)
};

// Layout of the transformed vectors Fh of a multi-vector sweep (b rows of J = Sx nrhs):
// up to 15 right-hand sides line by line, [m][c][i] (each scalar recursion reads one
// contiguous line; one warp per line); from 16 on in the node order [m][i][c] (one lane
// per right-hand side, a warp's loads contiguous).  fh_col: the Fh column of node column jj.
HH_HD bool eig_line_major(int nrhs) { return nrhs <= 15; }
HH_HD size_t fh_col(size_t jj, int Sx, int nrhs) {
    return eig_line_major(nrhs) ? (jj % (size_t)nrhs) * (size_t)Sx + jj / (size_t)nrhs : jj;
}

// ---- tensor-core transforms (k_tc.cu) -----------------------------------------------
// Bytes of one B operand (one leaf, one transform) for bands of up to b_max rows.
size_t tc_vemb_bytes(int b_max);
// Fills every task's vt_emb / vn_emb from its V (complex64).
void launch_tc_prepare_v(const EigTask* d_tasks, int ntasks, int b_max, cudaStream_t s);
// 1 when the transform kernel can run on the current device (its shared-memory limit set).
int tc_transform_ready();
// The complex64 sweep transforms on the tensor cores: which = 0, Fh = V^T F; which = 1,
// W = V Fh (layouts as the three-stage sweep).  err: device status word (DEV_TIMEOUT on a
// bounded wait that gave up).  gate (may be null): a device word; when it is nonzero at launch
// the launch does nothing.
void launch_tc_transform(int which, const EigTask* d_tasks, int ntasks, int b_max, int Sx, int nrhs, int* err,
                         cudaStream_t s, const int* gate = nullptr);
template <typename T>
void launch_eig_factor(const EigTask* d_tasks, int ntasks, int b_max, int Sx, double kh, int* err,
                       cudaStream_t s, int q1 = 0);
template <typename T>
void launch_eig_sweep(const EigTask* d_tasks, int ntasks, int b_max, int Sx, int nrhs, cudaStream_t s);
// One right-hand side (nrhs = 1, F/W [b][Sx]): the three stages in one launch, one
// thread-block cluster per leaf.  eig_sweep_fused_ready (call outside stream capture)
// prepares the kernel and returns the cluster size to launch with (16 or 8), or 0 when
// leaves of up to b_max rows do not fit a cluster's shared memory; the caller then runs
// the three stages instead.
constexpr int FS_SMEM_MAX = 220 * 1024;
template <typename T>
int eig_sweep_fused_ready(int b_max, int Sx);
// whether clusters of `cl` CTAs can run the one-launch sweep for these sizes
template <typename T>
bool eig_sweep_fused_feasible(int cl, int b_max, int Sx);
// b_max, Sx: the largest band and column count among the tasks (shared-memory size).
// gate (may be null): a device word; when it is nonzero at launch the launch does nothing.
template <typename T>
void launch_eig_sweep_fused(int cl, const EigTask* d_tasks, int ntasks, int b_max, int Sx, cudaStream_t s,
                            const int* gate = nullptr);
// stage 0: f^ = V^T f; 1: scalar recursions; 2: x = V x^.  gate as launch_eig_sweep_fused.
template <typename T>
void launch_eig_sweep_stage(int stage, const EigTask* d_tasks, int ntasks, int b_max, int Sx, int nrhs,
                            cudaStream_t s, const int* gate = nullptr);
int eig_bmax();

// ---- the iteration on the cut rows (k_cut.cu) ---------------------------------------
constexpr int CUT_MAXL = 6;               // levels of the hierarchy it takes
constexpr int CUT_KMAX = 32 * CUT_MAXL;   // basis columns at one cut row (r <= 32 per level)
constexpr int CUT_MGMAX = 40;             // modes of one item
constexpr int CUT_KG = 8;                 // shares of the columns in the update
constexpr int CUT_MAXD = 4096;            // corrections of one problem, 2 r (2^L - 1)
constexpr int CUT_NCUT = (1 << CUT_MAXL) - 1;
// why the steps stopped: the FP64 test is due, a new round is due, the step limit, not
// finite, no longer contracting (where that is asked for)
enum CutReason : int { CUT_TEST = 1, CUT_ANCHOR = 2, CUT_LIMIT = 3, CUT_NONFINITE = 4, CUT_STALL = 5 };
struct CutCtl {
    int it, in_round, reason, chk_it;
    double n2, n0;        // |v|^2 after the last step; the FP64 |r|^2 the round started from
    double best, chk;     // smallest |v|^2 so far, and that at step chk_it
    double ns[3];         // profiled phases (ns): leaf lines, projections and y, update
};
struct CutLeaf {
    const void *V, *xi, *sc;   // as EigTask
    const void* fh0;           // [b][Sx] the round's transformed residual
    void* fh;                  // [b][Sx] the recursions of the round's summed inputs
    int b;
    int rin[4], rout[4];       // local rows at the cut above (0, 1) and below (2, 3), -1: none
};
struct CutNode {
    const void* C;             // basis [2 r][N]
    size_t N;
    int ra;
};
struct CutProb {
    int Sx, L, r, ncut, D, q1;
    int MG, ngrp, nA, XC, nch, nB;    // items of the phases (cut_plan)
    int cl, dist, res, nbi;           // cluster form; y shared out; panels in shared memory, items a block
    int max_iter, stall;              // stall: stop when the steps no longer contract
    double kh, test2, anchor2;        // squares of the test and anchor factors (of |b|, |r_0|)
    int mid[CUT_NCUT];                // grid row below each cut
    size_t cp_off[CUT_NCUT], ep_off[CUT_NCUT];
    unsigned short yidx[CUT_NCUT * 2 * CUT_MAXL];   // first y index of each E group of a cut
    const CutLeaf* leaf;
    const CutNode* node;
    const void *Cp, *Ep, *M;
    const void* rt;                   // [Sy][Sx] the round's residual
    void *v, *vsum, *res0;            // [ncut][2][Sx]
    void *prow, *pd, *d, *y, *yacc;   // [nA][4][Sx], [nB][(L + 1) r], [D] each
    float* npart;                     // [nB] partial |v|^2
    const double *nrm, *b2;           // |r|^2 and |b|^2 (FP64)
    const c128* scale;                // of the round's residual in k_cut_lines (null: 1)
    CutCtl* ctl;
};
// panel entries (one group of r basis columns at one cut row / cut)
struct CutCpEntry { const void* src; void* dst; size_t ldc; int K; };
struct CutEpEntry { const void* src; void* dst; c128* d64; size_t ldc; int Ke, maskl, maskr; };
struct CutGramPair { const void* cp; const void* ep; int K, Ke, rows, low; };   // low: products in the basis precision
struct CutGramDest { c128* out; int ld, first, count; };
struct CutMinv { int p, s; const c128* Ainv; };
struct CutUpdJob { const CutProb* prob; const c128* u; c128* ut; const void* w; int Sy; };
template <typename T>
void launch_cut_panels(const CutCpEntry* cp, int ncp, const CutEpEntry* ep, int nep, int Sx, int r, OpGeom g,
                       cudaStream_t s);
size_t cut_gram_scratch(int npairs);
// sums of C_p^H E_q per pair into the destinations (pairs [first, first + count) each, prs[0]
// being pair `first0`)
template <typename T>
void launch_cut_gram(const CutGramPair* prs, int npairs, int first0, const CutGramDest* ds, int ndest, int Sx, int r,
                     c128* part, cudaStream_t s);
// blocks of the inverse of the corrections' triangular system (children before parents);
// G, M and MT packed: a node's 2 r rows hold the corrections of its subtree level by level
// (cut_m_packed entries in all; full matrices took 16 D^2 bytes each, 260 MB at D = 4032 against
// 21).  cut_m_offset: the node's first entry; cut_m_len: entries of a row of a node of level l;
// cut_m_col: first column of node s at or below p.  MT: row-major or (tr) transposed within a
// node's rows
HH_HD int cut_level_of(int p) {
    int l = 0;
    while ((2 << l) <= p + 1) ++l;
    return l;
}
HH_HD int cut_m_len(int l, int L, int r) { return 2 * r * ((1 << (L - l)) - 1); }
HH_HD size_t cut_m_offset(int p, int L, int r) {
    const int l = cut_level_of(p);
    size_t o = 0;
    for (int q = 0; q < l; ++q) o += ((size_t)1 << q) * 2 * r * cut_m_len(q, L, r);
    return o + (size_t)(p + 1 - (1 << l)) * 2 * r * cut_m_len(l, L, r);
}
HH_HD int cut_m_col(int p, int s, int r) {
    const int l = cut_level_of(p), d = cut_level_of(s) - l;
    return 2 * r * ((1 << d) - 1 + (s + 1 - (1 << (l + d))) - ((p + 1 - (1 << l)) << d));
}
size_t cut_m_packed(int L, int r);
template <typename T>
void launch_cut_minv(const CutMinv* prs, int n, int L, int p2, const c128* G, c128* M, cplx<T>* MT, int tr,
                     cudaStream_t s);
// whether the cluster form can run with this much shared memory on the current device (true
// without one)
bool cut_cluster_ready(size_t smem);
// fills the items of P; returns the steps' shared memory, 0 if the lines do not fit; cluster:
// the cluster form may be taken
template <typename T>
size_t cut_plan(CutProb& P, int b_max, bool cluster);
// Flexible GMRES on the cut rows: its vectors and the least-squares problem.
struct CutGmres {
    c128 *V, *alpha;           // [mk + 1][nG], [mk + 1]
    c128 *v1, *rG, *w;         // [nG]: S r, r on the cut rows, the vector in work
    void* y0;                  // [D]: the corrections of the first step
    c128 *part, *dots, *scale; // [CUT_GM_BLOCKS][72], [2][72], [1]
    double* npart;             // [CUT_GM_BLOCKS]
    GmresLs ls;
    double red, tol;           // a cycle ends when the estimate is below red |r| or tol |b| / 2
};
constexpr int CUT_GM_BLOCKS = 152;
// runs every problem with a nonzero mode (1: new round, 2: go on) until its next stop, at most
// max_steps steps (0: no limit); gm_steps > 0: one problem's GMRES cycle of at most so many;
// group: blocks per problem of a grid group (cl: one cluster); bars: a word per group; false if it cannot be launched
template <typename T>
bool launch_cut_steps(const CutProb* probs, int nprob, int group, bool cl, size_t smem, const int* modes, int mode_all,
                      unsigned* bars, int max_groups, int* err, int prof, cudaStream_t s, int max_steps = 0,
                      const CutGmres* gm = nullptr, int gm_steps = 0);
template <typename T>
void launch_cut_lines(const CutProb* probs, int nprob, const int* modes, int nleaf_max, int b_max, int Sx_max,
                      cudaStream_t s);
// end of a GMRES cycle: the combined input and its scale of r (nG = 2 (2^L - 1) Sx entries)
template <typename T>
void launch_cut_gm_combine(const CutProb* prob, const CutGmres& G, int nG, cudaStream_t s);
template <typename T>
void launch_cut_update(const CutUpdJob* jobs, int njobs, int nleaf_max, int own_max, int Sx_max, cudaStream_t s);

// ---- the set-up's sub-level solves from the interface rows (k_edge.cu) ---------------
// A node on the path from a child's edge leaf up to the child: its basis, the child that
// holds the inner cut and lies on the edge's side.
struct EdgePath {
    int id, ra, kin, kedge;
    const void* C;
    size_t N, mo;                     // points; first entry of its rows of M
};
struct EdgeTask {
    const void *V, *xi, *sc;          // edge leaf, as EigTask
    int b, node;
    int a_if, a_sif, a_sin;           // its local rows: the interface, the sibling's trace rows
    int o0, o1;                       // its rows at the inner cut (-1: the child is a leaf)
    int g_if, g_sif, g_sin;           // the grid rows of the first three
    int below, lev, npath, K;         // the leaf lies below the cut; the child's level; path; panel width
    int sb;                           // rows of the sibling's band
    void *Om, *Z, *Vc;                // sketch / Y / Q, T^* Q, V_c
    void *rows, *vin, *pd, *Fh;       // [4][Sx][nc], [2][Sx][nc], partial products, [b][Sx][r]
    c128* y;                          // [npath][2r][nc]
    const void* cp;                   // the cut's basis panel
    c128 *Gm, *U;                     // Gram matrix, eigenvectors
    double* lam;
    const void* W;                    // the extension's first owned point [.][r]
    void* Cout;                       // its columns of the parent's basis [r][Np]
    size_t Np;
    long long dst0, npts;             // the child's points in the parent
    EdgePath path[CUT_MAXL];
};
template <typename T>
bool edge_rows_fit(int Sx);
size_t edge_pd_elems(int npath, int r, int nc);
size_t edge_gram_scratch(int nchild);
// the edge leaves' rows; then the path's corrections y of nc columns, added to the trace rows
// (adj: the interface row) when rows_out
template <typename T>
void launch_edge_rows(const EdgeTask* tasks, int nchild, int Sx, int nc, int adj, cudaStream_t s);
template <typename T>
void launch_edge_path(const EdgeTask* tasks, int nchild, int L, int Sx, int nc, int r, const c128* M, OpGeom g, int adj,
                      bool rows_out, cudaStream_t s);
// recursions of the basis extension (into Fh, transformed layout of nc right-hand sides)
template <typename T>
void launch_edge_basis_lines(const EdgeTask* tasks, int nchild, int b_max, int Sx, int nc, cudaStream_t s);
// the two rows at the inner cut of those (rows 0, 1)
template <typename T>
void launch_edge_leaf_rows(const EdgeTask* tasks, int nchild, int Sx, int nc, cudaStream_t s);
// Gm = Z^H Z in FP64; part: edge_gram_scratch bytes
template <typename T>
void launch_edge_gram(const EdgeTask* tasks, int nchild, int Sx, int m, c128* part, cudaStream_t s);
// the extensions into the parents' bases (the other child's rows zero)
template <typename T>
void launch_edge_scatter(const EdgeTask* tasks, int nchild, size_t np_max, int r, cudaStream_t s);
// launch_sketch, launch_robin_trace (rows 2, 3 -> Om), launch_adjoint_place (Om -> vin), the
// conjugate of row 2 into Z (k_field.cu) and launch_form_v (k_dense.cu), for all children
template <typename T>
void launch_edge_sketch(const EdgeTask* tasks, int nchild, int Sx, int m, unsigned long long seed, cudaStream_t s);
template <typename T>
void launch_edge_robin(const EdgeTask* tasks, int nchild, int Sx, int nc, double kh, int q1, cudaStream_t s);
template <typename T>
void launch_edge_place(const EdgeTask* tasks, int nchild, int Sx, int nc, double kh, int q1, cudaStream_t s);
template <typename T>
void launch_edge_conj(const EdgeTask* tasks, int nchild, int Sx, int nc, cudaStream_t s);
template <typename T>
void launch_edge_form_v(const EdgeTask* tasks, int nchild, int Sx, int m, int r, cudaStream_t s);

}  // namespace hh
