// k_cut.cu -- the stationary iteration on the rows next to the leaf cuts.
//
// One coarse-corrected ORAS step (Eqs. (2)-(3), n_i = 1) leaves a residual that vanishes off
// the two rows at each cut between neighbouring leaves: inside a leaf's owned rows the leaf
// solve satisfies A~ w = v exactly, and every basis column is extended from an artificial
// boundary outside the owned rows, so A~_p C_p is zero there as well.  For L levels that is
// 2 (2^L - 1) of S rows (14 of 1025 for eight leaves).  The iteration
//     u <- u + M r,  r <- r - A M r
// can therefore be run on those rows alone, and by linearity the iterate after K steps is
//     u_K = u_0 + M (r_0 + r_1 + ... + r_{K-1}),
// one application of M to the summed inputs.  Per step that leaves, for each leaf, the
// scalar recursions of its b modes with a right-hand side on at most four rows and four rows
// of the result, and for each node p the products of its basis with the residual on its
// cuts: instead of 2 passes over every basis (HBM) and two dense transforms per leaf.
// In exact arithmetic the iterates are those of the full iteration; the rows left out carry
// the leaf solves' rounding, which the FP64 residual at the end of each round brings back
// (the driver in hh_solver.cu starts a new round from it).
//
// Corrections of all levels at once: with t the composition of the leaf solutions and
// res0 = v - A t, d_p = C_p^H res0 and E_q = A C_q on the cut rows (C_q restricted to the
// rows q owns), the corrections y of Eq. (3) solve the block triangular system
//     A_p y_p + sum_{q below p} (C_p^H E_q) y_q = d_p,
// so y = M d with M its explicit inverse (k_cut_minv), and r <- res0 - sum_q E_q y_q.
#include <algorithm>
#include <atomic>

#include <cooperative_groups.h>

#include "k_line.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace hh {

// ---------------------------------------------------------------- tree arithmetic
// Cut c (0-based) lies between leaves c and c + 1; its node has level l and position t.
__device__ __forceinline__ int cut_level(int c, int L) { return L - __ffs(c + 1); }

// Barrier over the n co-resident blocks of a group (cooperative launch), bounded: the polls
// run out after `limit` (0: at once, the testing form), DEV_TIMEOUT is recorded and false
// returned.  A release-add on a counter that only grows and acquire loads of it: 1.2 us over
// 152 blocks (a counter that is reset and a generation word behind full fences: 2.2 us).
struct GroupBar {
    unsigned* ctr;
    unsigned n, target;
    int* err;
    long long limit;
    __device__ void arrive() {
        __syncthreads();
        target += n;
        if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
    }
    __device__ bool operator()() {
        arrive();
        return wait();
    }
    __device__ bool wait() {
        bool ok = true;
        if (threadIdx.x == 0) {
            ok = false;
            for (long long it = 0; it < limit && !ok; ++it) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
                ok = (int)(v - target) >= 0;
                if (it > 4096) __nanosleep(64);
            }
            if (!ok) atomicExch(err, DEV_TIMEOUT);
        }
        return __syncthreads_and(ok);
    }
};

__device__ __forceinline__ c64 ldcg(const c64* p) {
    const float2 v = __ldcg((const float2*)p);
    return {v.x, v.y};
}
__device__ __forceinline__ c128 ldcg(const c128* p) {
    const double2 v = __ldcg((const double2*)p);
    return {v.x, v.y};
}
// asynchronous copy of one element (the panels: written by earlier launches alone)
__device__ __forceinline__ void cp_async_el(c64* s, const c64* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_el(c128* s, const c128* g) { cp_async16(s, g); }
__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// The tests after a step: |v|^2 relative to the round's start, n2, against the thresholds,
// and (P.stall) whether the steps still contract: a residual a hundred times its smallest, or
// one that fell less than tenfold over the last 25 steps, stops the problem (its owner solves
// it by GMRES).
struct StepWatch {
    float best, chk;
    int chk_it;
    __device__ StepWatch(const CutCtl& c, double n0) {
        best = c.it ? (float)(c.best / n0) : 1.f;
        chk = c.it ? (float)(c.chk / n0) : 1.f;
        chk_it = c.chk_it;
    }
    __device__ int test(float n2, int it, const CutProb& P, float anchor, float due) {
        if (!isfinite(n2)) return CUT_NONFINITE;
        best = fminf(best, n2);
        bool slow = n2 > 1e4f * best;
        if (it - chk_it >= 25) {
            slow = slow || n2 > 0.01f * chk;
            chk = n2;
            chk_it = it;
        }
        if (P.stall && slow && n2 >= due) return CUT_STALL;
        if (n2 <= anchor) return CUT_ANCHOR;
        if (n2 < due) return CUT_TEST;
        return it >= P.max_iter ? CUT_LIMIT : 0;
    }
    __device__ void store(CutCtl& c, double n0) const {
        c.best = best * n0;
        c.chk = chk * n0;
        c.chk_it = chk_it;
    }
};

// ------------------------------------------------------------------- the cut rows
// Rows of the bases at the cuts.  Cp: [row 0/1][x][K] per cut, K = (level + 1) r: the r
// columns of each ancestor's child that holds the cut, then the own node's (row 0, above
// the cut, its first child's columns, row 1 its second child's).  One block per entry and
// 32 columns of the grid, transposed through shared memory.
template <typename T>
__global__ void __launch_bounds__(256) k_cut_cp(const CutCpEntry* __restrict__ ent, int Sx, int r) {
    using C = cplx<T>;
    __shared__ C tile[32][33];
    const CutCpEntry e = ent[blockIdx.y];
    const int x0 = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const C* src = (const C*)e.src;
    C* dst = (C*)e.dst;
    for (int j = ty; j < r; j += 8)
        if (x0 + tx < Sx) tile[j][tx] = src[(size_t)j * e.ldc + x0 + tx];
    __syncthreads();
    for (int x = ty; x < 32; x += 8)
        if (x0 + x < Sx && tx < r) dst[(size_t)(x0 + x) * e.K + tx] = tile[tx][x];
}

// E = A C on the cut rows, in FP64 products of the stored basis (e64, for the Galerkin
// sums) and rounded to the basis precision (the iteration): [row][column][x].  maskl/maskr:
// whether the rows above / below the cut belong to the rows the node owns.
template <typename T>
__global__ void __launch_bounds__(256) k_cut_ep(const CutEpEntry* __restrict__ ent, int Sx, int r, OpGeom g) {
    using C = cplx<T>;
    const CutEpEntry e = ent[blockIdx.y];
    const int x = blockIdx.x * 256 + threadIdx.x, j = blockIdx.z;
    if (x >= Sx || j >= r) return;
    const C* src = (const C*)e.src + (size_t)j * e.ldc;   // row mid - 2 of column j
    auto at = [&](int a, int xx) -> c128 {                // row mid - 2 + a
        const bool in = a < 2 ? e.maskl : e.maskr;
        return in && xx >= 0 && xx < Sx ? cvt<double>(src[(size_t)a * Sx + xx]) : c128{0, 0};
    };
#pragma unroll
    for (int row = 0; row < 2; ++row) {
        c128 s;
        const int a0 = 1 + row;
        if (g.q1) {
            s = q1_row<double>(1, x, g, [&](int dj, int di) { return at(a0 + dj, x + di); });
        } else {
            s = op_diag(1, x, g) * at(a0, x);
            s = s - at(a0, x - 1) - at(a0, x + 1) - wcol(x, Sx) * (at(a0 - 1, x) + at(a0 + 1, x));
        }
        const size_t o = ((size_t)row * e.Ke + j) * Sx + x;
        ((c128*)e.d64)[o] = s;
        ((C*)e.dst)[o] = cvt<T>(s);
    }
}

// Partial sums of C_p^H E_q over the cut rows of one (cut, group of p, group of q) pair and
// one share of the columns x: r x r FP64 products of the stored rows.  Two by two outputs
// per thread, tiles of 16 x staged in FP64.
static constexpr int GRAM_SPLIT = 8;
template <typename T>
__global__ void __launch_bounds__(256) k_cut_gram(const CutGramPair* __restrict__ prs, int Sx, int r, c128* part) {
    using C = cplx<T>;
    __shared__ c128 cs[16][33], es[16][33];
    const CutGramPair p = prs[blockIdx.x];
    const int ti = threadIdx.x >> 4, tj = threadIdx.x & 15;
    const int xs = (Sx + GRAM_SPLIT - 1) / GRAM_SPLIT;
    const int xa = blockIdx.y * xs, xb = min(Sx, xa + xs);
    c128 acc[2][2] = {{{0, 0}, {0, 0}}, {{0, 0}, {0, 0}}};
    if (p.low) {
        // blocks that only enter M, which is kept in the basis precision
        C* ct = (C*)&cs[0][0];
        C* et = (C*)&es[0][0];
        C lc[2][2] = {{{0, 0}, {0, 0}}, {{0, 0}, {0, 0}}};
        for (int row = 0; row < 2; ++row) {
            if (!((p.rows >> row) & 1)) continue;
            const C* cp = (const C*)p.cp + (size_t)row * Sx * p.K;
            const C* ep = (const C*)p.ep + (size_t)row * p.Ke * Sx;
            for (int x0 = xa; x0 < xb; x0 += 16) {
                for (int t = threadIdx.x; t < 16 * 32; t += 256) {
                    const int x = t >> 5, j = t & 31, x2 = t & 15, j2 = t >> 4;
                    ct[x * 33 + j] = x0 + x < xb && j < r ? cp[(size_t)(x0 + x) * p.K + j] : C{0, 0};
                    et[x2 * 33 + j2] = x0 + x2 < xb && j2 < r ? ep[(size_t)j2 * Sx + x0 + x2] : C{0, 0};
                }
                __syncthreads();
#pragma unroll 4
                for (int x = 0; x < 16; ++x) {
                    const C a0 = ct[x * 33 + ti], a1 = ct[x * 33 + ti + 16], b0 = et[x * 33 + tj],
                            b1 = et[x * 33 + tj + 16];
                    cfma_cj(lc[0][0], a0, b0);
                    cfma_cj(lc[0][1], a0, b1);
                    cfma_cj(lc[1][0], a1, b0);
                    cfma_cj(lc[1][1], a1, b1);
                }
                __syncthreads();
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 2; ++v) acc[u][v] = cvt<double>(lc[u][v]);
    } else
    for (int row = 0; row < 2; ++row) {
        if (!((p.rows >> row) & 1)) continue;
        const C* cp = (const C*)p.cp + (size_t)row * Sx * p.K;
        const c128* ep = (const c128*)p.ep + (size_t)row * p.Ke * Sx;
        for (int x0 = xa; x0 < xb; x0 += 16) {
            for (int t = threadIdx.x; t < 16 * 32; t += 256) {
                const int x = t >> 5, j = t & 31, x2 = t & 15, j2 = t >> 4;
                cs[x][j] = x0 + x < xb && j < r ? cvt<double>(cp[(size_t)(x0 + x) * p.K + j]) : c128{0, 0};
                es[x2][j2] = x0 + x2 < xb && j2 < r ? ep[(size_t)j2 * Sx + x0 + x2] : c128{0, 0};
            }
            __syncthreads();
#pragma unroll 4
            for (int x = 0; x < 16; ++x) {
                const c128 a0 = cs[x][ti], a1 = cs[x][ti + 16], b0 = es[x][tj], b1 = es[x][tj + 16];
                cfma_cj(acc[0][0], a0, b0);
                cfma_cj(acc[0][1], a0, b1);
                cfma_cj(acc[1][0], a1, b0);
                cfma_cj(acc[1][1], a1, b1);
            }
            __syncthreads();
        }
    }
    c128* o = part + ((size_t)blockIdx.x * GRAM_SPLIT + blockIdx.y) * 1024;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) o[(ti + 16 * u) * 32 + tj + 16 * v] = acc[u][v];
}
__global__ void __launch_bounds__(256) k_cut_gram_red(const CutGramDest* __restrict__ ds, int first0, int r,
                                                      const c128* part) {
    const CutGramDest d = ds[blockIdx.x];
    for (int t = threadIdx.x; t < r * r; t += 256) {
        const int i = t / r, j = t - i * r;
        c128 s = {0, 0};
        for (int k = (d.first - first0) * GRAM_SPLIT; k < (d.first - first0 + d.count) * GRAM_SPLIT; ++k)
            s = s + part[(size_t)k * 1024 + i * 32 + j];
        d.out[(size_t)i * d.ld + j] = s;
    }
}

// Row e of the packed M (node p of level l at position t): its offset and its length, the
// corrections of p's subtree level by level.
__device__ __forceinline__ int cut_m_row(int e, int L, int r, int& l, int& t) {
    const int p2 = 2 * r, p = e / p2;
    l = 31 - __clz(p + 1);
    t = p + 1 - (1 << l);
    int o = 0;
    for (int q = 0; q < l; ++q) o += (1 << q) * p2 * p2 * ((1 << (L - q)) - 1);
    const int len = p2 * ((1 << (L - l)) - 1);
    return o + (t * p2 + (e - p * p2)) * len;
}

// M_ps for one pair (p, s below or equal p): Ainv_p if s = p, else
// -Ainv_p sum_{s <= q < p} G_pq M_qs, FP64.  A block takes MINV_ROWS rows: (Ainv_p G_pq) of
// those rows in shared memory, then its product with M_qs (bound by the latency of the FP64
// chains; a set-up of 1023^2 at 2r = 64 took 1.4 ms longer with one block a pair).
static constexpr int MINV_ROWS = 4;
template <typename T>
__global__ void __launch_bounds__(256) k_cut_minv(const CutMinv* __restrict__ prs, int L, int p2,
                                                  const c128* __restrict__ G, c128* M, cplx<T>* MT, int tr) {
    __shared__ c128 ai[MINV_ROWS][64], xs[MINV_ROWS][64];
    const CutMinv e = prs[blockIdx.x];
    const int i0 = blockIdx.y * MINV_ROWS, ni = min(MINV_ROWS, p2 - i0);
    if (ni <= 0) return;
    // all packed by subtree; this pair's first entry in p's rows
    const int r = p2 / 2, len = cut_m_len(cut_level_of(e.p), L, r), k0 = cut_m_col(e.p, e.s, r);
    const size_t op = cut_m_offset(e.p, L, r);
    cplx<T>* mt = MT + op;
    // (tr: the cluster form's order, transposed within the node's rows)
    auto put = [&](int i, int j, c128 v) {
        M[op + (size_t)i * len + k0 + j] = v;
        mt[tr ? (size_t)(k0 + j) * p2 + i : (size_t)i * len + k0 + j] = cvt<T>(v);
    };
    for (int q = threadIdx.x; q < ni * p2; q += 256) {
        const int i = q / p2, j = q - i * p2;
        ai[i][j] = e.Ainv[(size_t)(i0 + i) * p2 + j];
        if (e.p == e.s) put(i0 + i, j, ai[i][j]);
    }
    if (e.p == e.s) return;
    const int i = threadIdx.x >> 6, j = threadIdx.x & 63;
    const bool on = i < ni && j < p2;
    c128 acc = {0, 0};
    for (int q = e.s; q != e.p; q = (q - 1) >> 1) {   // s and its ancestors below p
        const int lenq = cut_m_len(cut_level_of(q), L, r);
        const c128* gq = G + op + cut_m_col(e.p, q, r) + j;
        const c128* mq = M + cut_m_offset(q, L, r) + cut_m_col(q, e.s, r) + j;
        __syncthreads();
        c128 h = {0, 0};
        if (on)
#pragma unroll 8
            for (int k = 0; k < p2; ++k) cfma(h, ai[i][k], gq[(size_t)k * len]);
        if (on) xs[i][j] = h;
        __syncthreads();
        if (on)
#pragma unroll 8
            for (int k = 0; k < p2; ++k) cfma(acc, xs[i][k], mq[(size_t)k * lenq]);
    }
    if (on) put(i0 + i, j, -acc);
}

// ----------------------------------------------------------------- GMRES on the cut rows
// Flexible GMRES's Krylov space from a residual r is spanned by r and vectors on the cut
// rows: A M v = v - S v with S v (one step's residual) on the cut rows for any v.  A basis
// vector is kept as (alpha, p): alpha times r off the cut rows and p on them, in FP64, with
// the inner product conj(alpha) alpha' rho^2 + p^H p', rho = |r| off the cut rows, so the
// Arnoldi process is that of the full vectors at 2 (2^L - 1) / S of their length.
// S (alpha r + g) = alpha v1 + S g, v1 = S r from the cycle's first step and g = p - alpha
// r_G on the cut rows, so every further step is one step of the iteration on g.
//
// One Arnoldi step inside the iteration's kernels, after phase C has left S g (the first
// time S r) in P.v: w = V_j - S V_j, classical Gram-Schmidt twice against V_0 .. V_j, V_{j+1}
// and the next g (into P.v), and in the first block the Givens update.  A block works on the
// entries of its own cut item, so only the dot products cross blocks: partial sums, one
// column a warp adds them, four barriers.  The second pass's products include |w|^2, which
// gives |V_{j+1}| before its correction: |w - V h|^2 = |w|^2 - |h|^2.  After the first pass |h|^2 is
// rounding (at most 1e-28 |w|^2 over 63^2 to 127^2, both schemes, one to three levels), so nothing
// cancels: against extended precision this norm is off by at most 3.4e-16, the norm of the corrected
// vector by 1.0e-15.
// What bounds it is the FP64 issue rate (a warp's multiply-add takes its scheduler 64 clocks)
// and the loads' latency: threads share out a column's entries in the products and an
// entry's columns in the updates, loads go four deep, scalars are left to one warp, and the
// Givens chain keeps only its own multiply-adds.  At 500^2 (148 blocks, 48 entries each,
// 36 columns) a step takes 26 us and the Givens update 9; with one thread an entry, w in the
// L2 and five barriers a solve took 13.7 ms instead of 12.6.
struct GmState {
    c128 h[72], al[72], hc[72], sn[72], b[72], a[72];
    double cs[72], red[32], rho2, inv, nn, beta;
    c128 an;
};
__device__ __forceinline__ double gm_block_sum(double x, double* red, int nw) {
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    double t = 0.0;
    for (int k = 0; k < nw; ++k) t += red[k];
    __syncthreads();
    return t;
}
// Sum of a over groups of W lanes: the first exchange leaves the real part's sums in the group's
// lower half and the imaginary part's in the upper, so the rest adds one number a lane.
template <int W> __device__ __forceinline__ c128 gm_sum(c128 a) {
    const bool up = threadIdx.x & (W / 2);
    const double give = up ? a.re : a.im;
    double k = (up ? a.im : a.re) + __shfl_xor_sync(0xffffffffu, give, W / 2);
#pragma unroll
    for (int o = W / 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    const double x = __shfl_xor_sync(0xffffffffu, k, W / 2);
    return up ? c128{x, k} : c128{k, x};
}
template <typename P> __device__ __forceinline__ c128* align16(P* p) { return (c128*)(((size_t)p + 15) & ~(size_t)15); }
// scr: shared memory for cap complex numbers, free here.
template <typename T, int NT>
__device__ __noinline__ bool gm_arnoldi(const CutProb& P, const CutGmres& G, GmState& M, GroupBar& bar, int rank, int gsz,
                                        int j, c128* scr, int cap) {
    using C = cplx<T>;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, Sx = P.Sx, nc = j + 1;
    const size_t nG = (size_t)2 * P.ncut * Sx;
    C* v = (C*)P.v;
    // one item a block: w stays in shared memory (else in G.w), and np * kg threads share
    // the update, partial sums behind w
    const int xw = min(P.XC, Sx - (rank % P.nch) * P.XC);
    const bool one = P.nB <= gsz && 2 * P.XC <= cap;
    int kg = 1;
    if (one && rank < P.nB) kg = max(1, min(min(8, NT / (2 * xw)), cap / (2 * P.XC) - 1));
    c128* part = scr + 2 * P.XC;
    // this block's items: f(entries, first column, columns, cut)
    auto items = [&](auto&& f) {
        for (int e = rank; e < P.nB; e += gsz) {
            const int c = e / P.nch, x0 = (e - c * P.nch) * P.XC;
            f(c, x0, min(P.XC, Sx - x0));
        }
    };
    auto entries = [&](auto&& f) {       // f(place in w, entry)
        items([&](int c, int x0, int xn) {
            for (int q = tid; q < 2 * xn; q += NT) {
                const size_t o = (size_t)(2 * c + (q >= xn)) * Sx + x0 + (q >= xn ? q - xn : q);
                f(one ? scr + q : G.w + o, o);
            }
        });
    };
    __syncthreads();
    if (j == 0) {
        const double beta = sqrt(*P.nrm), inv = beta > 0.0 ? 1.0 / beta : 0.0;
        double g2 = 0.0;
        entries([&](c128*, size_t o) {
            const int c = (int)(o / (2 * (size_t)Sx));
            const c128 r = cvt<double>(((const C*)P.rt)[(size_t)(P.mid[c] - 1) * Sx + (o - (size_t)2 * c * Sx)]);
            G.rG[o] = r;
            G.v1[o] = cvt<double>(v[o]);
            G.V[o] = inv * r;
            g2 += abs2(r);
        });
        g2 = gm_block_sum(g2, M.red, NW);
        if (tid == 0) {
            G.npart[rank] = g2;
            M.al[0] = c128{inv, 0.0};
            M.beta = beta;
            if (rank == 0) {
                G.alpha[0] = M.al[0];
                G.ls.g[0] = c128{beta, 0.0};
            }
        }
        if (!bar()) return false;
        double t = 0.0;
        for (int k = tid; k < gsz; k += NT) t += __ldcg(G.npart + k);
        t = gm_block_sum(t, M.red, NW);
        if (tid == 0) M.rho2 = fmax(0.0, *P.nrm - t);
        __syncthreads();
    }
    const double rho2 = M.rho2;
    c128 aw = M.al[j];                           // alpha of w: V_j's, as S V_j lies on the cut rows
    entries([&](c128* w, size_t o) {
        c128 sv = aw * G.v1[o];
        if (j > 0) sv = sv + cvt<double>(v[o]);
        *w = G.V[(size_t)j * nG + o] - sv;
    });
    for (int i = tid; i < nc; i += NT) M.hc[i] = {0, 0};
    __syncthreads();
    for (int pass = 0; pass < 2; ++pass) {
        // the products: tpc threads a column; in the second pass column nc is w itself
        const int ncp = nc + pass;
        int tpc = 32;
        while (tpc > 8 && NT / tpc < ncp) tpc >>= 1;
        const int sub = tid & (tpc - 1);
        for (int i0 = 0; i0 < ncp; i0 += NT / tpc) {
            const int i = i0 + tid / tpc;
            c128 a = {0, 0};
            if (i < ncp)
                items([&](int c, int x0, int xn) {
                    const size_t o0 = (size_t)2 * c * Sx + x0;
                    const c128* w = one ? scr : G.w + o0;
                    const c128* Vi = i < nc ? G.V + (size_t)i * nG + o0 : w;
                    const int gap = Sx - xn, wgap = one ? 0 : gap, vgap = i < nc ? gap : wgap;   // between the rows
                    for (int q0 = sub; q0 < 2 * xn; q0 += 4 * tpc) {
                        c128 x[4], y[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int q = q0 + u * tpc;
                            x[u] = y[u] = c128{0, 0};
                            if (q < 2 * xn) {
                                x[u] = Vi[q + (q >= xn ? vgap : 0)];
                                y[u] = w[q + (q >= xn ? wgap : 0)];
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (q0 + u * tpc < 2 * xn) cfma_cj(a, x[u], y[u]);
                    }
                });
            a = tpc == 32 ? gm_sum<32>(a) : tpc == 16 ? gm_sum<16>(a) : gm_sum<8>(a);
            if (i < ncp && sub == 0) G.part[(size_t)rank * 72 + i] = a;
        }
        if (!bar()) return false;
        for (int i = rank + gsz * warp; i < ncp; i += gsz * NW) {
            c128 a = {0, 0};
#pragma unroll 5
            for (int k = lane; k < gsz; k += 32) a = a + ldcg(G.part + (size_t)k * 72 + i);
            a = gm_sum<32>(a);
            if (lane == 0) G.dots[pass * 72 + i] = a + rho2 * (conj(i < nc ? M.al[i] : aw) * aw);
        }
        if (!bar()) return false;
        for (int i = tid; i < ncp; i += NT) M.h[i] = ldcg(G.dots + pass * 72 + i);
        __syncthreads();
        // the last warp: alpha of the new w, and after the second pass its norm
        if (warp == NW - 1) {
            c128 da = {0, 0};
            double hh = 0.0;
            for (int i = lane; i < nc; i += 32) {
                const c128 h = M.h[i];
                cfma(da, h, M.al[i]);
                M.hc[i] = M.hc[i] + h;
                if (pass) hh += abs2(h);
            }
            da = aw - gm_sum<32>(da);
            if (lane == 0) M.an = da;
            if (pass) {
                const double nn = fmax(0.0, M.h[nc].re - warp_sum(hh)), inv = nn > 0.0 ? rsqrt(nn) : 0.0;
                if (lane == 0) {
                    M.nn = nn;
                    M.inv = inv;
                }
            }
        }
        // w -= V h; after the second pass V_{j+1} and the next step's input
        items([&](int c, int x0, int xn) {
            const size_t o0 = (size_t)2 * c * Sx + x0;
            const int np = 2 * xn;
            for (int t = tid; t < np * kg; t += NT) {
                const int kk = t / np, q = t - kk * np;
                const c128* Vo = G.V + o0 + q + (q >= xn ? Sx - xn : 0);
                c128 a0 = {0, 0}, a1 = {0, 0};
                for (int i = kk; i < nc; i += 4 * kg) {
                    c128 x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) x[u] = i + u * kg < nc ? Vo[(size_t)(i + u * kg) * nG] : c128{0, 0};
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i + u * kg < nc) cfma(u & 1 ? a1 : a0, M.h[i + u * kg], x[u]);
                }
                c128* w = one ? scr + q : G.w + (Vo - G.V);
                if (kg > 1) part[kk * np + q] = a0 + a1;
                else *w = *w - (a0 + a1);
            }
        });
        __syncthreads();
        aw = M.an;
        const double inv = M.inv;
        const c128 an = inv * aw;
        if (pass || kg > 1)
            entries([&](c128* w, size_t o) {
                c128 x = *w;
                if (kg > 1)
                    for (int kk = 0; kk < kg; ++kk) x = x - part[kk * 2 * xw + (w - scr)];
                if (!pass) {
                    *w = x;
                    return;
                }
                x = inv * x;
                G.V[(size_t)(j + 1) * nG + o] = x;
                v[o] = cvt<T>(x - an * G.rG[o]);
            });
        if (pass && tid == 0) M.al[j + 1] = an;
        __syncthreads();
    }
    if (rank != 0 || warp != 0) return true;
    // The Givens update of column j (k_gmres_rotate's): with a_0 = h_0, a_{i+1} = cs_i h_{i+1} -
    // conj(sn_i) a_i and R_i = cs_i a_i + sn_i h_{i+1}; the chain of the a alone is serial.
    const GmresLs& ls = G.ls;
    for (int i = lane; i < j; i += 32) M.b[i] = M.cs[i] * M.hc[i + 1];
    __syncwarp();
    if (lane == 0) {
        c128 a = M.hc[0];
#pragma unroll 4
        for (int i = 0; i < j; ++i) {
            const c128 sn = M.sn[i], b = M.b[i];
            M.a[i] = a;
            a = c128{fma(-sn.im, a.im, fma(-sn.re, a.re, b.re)), fma(sn.im, a.re, fma(-sn.re, a.im, b.im))};
        }
        M.a[j] = a;
    }
    __syncwarp();
    for (int i = lane; i < j; i += 32) ls.H[(size_t)i * ls.mk + j] = M.cs[i] * M.a[i] + M.sn[i] * M.hc[i + 1];
    // the square roots and the quotients side by side in the lanes (each takes over a
    // thousand clocks): |a|, t, |V_{j+1}|, |b|, then 1 / |a|, |a| / t, |V_{j+1}| / t
    c128 a = M.a[j];
    const double nn = M.nn, a2 = abs2(a);
    const double root = sqrt(lane == 0 ? a2 : lane == 1 ? a2 + nn : lane == 2 ? nn : *P.b2);
    const double aa = __shfl_sync(0xffffffffu, root, 0), t = __shfl_sync(0xffffffffu, root, 1),
                 hn = __shfl_sync(0xffffffffu, root, 2), nbv = __shfl_sync(0xffffffffu, root, 3);
    const double quo = (lane == 0 ? 1.0 : lane == 1 ? aa : hn) / (lane == 0 ? aa : t);
    const double ia = __shfl_sync(0xffffffffu, quo, 0), at = __shfl_sync(0xffffffffu, quo, 1),
                 ht = __shfl_sync(0xffffffffu, quo, 2);
    if (lane != 0) return true;
    G.alpha[j + 1] = M.al[j + 1];
    double cs = 1.0;
    c128 sn = {0.0, 0.0};
    if (t != 0.0 && aa == 0.0) {
        cs = 0.0;
        sn = {1.0, 0.0};
        a = {hn, 0.0};
    } else if (t != 0.0) {
        const c128 ph = ia * a;
        cs = at;
        sn = ht * ph;
        a = t * ph;
    }
    ls.H[(size_t)j * ls.mk + j] = a;
    M.cs[j] = cs;
    M.sn[j] = sn;
    const c128 gj = ls.g[j], gn = -(conj(sn) * gj);
    ls.g[j + 1] = gn;
    ls.g[j] = cs * gj;
    GmresState* st = ls.st;
    st->steps = j + 1;
    const double beta = M.beta, gabs = sqrt(abs2(gn)), est = nbv > 0 ? gabs / nbv : 0.0;
    st->est = est;
    if (!isfinite(est)) {
        st->bad = 1;
        st->stop = 1;
        st->jstop = j + 1;
    } else if (est < 0.5 * G.tol || gabs < G.red * beta || hn == 0.0) {
        st->stop = 1;
        st->jstop = j + 1;
    }
    return true;
}

// ------------------------------------------------------------------- the iteration
// Shared memory of a step block, in elements: the xi lines and their lane products, the
// lines of one item, the input rows; M where every block forms y itself; the panels of the
// block's items where they fit (res); and the small arrays of phases B, Y and C.
struct CutSmem {
    int xi, ln, v, m, ce, t, rs, red, d, y, ya, up, own, total;
};
HH_HD int cut_m_elems(int L, int r) {
    int n = 0;
    for (int l = 0; l < L; ++l) n += (1 << l) * (2 * r) * (2 * r) * ((1 << (L - l)) - 1);
    return n;
}
HH_HD CutSmem cut_smem_layout(const CutProb& P, int nw) {
    CutSmem s;
    const int kmax = P.L * P.r;
    int o = 0;
    s.xi = o; o += P.MG * P.Sx;
    s.ln = o; o += P.MG * P.Sx;
    s.v = o; o += 4 * P.Sx;
    s.m = o; o += P.dist ? 0 : cut_m_elems(P.L, P.r);
    s.ce = o; o += P.res ? P.nbi * 2 * P.XC * (3 * P.L) * P.r : 0;
    s.t = o; o += 4 * (P.XC + 2);
    s.rs = o; o += 2 * P.XC;
    s.red = o; o += nw * 2 * kmax;
    s.d = o; o += P.D;
    s.y = o; o += P.D;
    s.ya = o; o += P.D;
    s.up = o; o += CUT_KG * 2 * P.XC;
    s.own = o; o += 4 * P.XC;
    s.total = o;
    return s;
}

// One group of co-resident blocks per problem runs its steps until the next test,
// anchor or limit; a launch's groups take the problems in turn.  The work is cut into
// items that depend on the problem alone, so the group's size changes no sum.
//   A: item (leaf, MG modes), one warp per mode: f^ = sum of at most four rows (the first
//      step of a round: the transformed full residual), both recursions, and the item's
//      share of the four rows of the result;
//   B: item (cut, XC columns): the rows' sums over the items, res0 = v - A t, and its
//      products with the basis rows of the cut's ancestors;
//   Y: d and y = M d, in every block, or (dist) one entry per warp and a barrier each;
//   C: the items of B again: v = res0 - sum E y, and its norm.
// What bounds it is latency: a barrier and a first load from the L2 per phase.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_cut_steps(const CutProb* __restrict__ probs, int nprob, int gsz,
                                                  const int* modes, int mode_all, unsigned* bars, int* err,
                                                  long long limit, int prof, int max_steps, CutGmres G, int gm_steps) {
    using C = cplx<T>;
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char csm[];
    __shared__ __align__(32) C s_vin[CUT_MGMAX][4], s_vout[CUT_MGMAX][4], s_sc[CUT_MGMAX];
    __shared__ float s_red[NW];
    // the descriptors in shared memory: the barriers' acquires drop the L1, so that every
    // phase would fetch them from the L2 again, one dependent load after another
    __shared__ CutProb P;
    __shared__ CutLeaf F;
    __shared__ GmState s_gm;
    const int ngroups = gridDim.x / gsz, group = blockIdx.x / gsz, rank = blockIdx.x - group * gsz;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    GroupBar bar{bars + group, (unsigned)gsz, 0u, err, limit};
    bool ok = true;
    // (before any wait: k_cut_gm_combine takes the number of columns from it, also of a cycle
    // whose first wait gave up)
    if (gm_steps && rank == 0 && tid == 0) *G.ls.st = GmresState{0, 0, 0, 0, 0.0, 0.0};
    for (int pi = group; ok && pi < nprob; pi += ngroups) {
        const int mode = modes ? modes[pi] : mode_all;
        if (!mode) continue;
        __syncthreads();   // the previous problem's arrays are no longer read
        for (int q = tid; q < (int)(sizeof(CutProb) / 4); q += NT) ((int*)&P)[q] = ((const int*)(probs + pi))[q];
        __syncthreads();
        const int Sx = P.Sx, r = P.r, L = P.L, nch = P.nch, XC = P.XC, D = P.D, MG = P.MG;
        const int kmax = L * r;
        const bool dist = P.dist, res = P.res && P.nB <= P.nbi * gsz;
        const bool one = P.nB <= gsz;   // at most one item of phases B and C a block: its rows stay here
        CutCtl* ctl = P.ctl;
        const CutSmem lay = cut_smem_layout(P, NW);
        C* const sm = (C*)csm;
        C* s_xi = sm + lay.xi;
        C* s_ln = sm + lay.ln;
        C* s_v = sm + lay.v;
        C* s_m = sm + lay.m;
        C* s_ce = sm + lay.ce;
        C* s_t = sm + lay.t;
        C* s_rs = sm + lay.rs;
        C* s_pd = sm + lay.red;
        C* s_d = sm + lay.d;
        C* s_y = sm + lay.y;
        C* s_up = sm + lay.up;
        C* s_own = sm + lay.own;
        C* s_vs = s_own + 2 * XC;
        C* s_ya = sm + lay.ya;
        C* v = (C*)P.v;
        C* vsum = (C*)P.vsum;
        C* res0 = (C*)P.res0;
        C* prow = (C*)P.prow;
        C* pd = (C*)P.pd;
        C* gd = (C*)P.d;
        C* gy = (C*)P.y;
        C* yacc = (C*)P.yacc;
        const C* Mt = (const C*)P.M;
        OpGeom g;
        g.b = 3;
        g.Sx = Sx;
        g.kh = P.kh;
        g.khr = nullptr;
        g.q1 = P.q1;
        // thresholds of this launch (the FP64 norms of the round's start)
        bool first = mode == 1;
        const double b2 = *P.b2, n0 = first ? *P.nrm : ctl->n0;
        // |v|^2 relative to the round's start, in single precision (an FP64 chain costs more
        // than a phase; the value only decides when the FP64 residual is formed)
        const float thr_test = (float)(P.test2 * b2 / n0), thr_anchor = (float)P.anchor2;
        const T inv0 = (T)(1.0 / sqrt(n0));
        int it = ctl->it, in_round = first ? 0 : ctl->in_round, reason = 0;
        StepWatch watch(*ctl, n0);
        int done = 0;
        float n2 = 0.f;
        int xi_item = -1;
        LineScan<T> scan;
        bool stepped = false;   // a step of this launch is done
        unsigned long long t0 = 0, tA = 0, tB = 0, tC = 0;
        const bool timing = prof && rank == 0 && tid == 0;
        if (!dist)
            for (int q = tid; q < cut_m_elems(L, r); q += NT) s_m[q] = Mt[q];
        // the panels of the block's items: C as [row][x][K], then E as [row][k][x]
        if (res) {
            for (int q = 0, e = rank; e < P.nB; ++q, e += gsz) {
                const int c = e / nch, x0 = (e - c * nch) * XC, xn = min(XC, Sx - x0);
                const int lev = cut_level(c, L), K = (lev + 1) * r, Ke = (2 * L - lev) * r;
                C* dc = s_ce + (size_t)q * 2 * XC * 3 * L * r;
                C* de = dc + 2 * XC * K;
                for (int row = 0; row < 2; ++row) {
                    const C* sc = (const C*)P.Cp + P.cp_off[c] + ((size_t)row * Sx + x0) * K;
                    for (int u = tid; u < xn * K; u += NT) dc[row * XC * K + u] = sc[u];
                    const C* se = (const C*)P.Ep + P.ep_off[c] + (size_t)row * Ke * Sx + x0;
                    for (int u = tid; u < Ke * xn; u += NT) {
                        const int k = u / xn, x = u - k * xn;
                        de[(row * Ke + k) * XC + x] = se[(size_t)k * Sx + x];
                    }
                }
            }
        }
        for (;;) {
            if (timing) t0 = gtime();
            // ------------------------------------------------------------------ A
            for (int a = rank; a < P.nA; a += gsz) {
                const int lf = a / P.ngrp, m0 = (a - lf * P.ngrp) * MG;
                if (xi_item != a) {
                    __syncthreads();
                    if (tid < (int)(sizeof(CutLeaf) / 4)) ((int*)&F)[tid] = ((const int*)(P.leaf + lf))[tid];
                }
                __syncthreads();
                const int b = F.b, nm = min(MG, b - m0);
                if (xi_item != a && nm > 0) {
                    const C* V = (const C*)F.V;
                    for (int q = tid; q < 4 * nm; q += NT) {
                        const int k = q / nm, w = q - k * nm;
                        const C sc = F.sc ? ((const C*)F.sc)[m0 + w] : C{1, 0};
                        s_vout[w][k] = F.rout[k] >= 0 ? V[(size_t)F.rout[k] * b + m0 + w] : C{0, 0};
                        const C vi = F.rin[k] >= 0 ? V[(size_t)F.rin[k] * b + m0 + w] : C{0, 0};
                        s_vin[w][k] = F.sc ? sc * vi : vi;
                        if (k == 0) s_sc[w] = sc;
                    }
                    if (warp < nm) {   // at most one mode a warp
                        const C* xi = (const C*)F.xi + (size_t)(m0 + warp) * Sx;
                        for (int i = lane; i < Sx; i += 32) s_xi[warp * Sx + i] = xi[i];
                        __syncwarp();
                        line_scan_init(s_xi + warp * Sx, Sx, lane, scan);
                    }
                }
                xi_item = a;
                if (nm <= 0) continue;
                if (!first) {
                    const C* src = v + (size_t)(lf - 1) * 2 * Sx;   // the cut above, then the cut below
                    const bool up = F.rin[0] >= 0, dn = F.rin[2] >= 0;
#pragma unroll 2
                    for (int i = tid; i < Sx; i += NT) {
                        const C a0 = up ? ldcg(src + i) : C{0, 0}, a1 = up ? ldcg(src + Sx + i) : C{0, 0};
                        const C a2 = dn ? ldcg(src + 2 * Sx + i) : C{0, 0}, a3 = dn ? ldcg(src + 3 * Sx + i) : C{0, 0};
                        s_v[i] = a0;
                        s_v[Sx + i] = a1;
                        s_v[2 * Sx + i] = a2;
                        s_v[3 * Sx + i] = a3;
                    }
                }
                __syncthreads();
                // the lines' right-hand sides, then the recursions, one warp a line
                if (first) {
                    for (int w = warp; w < nm; w += NW) {
                        const C* f0 = (const C*)F.fh0 + (size_t)(m0 + w) * Sx;
                        const C sc = s_sc[w];
                        for (int i = lane; i < Sx; i += 32) s_ln[w * Sx + i] = F.sc ? sc * f0[i] : f0[i];
                    }
                } else {
                    for (int i = tid; i < Sx; i += NT) {
                        const C v0 = s_v[i], v1 = s_v[Sx + i], v2 = s_v[2 * Sx + i], v3 = s_v[3 * Sx + i];
                        for (int w = 0; w < nm; ++w) {
                            const cpair<T> p0 = *(const cpair<T>*)&s_vin[w][0], p1 = *(const cpair<T>*)&s_vin[w][2];
                            C f = p0.x * v0;
                            cfma(f, p0.y, v1);
                            cfma(f, p1.x, v2);
                            cfma(f, p1.y, v3);
                            s_ln[w * Sx + i] = f;
                        }
                    }
                }
                __syncthreads();
                if (warp < nm) line_solve(s_xi + warp * Sx, s_ln + warp * Sx, Sx, lane, scan);
                __syncthreads();
                for (int i = tid; i < Sx; i += NT) {
                    C o[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
                    for (int w = 0; w < nm; ++w) {
                        const C f = s_ln[w * Sx + i];
                        const cpair<T> p0 = *(const cpair<T>*)&s_vout[w][0], p1 = *(const cpair<T>*)&s_vout[w][2];
                        cfma(o[0], p0.x, f);
                        cfma(o[1], p0.y, f);
                        cfma(o[2], p1.x, f);
                        cfma(o[3], p1.y, f);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (F.rout[k] >= 0) prow[((size_t)a * 4 + k) * Sx + i] = o[k];
                }
            }
            bar.arrive();
            // while the others arrive: the item's basis panel into the lines' place
            const bool stage = !res && one && rank < P.nB;
            const int sc_ = stage ? rank / nch : 0, sx0 = (rank - sc_ * nch) * XC, sxn = stage ? min(XC, Sx - sx0) : 0;
            const int slev = cut_level(sc_, L), sK = (slev + 1) * r, sKe = (2 * L - slev) * r;
            const int room = (MG + 4) * Sx;
            const bool stage_c = stage && 2 * XC * sK <= room;
            const int kfit = stage ? min(sKe, room / (2 * XC)) : 0;
            if (stage_c) {
                const C* src = (const C*)P.Cp + P.cp_off[sc_] + (size_t)sx0 * sK;
                for (int q = tid; q < sxn * sK; q += NT) {
                    cp_async_el(s_ln + q, src + q);
                    cp_async_el(s_ln + XC * sK + q, src + (size_t)Sx * sK + q);
                }
                cp_async_commit();
            }
            if (!(ok = bar.wait())) break;
            if (timing) { const unsigned long long t = gtime(); tA += t - t0; t0 = t; }
            // ------------------------------------------------------------------ B
            for (int e = rank, q0 = 0; e < P.nB; e += gsz, ++q0) {
                const int c = e / nch, x0 = (e - c * nch) * XC, xn = min(XC, Sx - x0);
                const int lev = cut_level(c, L), K = (lev + 1) * r;
                // the four rows next to the cut, halo of one column
                for (int q = tid; q < 4 * (xn + 2); q += NT) {
                    const int row = q / (xn + 2), il = q - row * (xn + 2), i = x0 - 1 + il;
                    C s = {0, 0};
                    if (i >= 0 && i < Sx) {
                        const int lf = c + (row >> 1), k = row < 2 ? row + 2 : row - 2;
                        const int ng = (P.leaf[lf].b + MG - 1) / MG;
                        const C* src = prow + ((size_t)lf * P.ngrp * 4 + k) * Sx + i;
                        for (int u0 = 0; u0 < ng; u0 += 18) {
                            C a[18];
#pragma unroll
                            for (int u = 0; u < 18; ++u)
                                a[u] = u0 + u < ng ? ldcg(src + (size_t)(u0 + u) * 4 * Sx) : C{0, 0};
#pragma unroll
                            for (int u = 0; u < 18; ++u) s = s + a[u];
                        }
                    }
                    s_t[row * (XC + 2) + il] = s;
                }
                __syncthreads();
                for (int q = tid; q < 2 * xn; q += NT) {
                    const int row = q / xn, il = q - row * xn, i = x0 + il;
                    const size_t o = ((size_t)c * 2 + row) * Sx + i;
                    const C vv = first ? ((const C*)P.rt)[(size_t)(P.mid[c] - 1 + row) * Sx + i]
                                       : (one && stepped ? s_own[row * XC + il] : ldcg(v + o));
                    if (one) s_vs[row * XC + il] = first ? C{0, 0} : (stepped ? s_vs[row * XC + il] : vsum[o]) + vv;
                    else vsum[o] = first ? C{0, 0} : vsum[o] + vv;
                    const C* tc = s_t + (row + 1) * (XC + 2) + il + 1;
                    C at;
                    if (P.q1) {
                        at = q1_row<T>(1, i, g, [&](int dj, int di) { return tc[dj * (XC + 2) + di]; });
                    } else {
                        at = op_diag_t<T>(1, i, g) * tc[0] - tc[-1] - tc[1] -
                             (T)wcol(i, Sx) * (tc[-(XC + 2)] + tc[XC + 2]);
                    }
                    const C rs = vv - at;
                    s_rs[row * XC + il] = rs;
                    if (!one) res0[o] = rs;
                }
                __syncthreads();
                if (stage_c) {
                    cp_async_wait_all();
                    __syncthreads();
                }
                {
                    const C* c0 = res ? s_ce + (size_t)q0 * 2 * XC * 3 * L * r
                                      : stage_c ? s_ln : (const C*)P.Cp + P.cp_off[c] + (size_t)x0 * K;
                    const C* c1 = c0 + (size_t)(res || stage_c ? XC : Sx) * K;
                    for (int k0 = 0; k0 < K; k0 += 32) {
                        const int k = k0 + lane;
                        C a0 = {0, 0}, a1 = {0, 0};
                        if (k < K) {
#pragma unroll 8
                            for (int il = warp; il < xn; il += NW) {
                                cfma_cj(a0, c0[(size_t)il * K + k], s_rs[il]);
                                cfma_cj(a1, c1[(size_t)il * K + k], s_rs[XC + il]);
                            }
                            s_pd[(warp * 2) * kmax + k] = a0;
                            s_pd[(warp * 2 + 1) * kmax + k] = a1;
                        }
                    }
                }
                __syncthreads();
                // slots: the ancestors' columns (both rows), the own node's first and second child
                for (int s = tid; s < (lev + 2) * r; s += NT) {
                    const bool own1 = s >= (lev + 1) * r;
                    const int k = own1 ? s - r : s;
                    C t = {0, 0};
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        if (!own1) t = t + s_pd[(w * 2) * kmax + k];
                        if (own1 || s < lev * r) t = t + s_pd[(w * 2 + 1) * kmax + k];
                    }
                    pd[(size_t)e * (L + 1) * r + s] = t;
                }
                __syncthreads();
            }
            bar.arrive();
            if (kfit) {
                // and as many columns of its E panel as fit there, for phase C: [row][k][XC]
                const C* src = (const C*)P.Ep + P.ep_off[sc_] + sx0;
                for (int k = warp; k < 2 * kfit; k += NW) {
                    const int row = k >= kfit, kk = k - row * kfit;
                    for (int x = lane; x < sxn; x += 32)
                        cp_async_el(s_ln + (size_t)k * XC + x, src + ((size_t)row * sKe + kk) * Sx + x);
                }
                cp_async_commit();
            }
            if (!(ok = bar.wait())) break;
            // ------------------------------------------------------------------ Y
            // d[e]: the partials of the cuts under the entry's child and of the own cut, by
            // eight lanes (dist: a warp) in a fixed order
            {
                const int EL = dist ? 32 : 8, EB = NT / EL;
                const int sub = tid & (EL - 1);
                for (int eb = dist ? rank * EB : 0; eb < D; eb += dist ? gsz * EB : EB) {
                    const int e = eb + tid / EL;
                    C s = {0, 0};
                    if (e < D) {
                        const int p = e / (2 * r), j = e - p * 2 * r, k = j >= r, jr = j - k * r;
                        const int l = 31 - __clz(p + 1), t = p + 1 - (1 << l);
                        const int span = 1 << (L - l), ca = t * span + k * (span / 2);
                        const int own = t * span + span / 2 - 1;
                        const int nin = span / 2 - 1;    // cuts inside the child
#pragma unroll 4
                        for (int q = sub; q < (nin + 1) * nch; q += EL) {
                            const int cc = q / nch, ch = q - cc * nch;
                            const int cut = cc < nin ? ca + cc : own;
                            const int slot = (cc < nin ? l : l + k) * r + jr;
                            s = s + ldcg(pd + ((size_t)cut * nch + ch) * (L + 1) * r + slot);
                        }
                    }
                    for (int o = EL / 2; o > 0; o >>= 1) {
                        s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
                        s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
                    }
                    if (sub == 0 && e < D) {
                        if (dist) gd[e] = s;
                        else s_d[e] = s;
                    }
                }
            }
            if (dist) {
                if (!(ok = bar())) break;
                for (int e = tid; e < D; e += NT) s_d[e] = ldcg(gd + e);
            }
            __syncthreads();
            for (int e = dist ? rank * NW + warp : warp; e < D; e += dist ? gsz * NW : NW) {
                int l, t;
                const int mo = cut_m_row(e, L, r, l, t);
                const C* mr = dist ? Mt + mo : s_m + mo;
                C s = {0, 0};
                for (int lv = l, k0 = 0; lv < L; ++lv) {
                    const int q0 = ((1 << lv) - 1 + (t << (lv - l))) * 2 * r, n = 2 * r << (lv - l);
#pragma unroll 8
                    for (int k = lane; k < n; k += 32) cfma(s, mr[k0 + k], s_d[q0 + k]);
                    k0 += n;
                }
                s = warp_sum(s);
                if (lane == 0) {
                    if (dist) gy[e] = s;
                    else s_y[e] = s;
                }
            }
            if (dist) {
                if (!(ok = bar())) break;
                for (int e = tid; e < D; e += NT) s_y[e] = ldcg(gy + e);
            }
            __syncthreads();
            if (rank == 0)
                for (int e = tid; e < D; e += NT)
                    s_ya[e] = first ? s_y[e] : (stepped ? s_ya[e] : yacc[e]) + s_y[e];
            if (timing) { const unsigned long long t = gtime(); tB += t - t0; t0 = t; }
            // ------------------------------------------------------------------ C
            for (int e = rank, q0 = 0; e < P.nB; e += gsz, ++q0) {
                const int c = e / nch, x0 = (e - c * nch) * XC, xn = min(XC, Sx - x0);
                const int lev = cut_level(c, L), ne = 2 * L - lev, Ke = ne * r;
                const C* E = res ? s_ce + (size_t)q0 * 2 * XC * 3 * L * r + 2 * XC * (lev + 1) * r
                                 : (const C*)P.Ep + P.ep_off[c] + x0;
                const int ldx = res ? XC : Sx;
                const unsigned short* yi = P.yidx + c * 2 * CUT_MAXL;
                // (row, x) pairs times shares of the columns; a share's partial per pair
                const int np = 2 * xn, kg = min(CUT_KG, max(1, NT / np));
                if (kfit) {
                    cp_async_wait_all();
                    __syncthreads();
                }
                for (int q = tid; q < np * kg; q += NT) {
                    const int kk = q / np, pr = q - kk * np, row = pr / xn, il = pr - row * xn;
                    const C* er = E + (size_t)row * Ke * ldx + il;
                    C s = {0, 0};
                    for (int gq = 0; gq < ne; ++gq) {
                        const C* yg = s_y + yi[gq];
                        const C* eg = er + (size_t)gq * r * ldx;
                        int j = kk;
                        if (gq * r < kfit) {
                            const C* es = s_ln + ((size_t)row * kfit + gq * r) * XC + il;
                            const int je = min(r, kfit - gq * r);
#pragma unroll 8
                            for (; j < je; j += kg) cfma(s, es[j * XC], yg[j]);
                        }
#pragma unroll 8
                        for (; j < r; j += kg) cfma(s, eg[(size_t)j * ldx], yg[j]);
                    }
                    s_up[kk * 2 * XC + row * XC + il] = s;
                }
                __syncthreads();
                float nn = 0.f;   // |v|^2, one partial a warp
                for (int q = tid; q < np; q += NT) {
                    const int row = q / xn, il = q - row * xn;
                    const size_t o = ((size_t)c * 2 + row) * Sx + x0 + il;
                    C s = one ? s_rs[row * XC + il] : res0[o];
                    for (int w = 0; w < kg; ++w) s = s - s_up[w * 2 * XC + row * XC + il];
                    v[o] = s;
                    if (one) s_own[row * XC + il] = s;
                    nn += (float)abs2(inv0 * s);
                }
                nn = warp_sum(nn);
                if (lane == 0) s_red[warp] = nn;
                __syncthreads();
                if (tid == 0) {
                    float t = 0.f;
#pragma unroll
                    for (int w = 0; w < NW; ++w) t += s_red[w];
                    P.npart[e] = t;
                }
            }
            stepped = true;
            if (gm_steps) {
                if (timing) tC += gtime() - t0;   // (the Arnoldi step is no phase of the iteration)
                // the Arnoldi step: P.v takes the next step's input
                if (first && rank == 0)
                    for (int e = tid; e < D; e += NT) ((C*)G.y0)[e] = s_ya[e];
                if (!(ok = gm_arnoldi<T, NT>(P, G, s_gm, bar, rank, gsz, in_round, align16(s_ln),
                                            (int)((MG + 4) * Sx * sizeof(C) / sizeof(c128)) - 1))) break;
                __syncthreads();
                if (one && rank < P.nB) {
                    const int c = rank / nch, x0 = (rank - c * nch) * XC, xn = min(XC, Sx - x0);
                    for (int q = tid; q < 2 * xn; q += NT) {
                        const int row = q >= xn, il = q - row * xn;
                        s_own[row * XC + il] = v[((size_t)c * 2 + row) * Sx + x0 + il];
                    }
                }
            }
            if (!(ok = bar())) break;
            // the norm, in the same order in every warp; then the tests
            n2 = 0.f;
#pragma unroll 5
            for (int e = lane; e < P.nB; e += 32) n2 += __ldcg(P.npart + e);
            n2 = warp_sum(n2);
            if (timing && !gm_steps) tC += gtime() - t0;
            first = false;
            ++it;
            ++in_round;
            reason = watch.test(n2, it, P, thr_anchor, thr_test);
            ++done;
            // (a GMRES cycle: at its stop, written before the barrier, or its last step)
            if (gm_steps) reason = __ldcg(&G.ls.st->stop) || done == gm_steps ? CUT_LIMIT : 0;
            else if (!reason && done == max_steps) reason = CUT_LIMIT;
            if (reason) break;
        }
        if (ok && one && rank < P.nB) {
            const int c = rank / nch, x0 = (rank - c * nch) * XC, xn = min(XC, Sx - x0);
            for (int q = tid; q < 2 * xn; q += NT) {
                const int row = q / xn, il = q - row * xn;
                vsum[((size_t)c * 2 + row) * Sx + x0 + il] = s_vs[row * XC + il];
            }
        }
        if (ok && rank == 0)
            for (int e = tid; e < D; e += NT) yacc[e] = s_ya[e];
        if (ok && rank == 0 && tid == 0) {
            ctl->it = it;
            ctl->in_round = in_round;
            ctl->reason = reason;
            ctl->n2 = (double)n2 * n0;
            ctl->n0 = n0;
            watch.store(*ctl, n0);
            ctl->ns[0] += (double)tA;
            ctl->ns[1] += (double)tB;
            ctl->ns[2] += (double)tC;
        }
    }
    if (!ok) cp_async_wait_all();   // the panels a barrier that gave up left on their way
}

// ------------------------------------------------- the iteration on one cluster
// The complex64 problems whose data fits sixteen blocks' shared memory (255 columns at
// r = 16: 205 KB a block) run on a cluster of sixteen with everything on chip.  The phases
// are those above with one item a block, and what they exchange goes straight into the
// consumers' shared memory (st.async, counted by the consumer's mbarrier), so that a phase
// waits for one remote store instead of draining its stores, a barrier and a load from the
// L2 (each 0.4 to 0.7 us):
//   1: rows of the leaf items to the blocks of their cuts (with the halo columns);
//   2: the products with the basis rows to every block, which forms y itself;
//   3: v to the blocks of the two leaves at the cut, and |v|^2 to every block.
// One buffer each is enough: 2 and 3 go from every block to every block (a word where there
// is nothing to tell), so a block that is a phase ahead has heard from all others that they
// are done with the buffer, and the mbarrier's phase, it writes next.
// 544 threads: a warp for each of the 17 modes a block has at 255^2 with four leaves and overlap
// 2; where a block has more (two levels: from 263^2; it takes grids up to 268^2), some warps have
// a second line.
static constexpr int CC_CL = 16, CC_NT = 544, CC_NW = CC_NT / 32;
struct CcSmem {
    int xi, ln, v, m, c, e, t, red, up, rs, d, y, ya, own, vs, bx, bd, total;
};
HH_HD CcSmem cc_layout(const CutProb& P) {
    CcSmem s;
    const int r = P.r, L = P.L, D = P.D, XC = P.XC, Ke = 2 * L * r;
    int o = 0;
    s.xi = o; o += P.MG * P.Sx;
    s.ln = o;                       // the lines; phases B, Y and C: the rows and partial sums
    s.t = o;
    s.red = s.t + 4 * (XC + 2);
    s.up = s.red + CC_NW * 2 * L * r;
    const int tmp = 4 * (XC + 2) + CC_NW * 2 * L * r + (CUT_KG * 2 * XC > CC_NT ? CUT_KG * 2 * XC : CC_NT);
    o += P.MG * P.Sx > tmp ? P.MG * P.Sx : tmp;
    s.v = o; o += 4 * P.Sx;
    s.m = o; o += cut_m_elems(L, r);
    s.c = o; o += 2 * XC * (2 * L + 1) * r;
    s.e = s.c;                      // E follows the block's C panel
    s.rs = o; o += 2 * XC;
    s.d = o; o += D;
    s.y = o; o += Ke;               // in the order of E's columns
    s.ya = o; o += D;
    s.own = o; o += 2 * XC;
    s.vs = o; o += 2 * XC;
    s.bx = o; o += 4 * P.ngrp * (XC + 2);
    s.bd = o; o += P.nB * (L + 1) * r;
    s.total = o;
    return s;
}
// GM: with the Arnoldi steps of a GMRES cycle (apart, for its registers).
template <bool GM>
__global__ void __launch_bounds__(CC_NT, 1) k_cut_cluster(const CutProb* __restrict__ probs, int nprob,
                                                          const int* modes, int mode_all, int* err, long long limit,
                                                          int prof, int max_steps, CutGmres G, int gm_steps,
                                                          unsigned* bars) {
    using C = c64;
    constexpr int NT = CC_NT, NW = CC_NW;
    extern __shared__ __align__(16) unsigned char csm[];
    __shared__ __align__(32) C s_vin[CUT_MGMAX][4], s_vout[CUT_MGMAX][4], s_sc[CUT_MGMAX];
    __shared__ float s_nrm[CC_CL][4], s_word[CC_CL];
    __shared__ unsigned short s_yi[CUT_KMAX * 2];
    __shared__ int s_ng[2];
    __shared__ __align__(8) uint64_t s_mb[3];
    __shared__ CutProb P;
    __shared__ CutLeaf F;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), ngroups = gridDim.x / CC_CL, group = blockIdx.x / CC_CL;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int k = 0; k < 3; ++k) mbar_init(&s_mb[k], 1);
        fence_barrier_init();
    }
    if (GM && rank == 0 && tid == 0) *G.ls.st = GmresState{0, 0, 0, 0, 0.0, 0.0};   // (as k_cut_steps)
    cluster.sync();
    const uint32_t mb = smem_u32(s_mb);
    unsigned phase = 0;   // steps this block has done: the mbarriers' parity
    [[maybe_unused]] GroupBar bar{bars + group, (unsigned)CC_CL, 0u, err, 16 * limit};   // of the Arnoldi steps
    bool ok = true;
    // wait for `bytes` of exchange k; bounded
    auto wait = [&](int k, unsigned bytes) -> bool {
        if (tid == 0) mbar_arrive_expect_tx(&s_mb[k], bytes);
        bool got = warp != 0;   // one warp polls
        for (long long q = 0; q < limit && !got; ++q) {
            uint32_t d;
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
                " selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(d) : "r"(mb + 8 * k), "r"(phase & 1u) : "memory");
            got = d != 0;
        }
        if (!got) atomicExch(err, DEV_TIMEOUT);
        return __syncthreads_and(got);
    };
    for (int pi = group; pi < nprob; pi += ngroups) {
        const int mode = modes ? modes[pi] : mode_all;
        if (!mode) continue;
        if (!ok) {
            // a wait gave up: only keep the cluster's barriers in step with the blocks that go on
            cluster.sync();
            continue;
        }
        __syncthreads();
        for (int q = tid; q < (int)(sizeof(CutProb) / 4); q += NT) ((int*)&P)[q] = ((const int*)(probs + pi))[q];
        __syncthreads();
        const int Sx = P.Sx, r = P.r, L = P.L, nch = P.nch, XC = P.XC, D = P.D, MG = P.MG, ngrp = P.ngrp;
        const CcSmem lay = cc_layout(P);
        C* const sm = (C*)csm;
        C *s_xi = sm + lay.xi, *s_ln = sm + lay.ln, *s_v = sm + lay.v, *s_m = sm + lay.m, *s_t = sm + lay.t,
          *s_red = sm + lay.red, *s_up = sm + lay.up, *s_rs = sm + lay.rs, *s_d = sm + lay.d, *s_y = sm + lay.y,
          *s_ya = sm + lay.ya, *s_own = sm + lay.own, *s_vs = sm + lay.vs, *s_bx = sm + lay.bx, *s_bd = sm + lay.bd;
        CutCtl* ctl = P.ctl;
        OpGeom g;
        g.b = 3;
        g.Sx = Sx;
        g.kh = P.kh;
        g.khr = nullptr;
        g.q1 = P.q1;
        // the block's leaf item and cut item
        const int lf = min(rank / ngrp, P.ncut), m0 = (rank - lf * ngrp) * MG;
        if (tid < (int)(sizeof(CutLeaf) / 4)) ((int*)&F)[tid] = ((const int*)(P.leaf + lf))[tid];
        const bool has_b = rank < P.nB;
        const int c = has_b ? rank / nch : 0, ch = rank - c * nch, x0 = has_b ? ch * XC : 0;
        const int xn = has_b ? min(XC, Sx - x0) : 0;   // at least one column by the plan's choice of XC
        const int lev = cut_level(c, L), K = (lev + 1) * r, Ke = (2 * L - lev) * r;
        C* s_c = sm + lay.c;
        C* s_e = s_c + 2 * XC * K;
        if (tid >= 64 && tid < 66) s_ng[tid - 64] = has_b ? (P.leaf[c + tid - 64].b + MG - 1) / MG : 0;
        __syncthreads();
        const int ng0 = s_ng[0], ng1 = s_ng[1];
        const int b = F.b, nm = rank < P.nA ? max(0, min(MG, b - m0)) : 0;
        bool first = mode == 1;
        const double n0 = first ? *P.nrm : ctl->n0;
        const float thr_test = (float)(P.test2 * *P.b2 / n0), thr_anchor = (float)P.anchor2;
        const float inv0 = (float)(1.0 / sqrt(n0));
        int it = ctl->it, in_round = first ? 0 : ctl->in_round, reason = 0;
        StepWatch watch(*ctl, n0);
        int done = 0;
        float n2 = 0.f;
        // resident data: V entries, xi and its lane products, M, the panels, the state
        for (int q = tid; q < 4 * nm; q += NT) {
            const C* V = (const C*)F.V;
            const int k = q / nm, w = q - k * nm;
            const C sc = F.sc ? ((const C*)F.sc)[m0 + w] : C{1, 0};
            s_vout[w][k] = F.rout[k] >= 0 ? V[(size_t)F.rout[k] * b + m0 + w] : C{0, 0};
            const C vi = F.rin[k] >= 0 ? V[(size_t)F.rin[k] * b + m0 + w] : C{0, 0};
            s_vin[w][k] = F.sc ? sc * vi : vi;
            if (k == 0) s_sc[w] = sc;
        }
        for (int w = warp; w < nm; w += NW) {
            const C* xi = (const C*)F.xi + (size_t)(m0 + w) * Sx;
            for (int i = lane; i < Sx; i += 32) cp_async_el(s_xi + w * Sx + i, xi + i);
        }
        for (int q = tid; q < cut_m_elems(L, r); q += NT) cp_async_el(s_m + q, (const C*)P.M + q);
        if (has_b) {
            for (int row = 0; row < 2; ++row) {
                const C* sc = (const C*)P.Cp + P.cp_off[c] + ((size_t)row * Sx + x0) * K;
                for (int u = tid; u < xn * K; u += NT) cp_async_el(s_c + row * XC * K + u, sc + u);
                const C* se = (const C*)P.Ep + P.ep_off[c] + (size_t)row * Ke * Sx + x0;
                for (int k = warp; k < Ke; k += NW)
                    for (int x = lane; x < xn; x += 32) cp_async_el(s_e + (row * Ke + k) * XC + x, se + (size_t)k * Sx + x);
            }
            for (int k = tid; k < Ke; k += NT) s_yi[k] = (unsigned short)(P.yidx[c * 2 * CUT_MAXL + k / r] + k % r);
            for (int q = tid; q < 2 * xn; q += NT) {
                const int row = q / xn, il = q - row * xn;
                const size_t o = ((size_t)c * 2 + row) * Sx + x0 + il;
                s_own[row * XC + il] =
                    first ? ((const C*)P.rt)[(size_t)(P.mid[c] - 1 + row) * Sx + x0 + il] : ((const C*)P.v)[o];
                s_vs[row * XC + il] = first ? C{0, 0} : ((const C*)P.vsum)[o];
            }
        }
        for (int q = tid; q < 4 * ngrp * (XC + 2); q += NT) s_bx[q] = C{0, 0};
        for (int e = tid; e < D; e += NT) s_ya[e] = first ? C{0, 0} : ((const C*)P.yacc)[e];
        for (int q = tid; q < 4 * Sx; q += NT) {
            const int k = q / Sx, i = q - k * Sx;
            s_v[q] = !first && F.rin[k] >= 0 ? ((const C*)P.v)[((size_t)(lf - (k < 2)) * 2 + (k & 1)) * Sx + i] : C{0, 0};
        }
        // bytes of the three exchanges
        const int xw = min(Sx, x0 + xn + 1) - max(0, x0 - 1);   // columns with the halo
        const unsigned by1 = has_b ? 8u * 2u * (unsigned)xw * (unsigned)(ng0 + ng1) : 0u;
        unsigned by2 = 4u * (unsigned)(CC_CL - P.nB);
        for (int q = 0; q < P.ncut; ++q) by2 += 8u * (unsigned)(nch * (cut_level(q, L) + 2) * r);
        const unsigned by3 = 4u * 4u * CC_CL + (nm > 0 ? 8u * 2u * (unsigned)Sx * ((F.rin[0] >= 0) + (F.rin[2] >= 0)) : 0u);
        unsigned long long t0 = 0, tA = 0, tB = 0, tC = 0;
        const bool timing = prof && rank == 0 && tid == 0;
        cp_async_commit();
        cp_async_wait_all();
        __syncwarp();
        LineScan<float> scan;   // of the warp's first line (its xi lines are its own copies)
        if (warp < nm) line_scan_init(s_xi + warp * Sx, Sx, lane, scan);
        // this thread's places in phases Y and C: an entry of d and its share of the partials, an
        // entry of y and its share of M's row, a cut point and its share of E's columns
        const int ke = tid >> 2;
        int kb[4] = {-1, -1, -1, -1};
        if (ke < D) {
            const int p = ke / (2 * r), j = ke - p * 2 * r, kc = j >= r, jr = j - kc * r;
            const int l = 31 - __clz(p + 1), t = p + 1 - (1 << l);
            const int span = 1 << (L - l), ca = t * span + kc * (span / 2), own = t * span + span / 2 - 1;
            const int nin = span / 2 - 1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int q = (tid & 3) + 4 * u;   // at most 16 items in all
                if (q < (nin + 1) * nch) {
                    const int cc = q / nch, cu = cc < nin ? ca + cc : own;
                    kb[u] = (cu * nch + q - cc * nch) * (L + 1) * r + (cc < nin ? l : l + kc) * r + jr;
                }
            }
        }
        const int ks = min(5, NT / D), msub = tid / D, me = tid - msub * D;
        const bool mon = msub < ks;
        int ml, mt;
        const int mi = me % (2 * r), mo = cut_m_row(me / (2 * r) * 2 * r, L, r, ml, mt) + mi;
        const int np = 2 * xn, kg = np ? min(CUT_KG, max(1, NT / np)) : 1;
        const int uk = np ? tid / np : kg, upr = np ? tid - uk * np : 0, urow = upr >= xn, uil = upr - urow * xn;
        cluster.sync();   // every block's buffers are ready
        for (;;) {
            if (timing) t0 = gtime();
            // ------------------------------------------------------------------ A
            for (int u = 0; u < 2; ++u) {
                const int w = warp + u * NW;
                if (w >= nm) break;
                C* fs = s_ln + w * Sx;
                if (first) {
                    const C* f0 = (const C*)F.fh0 + (size_t)(m0 + w) * Sx;
                    const C sc = s_sc[w];
                    for (int i = lane; i < Sx; i += 32) fs[i] = F.sc ? sc * f0[i] : f0[i];
                } else {
                    const C a0 = s_vin[w][0], a1 = s_vin[w][1], a2 = s_vin[w][2], a3 = s_vin[w][3];
#pragma unroll 3
                    for (int i = lane; i < Sx; i += 32) {
                        C f = a0 * s_v[i];
                        cfma(f, a1, s_v[Sx + i]);
                        cfma(f, a2, s_v[2 * Sx + i]);
                        cfma(f, a3, s_v[3 * Sx + i]);
                        fs[i] = f;
                    }
                }
                __syncwarp();
                if (u == 0) {
                    line_solve(s_xi + w * Sx, fs, Sx, lane, scan);
                } else {
                    LineScan<float> second;
                    line_scan_init(s_xi + w * Sx, Sx, lane, second);
                    line_solve(s_xi + w * Sx, fs, Sx, lane, second);
                }
            }
            __syncthreads();
            // rows of the result: up (to the cut above) and down, one thread a column and pair
            if (nm > 0)
                for (int q = tid; q < 2 * Sx; q += NT) {
                    const int h = q >= Sx, i = q - h * Sx;
                    if (F.rout[2 * h] < 0) continue;
                    C o0 = {0, 0}, o1 = {0, 0};
                    for (int w = 0; w < nm; ++w) {
                        const C f = s_ln[w * Sx + i];
                        const cpair<float> vo = *(const cpair<float>*)&s_vout[w][2 * h];
                        cfma(o0, vo.x, f);
                        cfma(o1, vo.y, f);
                    }
                    // h = 0: rows 2, 3 of cut lf - 1; h = 1: rows 0, 1 of cut lf
                    const int cc = lf - 1 + h, row = h ? 0 : 2, grp = rank - lf * ngrp;
                    const int k = i / XC;
                    const int ka = (i - k * XC == 0 && k > 0) ? k - 1 : k;
                    const int kb = (i - k * XC == XC - 1 && k + 1 < nch) ? k + 1 : k;
                    for (int kk = ka; kk <= kb; ++kk) {
                        const int dst = cc * nch + kk, il = i - kk * XC + 1;
                        const uint32_t rm = mapa(mb, dst);
                        const uint32_t ra = mapa(smem_u32(s_bx + (row * ngrp + grp) * (XC + 2) + il), dst);
                        st_async(ra, o0, rm);
                        st_async(ra + 8u * ngrp * (XC + 2), o1, rm);
                    }
                }
            if (!(ok = wait(0, by1))) break;
            if (timing) { const unsigned long long t = gtime(); tA += t - t0; t0 = t; }
            // ------------------------------------------------------------------ B
            if (has_b) {
                for (int q = tid; q < 4 * (XC + 2); q += NT) {
                    const int row = q / (XC + 2), il = q - row * (XC + 2);
                    C s = {0, 0};
                    for (int u = 0; u < ngrp; ++u) s = s + s_bx[(row * ngrp + u) * (XC + 2) + il];
                    s_t[q] = s;
                }
                __syncthreads();
                for (int q = tid; q < 2 * xn; q += NT) {
                    const int row = q / xn, il = q - row * xn, i = x0 + il;
                    const C vv = s_own[row * XC + il];
                    if (!first) s_vs[row * XC + il] = s_vs[row * XC + il] + vv;
                    const C* tc = s_t + (row + 1) * (XC + 2) + il + 1;
                    C at;
                    if (P.q1) {
                        at = q1_row<float>(1, i, g, [&](int dj, int di) { return tc[dj * (XC + 2) + di]; });
                    } else {
                        at = op_diag_t<float>(1, i, g) * tc[0] - tc[-1] - tc[1] -
                             (float)wcol(i, Sx) * (tc[-(XC + 2)] + tc[XC + 2]);
                    }
                    s_rs[row * XC + il] = vv - at;
                }
                __syncthreads();
                for (int k0 = 0; k0 < K; k0 += 32) {
                    const int k = k0 + lane;
                    if (k < K) {
                        C a0 = {0, 0}, a1 = {0, 0};
                        for (int il = warp; il < xn; il += NW) {
                            cfma_cj(a0, s_c[il * K + k], s_rs[il]);
                            cfma_cj(a1, s_c[(XC + il) * K + k], s_rs[XC + il]);
                        }
                        s_red[(warp * 2) * L * r + k] = a0;
                        s_red[(warp * 2 + 1) * L * r + k] = a1;
                    }
                }
                __syncthreads();
                // slots (the ancestors' columns, the own node's first and second child), four
                // lanes a slot, each sending to four blocks
                const int ns = (lev + 2) * r;
                for (int q = tid; q < (ns * 4 + 31) / 32 * 32; q += NT) {
                    const int s = q >> 2, sub = q & 3;
                    C t = {0, 0};
                    if (s < ns) {
                        const bool own1 = s >= (lev + 1) * r;
                        const int k = own1 ? s - r : s;
                        for (int w = sub; w < NW; w += 4) {
                            if (!own1) t = t + s_red[(w * 2) * L * r + k];
                            if (own1 || s < lev * r) t = t + s_red[(w * 2 + 1) * L * r + k];
                        }
                    }
#pragma unroll
                    for (int o = 1; o < 4; o <<= 1) {
                        t.re += __shfl_xor_sync(0xffffffffu, t.re, o);
                        t.im += __shfl_xor_sync(0xffffffffu, t.im, o);
                    }
                    if (s < ns) {
                        const uint32_t la = smem_u32(s_bd + rank * (L + 1) * r + s);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int dst = 4 * sub + u;
                            st_async(mapa(la, dst), t, mapa(mb + 8, dst));
                        }
                    }
                }
            }
            else if (tid < CC_CL) st_async(mapa(smem_u32(&s_word[rank]), tid), 0.f, mapa(mb + 8, tid));
            if (!(ok = wait(1, by2))) break;
            // ------------------------------------------------------------------ Y
            {
                C s = {0, 0};
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (kb[u] >= 0) s = s + s_bd[kb[u]];
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
                    s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
                }
                if ((tid & 3) == 0 && ke < D) s_d[ke] = s;
            }
            __syncthreads();
            // y = M d: M transposed within a node's rows, so that the lanes' reads are
            // consecutive; a row's columns shared out over NT / D threads
            if (mon) {
                C s = {0, 0};
                const C* mp = s_m + mo;
                for (int lv = ml; lv < L; ++lv) {   // the subtree's columns, level by level
                    const C* dl = s_d + ((1 << lv) - 1 + (mt << (lv - ml))) * 2 * r;
                    const int n = 2 * r << (lv - ml);
#pragma unroll 4
                    for (int k = msub; k < n; k += ks) cfma(s, mp[k * 2 * r], dl[k]);
                    mp += n * 2 * r;
                }
                s_up[tid] = s;
            }
            __syncthreads();
            // the entries of y this block's E columns take, in their order; all of them in the
            // block that sums them
            for (int k = has_b ? tid : Ke; k < Ke; k += NT) {
                const int e = s_yi[k];
                C s = s_up[e];
                for (int u = 1; u < ks; ++u) s = s + s_up[u * D + e];
                s_y[k] = s;
            }
            if (rank == 0)
                for (int e = tid; e < D; e += NT) {
                    C s = s_up[e];
                    for (int u = 1; u < ks; ++u) s = s + s_up[u * D + e];
                    s_ya[e] = s_ya[e] + s;
                }
            __syncthreads();
            if (timing) { const unsigned long long t = gtime(); tB += t - t0; t0 = t; }
            // ------------------------------------------------------------------ C
            float nn = 0.f;
            if (has_b) {
                if (uk < kg) {   // np kg <= NT
                    const C* er = s_e + urow * Ke * XC + uil;
                    C s = {0, 0};
#pragma unroll 8
                    for (int k = uk; k < Ke; k += kg) cfma(s, er[k * XC], s_y[k]);
                    s_up[uk * 2 * XC + urow * XC + uil] = s;
                }
                __syncthreads();
                for (int q = tid; q < np; q += NT) {
                    const int row = q >= xn, il = q - row * xn;
                    C s = s_rs[row * XC + il];
                    for (int w = 0; w < kg; ++w) s = s - s_up[w * 2 * XC + row * XC + il];
                    s_own[row * XC + il] = s;
                    nn += abs2(inv0 * s);
                }
                __syncthreads();
            }
            if constexpr (GM) {
                if (timing) tC += gtime() - t0;
                // the Arnoldi step: S v goes through P.v, which takes the next step's input
                C* vg = (C*)P.v;
                for (int q = tid; q < np; q += NT) {
                    const int row = q >= xn, il = q - row * xn;
                    vg[((size_t)c * 2 + row) * Sx + x0 + il] = s_own[row * XC + il];
                }
                if (first && rank == 0)
                    for (int e = tid; e < D; e += NT) ((C*)G.y0)[e] = s_ya[e];
                __shared__ GmState s_gm;
                if (!(ok = gm_arnoldi<float, NT>(P, G, s_gm, bar, rank, CC_CL, in_round, align16(s_ln),
                                                P.MG * Sx / 2 - 1))) break;
                __syncthreads();
                for (int q = tid; q < np; q += NT) {
                    const int row = q >= xn, il = q - row * xn;
                    s_own[row * XC + il] = vg[((size_t)c * 2 + row) * Sx + x0 + il];
                }
                __syncthreads();
                // the first block tells the others whether the cycle ends
                nn = rank == 0 && tid == 0 ? (float)*(volatile int*)&G.ls.st->stop : 0.f;
            }
            if (has_b) {
                const int nd = ng0 + ng1;
                for (int q = tid; q < np * nd; q += NT) {
                    const int dq = q / np, pr = q - dq * np, row = pr >= xn, il = pr - row * xn;
                    // leaf c (its cut below: input rows 2, 3), then leaf c + 1 (rows 0, 1)
                    const bool up = dq < ng0;
                    const int dst = up ? c * ngrp + dq : (c + 1) * ngrp + dq - ng0;
                    const uint32_t la = smem_u32(s_v + ((up ? 2 : 0) + row) * Sx + x0 + il);
                    st_async(mapa(la, dst), s_own[row * XC + il], mapa(mb + 16, dst));
                }
            }
            // |v|^2: one partial of the first four warps to every block
            nn = warp_sum(nn);
            if (warp < 4 && lane < CC_CL) st_async(mapa(smem_u32(&s_nrm[rank][warp]), lane), nn, mapa(mb + 16, lane));
            if (!(ok = wait(2, by3))) break;
            n2 = warp_sum((&s_nrm[0][0])[lane] + (&s_nrm[0][0])[lane + 32]);   // alike in every warp
            if (timing && !GM) tC += gtime() - t0;
            first = false;
            ++it;
            ++in_round;
            ++phase;
            reason = watch.test(n2, it, P, thr_anchor, thr_test);
            ++done;
            if (GM) reason = s_nrm[0][0] != 0.f || done == gm_steps ? CUT_LIMIT : 0;
            else if (!reason && done == max_steps) reason = CUT_LIMIT;
            if (reason) break;
        }
        if (ok && has_b)
            for (int q = tid; q < 2 * xn; q += NT) {
                const int row = q / xn, il = q - row * xn;
                const size_t o = ((size_t)c * 2 + row) * Sx + x0 + il;
                ((C*)P.vsum)[o] = s_vs[row * XC + il];
                ((C*)P.v)[o] = s_own[row * XC + il];
            }
        if (ok && rank == 0) {
            for (int e = tid; e < D; e += NT) ((C*)P.yacc)[e] = s_ya[e];
            if (tid == 0) {
                ctl->it = it;
                ctl->in_round = in_round;
                ctl->reason = reason;
                ctl->n2 = (double)n2 * n0;
                ctl->n0 = n0;
                watch.store(*ctl, n0);
                ctl->ns[0] += (double)tA;
                ctl->ns[1] += (double)tB;
                ctl->ns[2] += (double)tC;
            }
        }
    }
    // no block leaves while another's stores may still arrive (after a wait that gave up,
    // also those nobody waited for)
    cluster.sync();
    if (!ok) settle_remote_stores();
    cluster.sync();
}

// The round's summed inputs through the leaves: Fh = the recursions of f^_0 + V^T (the cut
// rows' sums), one warp per mode, for the transform back of every row.
template <typename T>
__global__ void __launch_bounds__(256) k_cut_lines(const CutProb* __restrict__ probs, const int* modes, int wpb) {
    using C = cplx<T>;
    if (modes && !modes[blockIdx.z]) return;
    const CutProb& P = probs[blockIdx.z];
    if ((int)blockIdx.y >= P.ncut + 1) return;
    const int Sx = P.Sx, lf = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const CutLeaf& F = P.leaf[lf];
    const int m = blockIdx.x * wpb + warp;
    if (warp >= wpb || m >= F.b) return;
    extern __shared__ __align__(16) unsigned char lsm[];
    C* as = (C*)lsm + (size_t)warp * 2 * Sx;
    C* fs = as + Sx;
    const C* xi = (const C*)F.xi + (size_t)m * Sx;
    const C* f0 = (const C*)F.fh0 + (size_t)m * Sx;
    const C sc = F.sc ? ((const C*)F.sc)[m] : C{1, 0};
    C vin[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) vin[k] = F.rin[k] >= 0 ? ((const C*)F.V)[(size_t)F.rin[k] * F.b + m] : C{0, 0};
    for (int i = lane; i < Sx; i += 32) {
        C f = P.scale ? cvt<T>(*P.scale) * f0[i] : f0[i];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (F.rin[k] >= 0)
                cfma(f, vin[k], ((const C*)P.vsum)[((size_t)(lf - (k < 2)) * 2 + (k & 1)) * Sx + i]);
        as[i] = xi[i];
        fs[i] = F.sc ? sc * f : f;
    }
    __syncwarp();
    warp_line_solve(as, fs, Sx, lane);
    C* fh = (C*)F.fh + (size_t)m * Sx;
    for (int i = lane; i < Sx; i += 32) fh[i] = fs[i];
}

// ut = u + w + sum over the levels of C_p y_p at every grid point (w: the composed leaf
// solutions; y: the round's summed corrections).  HBM-bound: each level's basis read once,
// L r values a point.  The rows between two cuts share the nodes and are contiguous, so a
// block takes 256 PT points of them, whatever the columns.  1023^2, r = 32, complex64:
// 193 us with a block per row and 256 columns, 148 here (PT = 4); 255^2 20 and 11 us (PT = 1).
template <typename T, int PT>
__global__ void __launch_bounds__(256) k_cut_update(const CutUpdJob* __restrict__ jobs) {
    using C = cplx<T>;
    __shared__ C sy[CUT_KMAX];
    __shared__ const C* sc[CUT_MAXL];
    __shared__ size_t sn[CUT_MAXL];
    const CutUpdJob& J = jobs[blockIdx.z];
    const CutProb& P = *J.prob;
    const int Sx = P.Sx, r = P.r, L = P.L, lf = blockIdx.y;
    if (lf > P.ncut) return;
    const int m0 = lf ? P.mid[lf - 1] : 0, m1 = lf < P.ncut ? P.mid[lf] : J.Sy;
    const size_t n = (size_t)(m1 - m0) * Sx, t0 = blockIdx.x * (size_t)(256 * PT), t = t0 + threadIdx.x;
    if (t0 >= n) return;
    for (int q = threadIdx.x; q < L * r; q += 256) {
        const int l = q / r, j = q - l * r;
        const int p = (1 << l) - 1 + (lf >> (L - l)), k = (lf >> (L - l - 1)) & 1;
        sy[q] = ((const C*)P.yacc)[(size_t)p * 2 * r + k * r + j];
        if (j == 0) {
            const CutNode& nd = P.node[p];
            sn[l] = nd.N;
            sc[l] = (const C*)nd.C + (size_t)(k * r) * nd.N + (size_t)(m0 - nd.ra) * Sx;
        }
    }
    __syncthreads();
    const size_t o = (size_t)m0 * Sx;
    size_t ti[PT];             // (past the end: the last point again, so that no load is guarded)
    C acc[PT];
    c128 u[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        ti[i] = t + 256 * i < n ? t + 256 * i : n - 1;
        acc[i] = ((const C*)J.w)[o + ti[i]];
        u[i] = J.u[o + ti[i]];
    }
    for (int l = 0; l < L; ++l) {
        const C* c = sc[l];
        const size_t N = sn[l];
#pragma unroll 16 / PT
        for (int j = 0; j < r; ++j, c += N)
#pragma unroll
            for (int i = 0; i < PT; ++i) cfma(acc[i], c[ti[i]], sy[l * r + j]);
    }
#pragma unroll
    for (int i = 0; i < PT; ++i)
        if (t + 256 * i < n) J.ut[o + ti[i]] = u[i] + cvt<double>(acc[i]);
}

// ----------------------------------------------------- end of a GMRES cycle (CutGmres)
// Coefficients c = R^{-1} g (back substitution by one warp, in every block: R and the
// reciprocals of its diagonal in shared memory first), the scale sum c_j alpha_j of r, and
// the input sum c_j g_j on the cut rows, into P.v; its corrections and sums start from the
// first step's, scaled, and zero.  Four threads an entry.
template <typename T>
__global__ void __launch_bounds__(256) k_cut_gm_combine(const CutProb* __restrict__ prob, CutGmres G, int nG) {
    using C = cplx<T>;
    __shared__ c128 c[72], dinv[72], s_a;
    extern __shared__ __align__(16) unsigned char rsm[];
    c128* R = (c128*)rsm;                        // [jn][jn]
    const CutProb& P = *prob;
    const int tid = threadIdx.x, mk = G.ls.mk;
    const int jn = G.ls.st->stop ? G.ls.st->jstop : G.ls.st->steps;
    for (int q = tid; q < jn * jn; q += 256) R[q] = G.ls.H[(size_t)(q / jn) * mk + q % jn];
    for (int i = tid; i < jn; i += 256) {
        const c128 d = G.ls.H[(size_t)i * mk + i];
        dinv[i] = abs2(d) > 0 ? cinv(d) : c128{0.0, 0.0};
        c[i] = G.ls.g[i];
    }
    __syncthreads();
    if (tid < 32)
        for (int i = jn - 1; i >= 0; --i) {
            const c128 y = c[i] * dinv[i];
            __syncwarp();
            if (tid == 0) c[i] = y;
            for (int k = tid; k < i; k += 32) c[k] = c[k] - R[k * jn + i] * y;
            __syncwarp();
        }
    __syncthreads();
    if (tid < 32) {
        c128 a = {0, 0};
        for (int i = tid; i < jn; i += 32) cfma(a, c[i], G.alpha[i]);
        a = warp_sum(a);
        if (tid == 0) {
            s_a = a;
            if (blockIdx.x == 0) *G.scale = a;
        }
    }
    __syncthreads();
    const c128 a = s_a;
    const int sub = tid & 3;
    for (int e0 = blockIdx.x * 64; e0 < nG; e0 += gridDim.x * 64) {
        const int e = e0 + (tid >> 2);
        c128 x = {0, 0};
        if (e < nG)
            for (int i = sub; i < jn; i += 4) cfma(x, c[i], G.V[(size_t)i * nG + e]);
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            x.re += __shfl_xor_sync(0xffffffffu, x.re, o);
            x.im += __shfl_xor_sync(0xffffffffu, x.im, o);
        }
        if (e < nG && sub == 0) {
            ((C*)P.v)[e] = cvt<T>(x - a * G.rG[e]);
            ((C*)P.vsum)[e] = C{0, 0};
        }
    }
    if (blockIdx.x == 0)
        for (int d = tid; d < P.D; d += 256) ((C*)P.yacc)[d] = cvt<T>(a * cvt<double>(((const C*)G.y0)[d]));
}

// ---------------------------------------------------------------------- launchers
template <typename T>
void launch_cut_panels(const CutCpEntry* cp, int ncp, const CutEpEntry* ep, int nep, int Sx, int r, OpGeom g,
                       cudaStream_t s) {
    g.b = 3;
    k_cut_cp<T><<<dim3((Sx + 31) / 32, ncp), 256, 0, s>>>(cp, Sx, r);
    note_launch();
    k_cut_ep<T><<<dim3((Sx + 255) / 256, nep, r), 256, 0, s>>>(ep, Sx, r, g);
    note_launch();
}
size_t cut_gram_scratch(int npairs) { return (size_t)npairs * GRAM_SPLIT * 1024 * sizeof(c128); }
template <typename T>
void launch_cut_gram(const CutGramPair* prs, int npairs, int first0, const CutGramDest* ds, int ndest, int Sx, int r,
                     c128* part, cudaStream_t s) {
    k_cut_gram<T><<<dim3(npairs, GRAM_SPLIT), 256, 0, s>>>(prs, Sx, r, part);
    note_launch();
    k_cut_gram_red<<<ndest, 256, 0, s>>>(ds, first0, r, part);
    note_launch();
}
template <typename T>
void launch_cut_minv(const CutMinv* prs, int n, int L, int p2, const c128* G, c128* M, cplx<T>* MT, int tr,
                     cudaStream_t s) {
    k_cut_minv<T><<<dim3(n, (p2 + MINV_ROWS - 1) / MINV_ROWS), 256, 0, s>>>(prs, L, p2, G, M, MT, tr);
    note_launch();
}

size_t cut_m_packed(int L, int r) { return (size_t)cut_m_elems(L, r); }

// Items of a problem and the shared memory of its steps; 0 bytes when the lines do not fit.
// Two forms, by what bounds them:
//  * the complex64 problems whose lines, panels and M fit sixteen blocks' shared memory run
//    on one cluster of sixteen (k_cut_cluster), bound by latency alone;
//  * the others on a grid group of up to one block per SM (k_cut_steps): there the lines
//    (FP64: the pipe, four warps fill it) and the panels' bytes want every SM.
// (148: items and blocks of a group, a block an SM of the 152 with a few to spare; only this
// value was measured.)
static constexpr int CUT_NT = 256, CUT_SMEM = 210 * 1024;
static bool cluster_form(CutProb& P, int b_max) {
    const int NL = P.ncut + 1;
    if (P.D > 128 || NL > CC_CL) return false;
    P.MG = (b_max + CC_CL / NL - 1) / (CC_CL / NL);
    P.ngrp = (b_max + P.MG - 1) / P.MG;
    P.nA = NL * P.ngrp;
    P.XC = (P.Sx + CC_CL / P.ncut - 1) / (CC_CL / P.ncut);
    P.nch = (P.Sx + P.XC - 1) / P.XC;
    P.nB = P.ncut * P.nch;
    // two lines a warp; |v|^2 comes from the first four warps; the halo is one neighbour's
    return P.MG <= 2 * CC_NW && P.MG <= CUT_MGMAX && 2 * P.XC <= 128 && P.XC >= 2 &&
           (2 * P.L) * P.r <= 2 * CUT_KMAX && sizeof(c64) * cc_layout(P).total <= (size_t)CUT_SMEM;
}
template <typename T>
size_t cut_plan(CutProb& P, int b_max, bool cluster) {
    const size_t c = sizeof(cplx<T>), cap = CUT_SMEM;
    const int NL = P.ncut + 1;
    P.res = P.dist = 0;
    P.nbi = 1;
    P.cl = cluster && sizeof(T) == 4 && cluster_form(P, b_max);
    if (P.cl) return c * cc_layout(P).total;
    P.XC = std::min(64, std::max(8, (P.ncut * P.Sx + 147) / 148));
    P.nch = (P.Sx + P.XC - 1) / P.XC;
    P.nB = P.ncut * P.nch;
    P.nbi = (P.nB + 147) / 148;
    for (int mg = std::min(8, std::max(2, (NL * b_max + 147) / 148)); mg >= 1; --mg) {
        P.MG = mg;
        // every block's y = M d while D is small (FP64: its products cost more than the two
        // barriers); the panels kept where there is room
        for (int o = P.D > (sizeof(T) == 4 ? 128 : 32) ? 2 : 0; o < 4; ++o) {
            P.dist = o >> 1;
            P.res = !(o & 1);
            const size_t b = c * cut_smem_layout(P, CUT_NT / 32).total;
            if (b > cap) continue;
            P.ngrp = (b_max + mg - 1) / mg;
            P.nA = NL * P.ngrp;
            return b;
        }
    }
    return 0;
}
// Clusters of CC_CL blocks with this much shared memory that run at once (0: none).
static int cluster_count(size_t smem) {
    static std::atomic<unsigned long long> attr{0};
    if (!once_per_device(attr, [] {
            for (auto fn : {k_cut_cluster<false>, k_cut_cluster<true>})
                if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, CUT_SMEM) != cudaSuccess ||
                    cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
                    return false;
            return true;
        })) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(CC_CL);
    cfg.blockDim = dim3(CC_NT);
    cfg.dynamicSmemBytes = smem;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CC_CL;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_cut_cluster<true>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    return n;
}
bool cut_cluster_ready(size_t smem) {
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || n < 1) {   // planning without a device (hh_footprint)
        cudaGetLastError();
        return true;
    }
    return cluster_count(smem) > 0;
}
template <typename T>
bool launch_cut_steps(const CutProb* probs, int nprob, int group, bool cl, size_t smem, const int* modes, int mode_all,
                      unsigned* bars, int max_groups, int* err, int prof, cudaStream_t s, int max_steps,
                      const CutGmres* gm, int gm_steps) {
    const CutGmres G = gm ? *gm : CutGmres{};
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e;
    const long long polls = wait_polls(1ll << 24);
    if (cl) {
        const int nmax = cluster_count(smem);
        if (nmax < 1) return false;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CC_CL;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(CC_CL * std::min(nprob, nmax));
        cfg.blockDim = dim3(CC_NT);
        if (gm_steps) cudaMemsetAsync(bars, 0, sizeof(unsigned), s);
        // (a try_wait suspends for up to microseconds: fewer of them make about a second)
        e = cudaLaunchKernelEx(&cfg, gm_steps ? k_cut_cluster<true> : k_cut_cluster<false>, probs, nprob, modes, mode_all, err, std::min(polls, 1ll << 20),
                               prof, max_steps, G, gm_steps, bars);
    } else {
        static std::atomic<unsigned long long> attr{0};
        smem_limit_once(attr, k_cut_steps<T, CUT_NT>, CUT_SMEM);
        int sms = 0, nb = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, current_device());
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_cut_steps<T, CUT_NT>, CUT_NT, smem) != cudaSuccess ||
            nb < 1) {
            cudaGetLastError();
            return false;
        }
        const int gsz = std::min(group, sms * nb), ng = std::max(1, std::min({nprob, sms * nb / gsz, max_groups}));
        cudaMemsetAsync(bars, 0, sizeof(unsigned) * ng, s);
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.gridDim = dim3(gsz * ng);
        cfg.blockDim = dim3(CUT_NT);
        e = cudaLaunchKernelEx(&cfg, k_cut_steps<T, CUT_NT>, probs, nprob, gsz, modes, mode_all, bars, err, polls,
                               prof, max_steps, G, gm_steps);
    }
    note_launch();
    return e == cudaSuccess;
}
template <typename T>
void launch_cut_lines(const CutProb* probs, int nprob, const int* modes, int nleaf_max, int b_max, int Sx_max,
                      cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(attr, k_cut_lines<T>, 200 * 1024);
    const size_t per = 2 * sizeof(cplx<T>) * (size_t)Sx_max;
    const int wpb = (int)std::max<size_t>(1, std::min<size_t>(8, (200u << 10) / per));
    k_cut_lines<T><<<dim3((b_max + wpb - 1) / wpb, nleaf_max, nprob), 256, per * wpb, s>>>(probs, modes, wpb);
    note_launch();
}
template <typename T>
void launch_cut_gm_combine(const CutProb* prob, const CutGmres& G, int nG, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(attr, k_cut_gm_combine<T>, 64 * 64 * (int)sizeof(c128));
    k_cut_gm_combine<T><<<std::min(152, (nG + 63) / 64), 256, sizeof(c128) * G.ls.mk * G.ls.mk, s>>>(prob, G, nG);
    note_launch();
}
// four points a thread once that leaves two blocks an SM
static constexpr size_t UPD_WIDE = (size_t)152 * 2 * 1024;
template <typename T>
void launch_cut_update(const CutUpdJob* jobs, int njobs, int nleaf_max, int own_max, int Sx_max, cudaStream_t s) {
    const size_t n = (size_t)own_max * Sx_max;
    const int pt = n * nleaf_max * njobs >= UPD_WIDE ? 4 : 1;
    const dim3 grid((unsigned)((n + 256 * pt - 1) / (256 * pt)), nleaf_max, njobs);
    if (pt == 4) k_cut_update<T, 4><<<grid, 256, 0, s>>>(jobs);
    else k_cut_update<T, 1><<<grid, 256, 0, s>>>(jobs);
    note_launch();
}

#define HH_CUT_INST(T)                                                                                             \
    template void launch_cut_panels<T>(const CutCpEntry*, int, const CutEpEntry*, int, int, int, OpGeom, cudaStream_t); \
    template void launch_cut_gram<T>(const CutGramPair*, int, int, const CutGramDest*, int, int, int, c128*, cudaStream_t); \
    template void launch_cut_minv<T>(const CutMinv*, int, int, int, const c128*, c128*, cplx<T>*, int, cudaStream_t); \
    template size_t cut_plan<T>(CutProb&, int, bool);                                                                       \
    template bool launch_cut_steps<T>(const CutProb*, int, int, bool, size_t, const int*, int, unsigned*, int, int*, int,   \
                                      cudaStream_t, int, const CutGmres*, int);                                                                  \
    template void launch_cut_lines<T>(const CutProb*, int, const int*, int, int, int, cudaStream_t);                  \
    template void launch_cut_gm_combine<T>(const CutProb*, const CutGmres&, int, cudaStream_t);                       \
    template void launch_cut_update<T>(const CutUpdJob*, int, int, int, int, cudaStream_t);
HH_CUT_INST(float)
HH_CUT_INST(double)

}  // namespace hh
