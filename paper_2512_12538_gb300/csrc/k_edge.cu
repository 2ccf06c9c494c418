// k_edge.cu -- the set-up's sub-level solves with their structure used.
//
// The sketches and the basis extension (Sec. 2) apply M_c to vectors that live on one or two
// rows next to child c's interface, and the sketches read two rows (T_c: the sibling's trace)
// or one (its adjoint) of the result.  Such rows lie in one leaf, the edge leaf of c, so
//  * of c's leaves only the edge leaf has a solution, and f^ = V^T f is an outer product;
//  * the residual after the leaf solves vanishes off the cut between the edge leaf and its
//    neighbour in c (see k_cut.cu), so only the nodes on the path from that cut up to c are
//    corrected, from the two rows of their bases at the cut;
//  * the sketches need the recursions and a few rows of V x^, no transform; the extension
//    needs the edge leaf's transform back and the path's bases.
// A pass over all children of a level is then bound by the recursions (FP32 or FP64
// multiply-adds, 44 an element), where it had been two dense b x b transforms per leaf and
// two passes over every basis below the level.
#include <algorithm>
#include <atomic>

#include "k_line.cuh"
#include "kernels.h"

namespace hh {

// Solution rows of the edge leaves: one block per (column, child).  The modes in batches of
// MG lines, one warp a line (xi and the lines in shared memory); after a batch each thread
// adds the batch's share of the rows at its own grid columns.  rows: [4][Sx][nc]: the two
// rows at the inner cut, then the trace rows.  FP64-issue bound in the FP64 form, so a row
// nobody asked for costs nothing, and a single source row's factor goes with the results'
// (383^2, 40 columns, FP64: 656 and 644 us a call).
template <typename T>
__global__ void __launch_bounds__(256) k_edge_rows(const EdgeTask* __restrict__ tasks, int Sx, int nc, int adj, int MG) {
    using C = cplx<T>;
    extern __shared__ __align__(16) unsigned char esm[];
    __shared__ C s_v[6][8];
    __shared__ EdgeTask E;
    C* xs = (C*)esm;                        // [MG][Sx]
    C* ls = xs + (size_t)MG * Sx;           // [MG][Sx]
    C* in = ls + (size_t)MG * Sx;           // [2][Sx]
    C* out = in + 2 * Sx;                   // [4][Sx]
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < (int)(sizeof(EdgeTask) / 4); q += 256) ((int*)&E)[q] = ((const int*)(tasks + blockIdx.y))[q];
    __syncthreads();
    // T_c: data on the interface row, traces on the sibling's two rows; T_c^*: data on those,
    // the interface row read
    const int ai0 = adj ? E.a_sif : E.a_if, ai1 = adj ? E.a_sin : -1;
    const int ao[4] = {E.o0, E.o1, adj ? E.a_if : E.a_sif, adj ? -1 : E.a_sin};
    const C* i0 = (const C*)(adj ? E.vin : E.Om);
    const int b = E.b;
    const C* V = (const C*)E.V;
    for (int i = tid; i < Sx; i += 256) {
        in[i] = i0[(size_t)i * nc + c];
        if (adj) in[Sx + i] = i0[((size_t)Sx + i) * nc + c];
#pragma unroll
        for (int k = 0; k < 4; ++k) out[k * Sx + i] = C{0, 0};
    }
    for (int m0 = 0; m0 < b; m0 += MG) {
        const int nm = min(MG, b - m0);
        __syncthreads();
        if (tid < 6 * nm) {
            const int k = tid / nm, w = tid - k * nm;
            const int a = k == 0 ? ai0 : k == 1 ? ai1 : ao[k - 2];
            C v = a >= 0 ? V[(size_t)a * b + m0 + w] : C{0, 0};
            if (k < 2 && E.sc) v = ((const C*)E.sc)[m0 + w] * v;
            if (k >= 2 && !adj && a >= 0) {          // one source row: its factor here
                C vi = V[(size_t)ai0 * b + m0 + w];
                if (E.sc) vi = ((const C*)E.sc)[m0 + w] * vi;
                v = v * vi;
            }
            s_v[k][w] = v;
        }
        __syncthreads();
        if (warp < nm) {
            C* as = xs + warp * Sx;
            C* fs = ls + warp * Sx;
            const C* xi = (const C*)E.xi + (size_t)(m0 + warp) * Sx;
            const C v0 = s_v[0][warp], v1 = s_v[1][warp];
            for (int i = lane; i < Sx; i += 32) {
                as[i] = xi[i];
                C f = in[i];
                if (adj) {
                    f = v0 * f;
                    cfma(f, v1, in[Sx + i]);
                }
                fs[i] = f;
            }
            __syncwarp();
            LineScan<T> sc;
            line_scan_init(as, Sx, lane, sc);
            line_solve(as, fs, Sx, lane, sc);
        }
        __syncthreads();
        for (int i = tid; i < Sx; i += 256) {
            C o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = out[k * Sx + i];
            for (int w = 0; w < nm; ++w) {
                const C f = ls[w * Sx + i];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (ao[k] >= 0) cfma(o[k], s_v[2 + k][w], f);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) out[k * Sx + i] = o[k];
        }
    }
    C* rows = (C*)E.rows;
    for (int i = tid; i < Sx; i += 256)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (ao[k] >= 0) rows[((size_t)k * Sx + i) * nc + c] = out[k * Sx + i];
}

// Products of the path's bases with the residual -A t at the inner cut (t: the edge leaf's
// two rows there): partial sums over one share of the columns x per block, in the order
// [slot][column]; slots: the ancestors' r columns from level `lev` down, then the own node's
// two children (row above, row below).
static constexpr int EDGE_CH = 24, EDGE_XT = 16;
template <typename T>
__global__ void __launch_bounds__(256) k_edge_proj(const EdgeTask* __restrict__ tasks, int Sx, int nc, int r, OpGeom g) {
    using C = cplx<T>;
    __shared__ EdgeTask E;
    __shared__ C s_r[2][EDGE_XT][64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < (int)(sizeof(EdgeTask) / 4); q += 256) ((int*)&E)[q] = ((const int*)(tasks + blockIdx.y))[q];
    __syncthreads();
    const C* rows = (const C*)E.rows;
    const int na = E.npath - 1, ns = (na + 2) * r;    // ancestors on the path, slots
    const int xs = (Sx + EDGE_CH - 1) / EDGE_CH, xa = blockIdx.x * xs, xb = min(Sx, xa + xs);
    // per slot: panel column and which rows of the cut it takes
    constexpr int SPW = 8;                             // slots a warp takes, 64 a block
    const int s0 = blockIdx.z * 64;
    if (s0 >= ns) return;
    C acc[SPW][2];
#pragma unroll
    for (int u = 0; u < SPW; ++u) acc[u][0] = acc[u][1] = C{0, 0};
    for (int x0 = xa; x0 < xb; x0 += EDGE_XT) {
        __syncthreads();
        for (int q = tid; q < EDGE_XT * nc; q += 256) {
            const int il = q / nc, c = q - il * nc, x = x0 + il;
            C r0 = {0, 0}, r1 = {0, 0};
            if (x < xb) {
                // t(a, x): a = 0..3 the rows mid - 2 .. mid + 1, two of them the edge leaf's
                auto t = [&](int a, int xx) -> C {
                    const int k = E.below ? a - 2 : a;
                    return k >= 0 && k < 2 && xx >= 0 && xx < Sx ? rows[((size_t)k * Sx + xx) * nc + c] : C{0, 0};
                };
                auto at = [&](int a) -> C {
                    if (g.q1) return q1_row<T>(1, x, g, [&](int dj, int di) { return t(a + dj, x + di); });
                    return op_diag_t<T>(1, x, g) * t(a, x) - t(a, x - 1) - t(a, x + 1) -
                           (T)wcol(x, Sx) * (t(a - 1, x) + t(a + 1, x));
                };
                r0 = -at(1);
                r1 = -at(2);
            }
            s_r[0][il][c] = r0;
            s_r[1][il][c] = r1;
        }
        __syncthreads();
        const int xn = min(EDGE_XT, xb - x0);
#pragma unroll
        for (int u = 0; u < SPW; ++u) {
            const int s = s0 + warp + 8 * u;
            if (s >= ns) break;
            const int gs = s / r, j = s - gs * r;
            // ancestor of level lev + gs: both rows; own node: one
            const int k = (gs < na ? E.lev + gs : E.lev + na) * r + j;
            const bool t0 = gs <= na, t1 = gs < na || gs == na + 1;
            const C* p0 = (const C*)E.cp + (size_t)x0 * E.K + k;
            const C* p1 = p0 + (size_t)Sx * E.K;
            for (int il = 0; il < xn; ++il) {
                const C a0 = t0 ? p0[(size_t)il * E.K] : C{0, 0}, a1 = t1 ? p1[(size_t)il * E.K] : C{0, 0};
                if (lane < nc) {
                    cfma_cj(acc[u][0], a0, s_r[0][il][lane]);
                    cfma_cj(acc[u][0], a1, s_r[1][il][lane]);
                }
                if (lane + 32 < nc) {
                    cfma_cj(acc[u][1], a0, s_r[0][il][lane + 32]);
                    cfma_cj(acc[u][1], a1, s_r[1][il][lane + 32]);
                }
            }
        }
    }
    C* pd = (C*)E.pd + (size_t)blockIdx.x * ns * nc;
#pragma unroll
    for (int u = 0; u < SPW; ++u) {
        const int s = s0 + warp + 8 * u;
        if (s >= ns) break;
        if (lane < nc) pd[(size_t)s * nc + lane] = acc[u][0];
        if (lane + 32 < nc) pd[(size_t)s * nc + lane + 32] = acc[u][1];
    }
}

// The path's corrections of one column (block) of one child, FP64: d from the partials, then
// y_q = sum over the path below and at q of M_qs d_s (M packed by subtree, cut_m_offset).
// y: [npath][2r][nc], the node nearest the leaf first.
template <typename T>
__global__ void __launch_bounds__(256) k_edge_y(const EdgeTask* __restrict__ tasks, int L, int nc, int r,
                                                const c128* __restrict__ M) {
    using C = cplx<T>;
    __shared__ EdgeTask E;
    extern __shared__ __align__(16) unsigned char ysm[];
    c128* d = (c128*)ysm;                              // [slots]
    const int tid = threadIdx.x, c = blockIdx.x, p2 = 2 * r;
    for (int q = tid; q < (int)(sizeof(EdgeTask) / 4); q += 256) ((int*)&E)[q] = ((const int*)(tasks + blockIdx.y))[q];
    __syncthreads();
    const int na = E.npath - 1, ns = (na + 2) * r;
    for (int s = tid; s < ns; s += 256) {
        c128 a = {0, 0};
        for (int ch = 0; ch < EDGE_CH; ++ch) a = a + cvt<double>(((const C*)E.pd)[((size_t)ch * ns + s) * nc + c]);
        d[s] = a;
    }
    __syncthreads();
    // rows in turn to eight lanes each
    const int sub = tid & 7;
    for (int e0 = 0; e0 < E.npath * p2; e0 += 32) {
        const int e = e0 + (tid >> 3);
        c128 a = {0, 0};
        if (e < E.npath * p2) {
            const int u = e / p2, i = e - u * p2;      // path node u (0: own), its row i
            const int pu = E.path[u].id;               // of level L - 1 - u
            const c128* mr = M + E.path[u].mo + (size_t)i * cut_m_len(L - 1 - u, L, r);
            const c128* m0 = mr + cut_m_col(pu, E.path[0].id, r);
            for (int s = sub; s < p2; s += 8) cfma(a, m0[s], d[na * r + s]);
            // ancestors below and at u: their columns of the child that holds the cut
            for (int w = 1; w <= u; ++w) {
                const c128* mw = mr + cut_m_col(pu, E.path[w].id, r) + E.path[w].kin * r;
                for (int s = sub; s < r; s += 8) cfma(a, mw[s], d[(na - w) * r + s]);
            }
        }
        for (int o = 4; o > 0; o >>= 1) {
            a.re += __shfl_xor_sync(0xffffffffu, a.re, o);
            a.im += __shfl_xor_sync(0xffffffffu, a.im, o);
        }
        if (sub == 0 && e < E.npath * p2) E.y[(size_t)e * nc + c] = a;
    }
}

// rows 2 and 3 (adj: 2) += sum over the path of C_q y_q at those grid rows: one block per 32
// columns x, row and child; the rows lie with the path nodes' child on the edge's side.
template <typename T>
__global__ void __launch_bounds__(256) k_edge_out(const EdgeTask* __restrict__ tasks, int Sx, int nc, int r, int adj) {
    using C = cplx<T>;
    __shared__ EdgeTask E;
    __shared__ C cs[16][33];
    __shared__ C ys[16][64];
    const int tid = threadIdx.x;
    for (int q = tid; q < (int)(sizeof(EdgeTask) / 4); q += 256) ((int*)&E)[q] = ((const int*)(tasks + blockIdx.z))[q];
    __syncthreads();
    const int x0 = blockIdx.x * 32, grow = adj ? E.g_if : blockIdx.y == 0 ? E.g_sif : E.g_sin;
    C* out = (C*)E.rows + (size_t)(2 + blockIdx.y) * Sx * nc;
    C acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u] = C{0, 0};
    for (int w = 0; w < E.npath; ++w) {
        const EdgePath& P = E.path[w];
        const C* src = (const C*)P.C + (size_t)(P.kedge * r) * P.N + (size_t)(grow - P.ra) * Sx + x0;
        for (int j0 = 0; j0 < r; j0 += 16) {
            const int jn = min(16, r - j0);
            __syncthreads();
            for (int q = tid; q < jn * 32; q += 256) {
                const int j = q >> 5, x = q & 31;
                cs[j][x] = x0 + x < Sx ? src[(size_t)(j0 + j) * P.N + x] : C{0, 0};
            }
            for (int q = tid; q < jn * nc; q += 256) {
                const int j = q / nc, c = q - j * nc;
                ys[j][c] = cvt<T>(E.y[((size_t)w * 2 * r + P.kedge * r + j0 + j) * nc + c]);
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int q = tid + 256 * u;
                if (q >= 32 * nc) break;
                const int x = q / nc, c = q - x * nc;
                for (int j = 0; j < jn; ++j) cfma(acc[u], cs[j][x], ys[j][c]);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int q = tid + 256 * u;
        if (q >= 32 * nc) break;
        const int x = q / nc, c = q - x * nc;
        if (x0 + x < Sx) {
            C& o = out[(size_t)(x0 + x) * nc + c];
            o = o + acc[u];
        }
    }
}

// The recursions of the basis extension, right-hand side V_c on the interface row: Fh as
// k_eig_recur(_cols) leaves it.  Up to 15 columns: one warp per line; from 16 on one warp
// per mode and 32 columns, each lane its column's chain.
template <typename T>
__global__ void __launch_bounds__(256) k_edge_lines(const EdgeTask* __restrict__ tasks, int Sx, int nc, int wpb) {
    using C = cplx<T>;
    const EdgeTask& E = tasks[blockIdx.y];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, line = blockIdx.x * wpb + warp;
    if (warp >= wpb || line >= E.b * nc) return;
    const int m = line / nc, c = line - m * nc;
    extern __shared__ __align__(16) unsigned char esm[];
    C* as = (C*)esm + (size_t)warp * 2 * Sx;
    C* fs = as + Sx;
    const C* xi = (const C*)E.xi + (size_t)m * Sx;
    C v = ((const C*)E.V)[(size_t)E.a_if * E.b + m];
    if (E.sc) v = ((const C*)E.sc)[m] * v;
    for (int i = lane; i < Sx; i += 32) {
        as[i] = xi[i];
        fs[i] = v * ((const C*)E.Vc)[(size_t)i * nc + c];
    }
    __syncwarp();
    warp_line_solve(as, fs, Sx, lane);
    C* fh = (C*)E.Fh + (size_t)line * Sx;
    for (int i = lane; i < Sx; i += 32) fh[i] = fs[i];
}
// Blocks of two warps: a chain is bound by its own latency and, in FP64, by its scheduler's issue
// rate (64 clocks a multiply-add), so the warps go one to a scheduler over all SMs (383^2, r = 32,
// FP64: 442 us in blocks of eight, 226 here).
template <typename T>
__global__ void __launch_bounds__(64) k_edge_chains(const EdgeTask* __restrict__ tasks, int Sx, int nc) {
    using C = cplx<T>;
    constexpr int RB = 16;
    const EdgeTask& E = tasks[blockIdx.y];
    const int cgs = (nc + 31) / 32, wg = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (wg >= E.b * cgs) return;
    const int m = wg / cgs, c = (wg - m * cgs) * 32 + (threadIdx.x & 31);
    if (c >= nc) return;
    const C* xi = (const C*)E.xi + (size_t)m * Sx;
    const C* in = (const C*)E.Vc + c;
    C* fh = (C*)E.Fh + (size_t)m * Sx * nc + c;
    C v = ((const C*)E.V)[(size_t)E.a_if * E.b + m];
    if (E.sc) v = ((const C*)E.sc)[m] * v;
    C y = {0, 0};
    for (int i0 = 0; i0 < Sx; i0 += RB) {
        C a[RB], f[RB];
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            const int i = min(i0 + u, Sx - 1);
            a[u] = xi[i];
            f[u] = v * in[(size_t)i * nc];
        }
#pragma unroll
        for (int u = 0; u < RB; ++u)
            if (i0 + u < Sx) {
                y = a[u] * (f[u] + y);
                fh[(size_t)(i0 + u) * nc] = y;
            }
    }
    C x = y;
    for (int i1 = Sx - 1; i1 > 0; i1 -= RB) {
        C a[RB], yv[RB];
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            const int i = max(i1 - 1 - u, 0);
            a[u] = xi[i];
            yv[u] = fh[(size_t)i * nc];
        }
#pragma unroll
        for (int u = 0; u < RB; ++u) {
            const int i = i1 - 1 - u;
            if (i >= 0) {
                x = yv[u] + a[u] * x;
                fh[(size_t)i * nc] = x;
            }
        }
    }
}

// The extension's two rows at the inner cut, V x^ of the modes' results Fh: one thread per
// (grid column, right-hand side), in the layout of the rows.
template <typename T>
__global__ void __launch_bounds__(256) k_edge_leaf_rows(const EdgeTask* __restrict__ tasks, int Sx, int nc) {
    using C = cplx<T>;
    const EdgeTask& E = tasks[blockIdx.y];
    const int J = Sx * nc, jj = blockIdx.x * 256 + threadIdx.x;
    if (jj >= J) return;
    const C* V0 = (const C*)E.V + (size_t)E.o0 * E.b;
    const C* fh = (const C*)E.Fh + fh_col((size_t)jj, Sx, nc);
    C a0 = {0, 0}, a1 = {0, 0};
#pragma unroll 8
    for (int m = 0; m < E.b; ++m) {
        const C f = fh[(size_t)m * J];
        cfma(a0, V0[m], f);
        cfma(a1, V0[E.b + m], f);
    }
    C* rows = (C*)E.rows;
    rows[jj] = a0;
    rows[(size_t)J + jj] = a1;
}

// Z^H Z of the sketches in FP64 (the stored sketch widens exactly): partial sums over one
// share of the rows per block, 4 x 4 outputs a thread; then the sums in order.
static constexpr int ZG_SPLIT = 16, ZG_T = 16;
template <typename T>
__global__ void __launch_bounds__(256) k_edge_gram(const EdgeTask* __restrict__ tasks, int Sx, int m, c128* part) {
    using C = cplx<T>;
    __shared__ c128 zs[ZG_T][65];
    const C* Z = (const C*)tasks[blockIdx.y].Z;
    const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
    const int xs = (Sx + ZG_SPLIT - 1) / ZG_SPLIT, xa = blockIdx.x * xs, xb = min(Sx, xa + xs);
    c128 acc[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = {0, 0};
    for (int x0 = xa; x0 < xb; x0 += ZG_T) {
        __syncthreads();
        for (int q = tid; q < ZG_T * 64; q += 256) {
            const int x = q >> 6, j = q & 63;
            zs[x][j] = x0 + x < xb && j < m ? cvt<double>(Z[(size_t)(x0 + x) * m + j]) : c128{0, 0};
        }
        __syncthreads();
        // (the matrix is Hermitian: the tiles on and above the diagonal)
        for (int x = 0; x < ZG_T; ++x) {
            c128 a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) { a[u] = zs[x][ti + 16 * u]; b[u] = zs[x][tj + 16 * u]; }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (u <= v && 16 * v < m) cfma_cj(acc[u][v], a[u], b[v]);
        }
    }
    c128* o = part + ((size_t)blockIdx.y * ZG_SPLIT + blockIdx.x) * 4096;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (u <= v) o[(ti + 16 * u) * 64 + tj + 16 * v] = acc[u][v];
}
__global__ void __launch_bounds__(256) k_edge_gram_red(const EdgeTask* __restrict__ tasks, int m, const c128* part) {
    c128* G = tasks[blockIdx.y].Gm;
    const int t = blockIdx.x * 256 + threadIdx.x;
    if (t >= m * m) return;
    const int i = t / m, j = t - i * m;
    const bool low = (i >> 4) > (j >> 4);
    const c128* p = part + (size_t)blockIdx.y * ZG_SPLIT * 4096 + (low ? j * 64 + i : i * 64 + j);
    c128 s = {0, 0};
    for (int k = 0; k < ZG_SPLIT; ++k) s = s + p[(size_t)k * 4096];
    G[t] = low ? conj(s) : s;
}

// Child c's extension W [rows][Sx][r] into its columns of the parent's basis [2r][N] (zero on
// the other child's rows): one block per 32 points and child, transposed in shared memory.
template <typename T>
__global__ void __launch_bounds__(256) k_edge_scatter(const EdgeTask* __restrict__ tasks, int r) {
    using C = cplx<T>;
    __shared__ C tile[32][33];
    const EdgeTask& E = tasks[blockIdx.y];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (size_t p0 = (size_t)blockIdx.x * 32; p0 < E.Np; p0 += (size_t)gridDim.x * 32) {
        __syncthreads();
        for (int y = ty; y < 32; y += 8) {
            const long long q = (long long)(p0 + y) - E.dst0;   // point within the child's rows
            tile[y][tx] = tx < r && q >= 0 && q < E.npts ? ((const C*)E.W)[(size_t)q * r + tx] : C{0, 0};
        }
        __syncthreads();
        if (p0 + tx < E.Np)
            for (int j = ty; j < r; j += 8) ((C*)E.Cout)[(size_t)j * E.Np + p0 + tx] = tile[tx][j];
    }
}

// ---------------------------------------------------------------------- launchers
template <typename T>
void launch_edge_scatter(const EdgeTask* tasks, int nchild, size_t np_max, int r, cudaStream_t s) {
    const int gx = (int)std::min<size_t>((np_max + 31) / 32, 152 * 16);
    k_edge_scatter<T><<<dim3(gx, nchild), 256, 0, s>>>(tasks, r);
    note_launch();
}
template <typename T>
static int edge_lines_per_batch(int Sx) {
    int mg = 8;
    while (mg > 1 && sizeof(cplx<T>) * Sx * (2 * mg + 6) > (size_t)(212 * 1024)) --mg;
    return mg;
}
template <typename T>
bool edge_rows_fit(int Sx) {
    return sizeof(cplx<T>) * Sx * (2 * edge_lines_per_batch<T>(Sx) + 6) <= (size_t)(212 * 1024);
}
size_t edge_pd_elems(int npath, int r, int nc) { return (size_t)EDGE_CH * (npath + 1) * r * nc; }
size_t edge_gram_scratch(int nchild) { return (size_t)nchild * ZG_SPLIT * 4096 * sizeof(c128); }
template <typename T>
void launch_edge_rows(const EdgeTask* tasks, int nchild, int Sx, int nc, int adj, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(attr, k_edge_rows<T>, 212 * 1024);
    const int mg = edge_lines_per_batch<T>(Sx);
    const size_t sm = sizeof(cplx<T>) * (size_t)Sx * (2 * mg + 6);
    k_edge_rows<T><<<dim3(nc, nchild), 256, sm, s>>>(tasks, Sx, nc, adj, mg);
    note_launch();
}
// the path's corrections of nc columns from the leaf rows: y, and (rows_out) the trace rows
template <typename T>
void launch_edge_path(const EdgeTask* tasks, int nchild, int L, int Sx, int nc, int r, const c128* M, OpGeom g, int adj,
                      bool rows_out, cudaStream_t s) {
    g.b = 3;
    k_edge_proj<T><<<dim3(EDGE_CH, nchild, ((CUT_MAXL + 1) * r + 63) / 64), 256, 0, s>>>(tasks, Sx, nc, r, g);
    note_launch();
    k_edge_y<T><<<dim3(nc, nchild), 256, sizeof(c128) * (size_t)(CUT_MAXL + 1) * r, s>>>(tasks, L, nc, r, M);
    note_launch();
    if (!rows_out) return;
    k_edge_out<T><<<dim3((Sx + 31) / 32, adj ? 1 : 2, nchild), 256, 0, s>>>(tasks, Sx, nc, r, adj);
    note_launch();
}
template <typename T>
void launch_edge_basis_lines(const EdgeTask* tasks, int nchild, int b_max, int Sx, int nc, cudaStream_t s) {
    if (!eig_line_major(nc)) {
        k_edge_chains<T><<<dim3((b_max * ((nc + 31) / 32) + 1) / 2, nchild), 64, 0, s>>>(tasks, Sx, nc);
    } else {
        static std::atomic<unsigned long long> attr{0};
        smem_limit_once(attr, k_edge_lines<T>, 200 * 1024);
        const size_t per = 2 * sizeof(cplx<T>) * (size_t)Sx;
        const int wpb = (int)std::max<size_t>(1, std::min<size_t>(8, (200u << 10) / per));
        k_edge_lines<T><<<dim3((b_max * nc + wpb - 1) / wpb, nchild), 256, per * wpb, s>>>(tasks, Sx, nc, wpb);
    }
    note_launch();
}
template <typename T>
void launch_edge_leaf_rows(const EdgeTask* tasks, int nchild, int Sx, int nc, cudaStream_t s) {
    k_edge_leaf_rows<T><<<dim3((Sx * nc + 255) / 256, nchild), 256, 0, s>>>(tasks, Sx, nc);
    note_launch();
}
template <typename T>
void launch_edge_gram(const EdgeTask* tasks, int nchild, int Sx, int m, c128* part, cudaStream_t s) {
    k_edge_gram<T><<<dim3(ZG_SPLIT, nchild), 256, 0, s>>>(tasks, Sx, m, part);
    note_launch();
    k_edge_gram_red<<<dim3((m * m + 255) / 256, nchild), 256, 0, s>>>(tasks, m, part);
    note_launch();
}
#define HH_EDGE_INST(T)                                                                                               \
    template bool edge_rows_fit<T>(int);                                                                              \
    template void launch_edge_rows<T>(const EdgeTask*, int, int, int, int, cudaStream_t);                             \
    template void launch_edge_path<T>(const EdgeTask*, int, int, int, int, int, const c128*, OpGeom, int, bool,       \
                                      cudaStream_t);                                                                  \
    template void launch_edge_basis_lines<T>(const EdgeTask*, int, int, int, int, cudaStream_t);                      \
    template void launch_edge_gram<T>(const EdgeTask*, int, int, int, c128*, cudaStream_t);                           \
    template void launch_edge_leaf_rows<T>(const EdgeTask*, int, int, int, cudaStream_t);                             \
    template void launch_edge_scatter<T>(const EdgeTask*, int, size_t, int, cudaStream_t);
HH_EDGE_INST(float)
HH_EDGE_INST(double)

}  // namespace hh
