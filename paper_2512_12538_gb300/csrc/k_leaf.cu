// k_leaf.cu -- leaf subdomain solves A~_leaf^{-1} v (the subdomain solves of Eq. (2),
// the sketches and the basis extension of Sec. 2).
//
// 2D leaf = band of b rows x Sx columns.  Ordered column by column (block index i
// along x), A~_leaf is block tridiagonal with b x b blocks:
//     D_i  (tridiagonal: the y-coupling inside column i, plus the diagonal terms),
//     L_i = U_{i-1} = -W (W = diag of the row weights w_a: 1/2 on the band edges).
// Factorisation (Schur recursion) from both ends towards the middle column m, two chains of
// half the length that run side by side: S_0 = D_0, S_i = D_i - W X_{i-1} W left of m (the
// mirror image right of it), S_m = D_m - W X_{m-1} W - W X_{m+1} W; the kernels store
// X_i = S_i^{-1} (dense, explicit inverse by Gauss-Jordan with partial pivoting).
// Solve: inwards   y_i = X_i (f_i + W y_{i-1}) (right of m: W y_{i+1}),
//                  x_m = X_m (f_m + W y_{m-1} + W y_{m+1});
//        outwards  x_i = y_i + X_i W x_{i+1}   (right of m: W x_{i-1}).
// 1D leaf (Sx = 1): the same recursion with 1 x 1 blocks along the band's rows.
#include <algorithm>
#include <atomic>

#include <cooperative_groups.h>

#include "k_line.cuh"
#include "kernels.h"

namespace hh {

int leaf_ldx(int b, int elem_bytes) {
    // every row of a stored X_i is a multiple of 16 bytes (bulk-copy granularity)
    const int per16 = 16 / elem_bytes;      // elements per 16 bytes: 2 (c64) or 1 (c128)
    return (b + per16 - 1) / per16 * per16;
}

static constexpr uint32_t WAIT_LIMIT = 1u << 21;   // bounded mbarrier polls (~0.1-0.3 s)
static constexpr int MAXP = 4;                       // row pieces per step in the sweep
static constexpr int SW_SLOTS = 12;                  // pieces in flight in the sweep, at most
static constexpr int SW_SMEM = 220 * 1024;           // shared memory of a sweep block, at most

// ------------------------------------------------------------- factorisation (2D)
template <typename T>
__device__ void gj_invert(cplx<T>* M, int ld, int b, cplx<T>* col, cplx<T>* row, int* perm, int* err) {
    __shared__ int s_piv;
    __shared__ cplx<T> s_pv, s_akk;
    for (int k = 0; k < b; ++k) {
        if (threadIdx.x < 32) {
            T best = (T)-1;
            int bi = k;
            for (int r = k + threadIdx.x; r < b; r += 32) {
                const T a = abs2(M[r * ld + k]);
                if (a > best) { best = a; bi = r; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const T ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (threadIdx.x == 0) {
                s_piv = bi;
                perm[k] = bi;
                s_pv = M[bi * ld + k];
                s_akk = M[k * ld + k];
                if (!(best > (T)0) || !isfinite(best)) {
                    atomicExch(err, DEV_BREAKDOWN);
                    s_pv = cplx<T>{(T)1, (T)0};
                }
            }
        }
        __syncthreads();
        const int p = s_piv;
        const cplx<T> pv = s_pv, ip = cinv(pv);
        for (int t = threadIdx.x; t < b; t += blockDim.x) {
            col[t] = (t == k) ? pv : (t == p ? s_akk : M[t * ld + k]);
            const cplx<T> rp = M[p * ld + t];
            if (p != k) { M[p * ld + t] = M[k * ld + t]; M[k * ld + t] = rp; }
            row[t] = rp * ip;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
            const int r = e / b, c = e - r * b;
            cplx<T>& m = M[r * ld + c];
            if (r == k) {
                m = (c == k) ? ip : row[c];
            } else {
                const cplx<T> f = col[r];
                m = (c == k) ? -(f * ip) : m - f * row[c];
            }
        }
        __syncthreads();
    }
    // unscramble columns in reverse pivot order; one thread per row, in place
    for (int r = threadIdx.x; r < b; r += blockDim.x) {
        for (int k = b - 1; k >= 0; --k) {
            const int p = perm[k];
            if (p != k) {
                const cplx<T> t = M[r * ld + k];
                M[r * ld + k] = M[r * ld + p];
                M[r * ld + p] = t;
            }
        }
    }
    __syncthreads();
}

// One of the two chains' columns in order: column t of side 0 (left) or 1 (right); a chain
// has chain_len columns, the middle one belongs to neither.
__device__ __forceinline__ int chain_mid(int Sx) { return Sx / 2; }
__device__ __forceinline__ int chain_len(int Sx, int side) { return side ? Sx - 1 - Sx / 2 : Sx / 2; }
__device__ __forceinline__ int chain_col(int Sx, int side, int t) { return side ? Sx - 1 - t : t; }

// Entry (r, c) of S_i without the neighbour columns' terms.
template <typename T>
__device__ __forceinline__ cplx<T> block_entry(int r, int c, int i, const OpGeom& g, T wi) {
    if (r == c) {
        const c128 d = op_diag(r, i, g);
        return {(T)d.re, (T)d.im};
    }
    if (r - c == 1 || c - r == 1) return {-wi, (T)0};
    return {(T)0, (T)0};
}

// The bands too tall for k_factor2d_reg: the block in shared memory.  mid: the middle column,
// from the stored inverses of its neighbours; else blockIdx.y is the chain.
template <typename T>
__global__ void __launch_bounds__(256) k_factor2d(const LeafTask* __restrict__ tasks, int Sx, double kh, int mid,
                                                  int* err) {
    const LeafTask tk = tasks[blockIdx.x];
    const int b = tk.b, ldx = tk.ldx, side = blockIdx.y;
    cplx<T>* X = (cplx<T>*)tk.X;
    extern __shared__ __align__(16) unsigned char smf[];
    cplx<T>* M = (cplx<T>*)smf;      // b x b, leading dimension b
    cplx<T>* col = M + b * b;
    cplx<T>* row = col + b;
    int* perm = (int*)(row + b);
    const OpGeom g{b, Sx, kh, tk.khr};
    const size_t step = (size_t)b * ldx;
    const int n = mid ? 1 : chain_len(Sx, side);
    for (int t = 0; t < n; ++t) {
        const int i = mid ? chain_mid(Sx) : chain_col(Sx, side, t);
        // built in place over the previous column's inverse
        const T wi = (T)wcol(i, Sx);
        for (int e = threadIdx.x; e < b * b; e += blockDim.x) {
            const int r = e / b, c = e - r * b;
            cplx<T> q = {0, 0};
            if (mid) {
                q = X[(size_t)(i - 1) * step + (size_t)r * ldx + c];
                if (i + 1 < Sx) q = q + X[(size_t)(i + 1) * step + (size_t)r * ldx + c];
            } else if (t > 0) {
                q = M[e];
            }
            M[e] = (-(T)(wrow(r, b) * wrow(c, b))) * q + block_entry<T>(r, c, i, g, wi);
        }
        __syncthreads();
        gj_invert(M, b, b, col, row, perm, err);
        cplx<T>* Xi = X + (size_t)i * step;
        for (int e = threadIdx.x; e < b * ldx; e += blockDim.x) {
            const int r = e / ldx, c = e - r * ldx;
            Xi[e] = c < b ? M[r * b + c] : cplx<T>{0, 0};
        }
        __syncthreads();
    }
}

// The same with the block in registers: lane and slot give a thread's rows (lane + 32 rs),
// warp and slot its columns (warp + NW cs).  Rows are not exchanged: a pivot row is marked,
// column k of the tableau ends up as the column of the pivot row p_k, and the store puts
// entry (p_k, c) at (k, p_c).  The chain of pivots bounds it (b columns x Sx / 2 blocks, each
// pivot waiting for the one before): a pivot costs one barrier, its search stays in the
// warp that owns the column (by the high word of |a|^2: within 1e-6 of the largest), and the pivot
// row's entries come by shuffles.  4 bands of 37 rows
// x 129 columns in complex64: 7.4 ms with the block in shared memory and one chain, 1.45 ms here.
template <typename T> __device__ __forceinline__ unsigned pivot_key(T a) {
    if constexpr (sizeof(T) == 8) return (unsigned)__double2hiint(a) + 1u;
    else return __float_as_uint(a) + 1u;
}
template <typename T, int RS, int NW>
__global__ void __launch_bounds__(NW * 32, 1) k_factor2d_reg(const LeafTask* __restrict__ tasks, int Sx, double kh,
                                                             int mid, int* err) {
    using C = cplx<T>;
    constexpr int CS = (RS * 32 + NW - 1) / NW;
    __shared__ C s_col[2][RS * 32];
    __shared__ C s_ip[2];
    __shared__ int s_p[RS * 32];
    extern __shared__ __align__(16) unsigned char smf[];
    C* sx = (C*)smf;                            // [b][b | 1]: the finished inverse
    const LeafTask tk = tasks[blockIdx.x];
    const int b = tk.b, ldx = tk.ldx, ld = b | 1, side = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    C* X = (C*)tk.X;
    const OpGeom g{b, Sx, kh, tk.khr};
    const size_t step = (size_t)b * ldx;
    const int n = mid ? 1 : chain_len(Sx, side);
    C m[RS][CS];
    for (int t = 0; t < n; ++t) {
        const int i = mid ? chain_mid(Sx) : chain_col(Sx, side, t);
        const T wi = (T)wcol(i, Sx);
        unsigned used = 0;                      // this lane's rows that have been pivots
        int kk[RS];                             // and for which column
#pragma unroll
        for (int rs = 0; rs < RS; ++rs) {
            const int r = lane + 32 * rs;
            kk[rs] = 0;
            if (r >= b) used |= 1u << rs;
#pragma unroll
            for (int cs = 0; cs < CS; ++cs) {
                const int c = warp + NW * cs;
                m[rs][cs] = C{0, 0};
                if (r >= b || c >= b) continue;
                C q = {0, 0};
                if (mid) {
                    q = X[(size_t)(i - 1) * step + (size_t)r * ldx + c];
                    if (i + 1 < Sx) q = q + X[(size_t)(i + 1) * step + (size_t)r * ldx + c];
                } else if (t > 0) {
                    q = sx[r * ld + c];
                }
                m[rs][cs] = (-(T)(wrow(r, b) * wrow(c, b))) * q + block_entry<T>(r, c, i, g, wi);
            }
        }
#pragma unroll
        for (int cs = 0; cs < CS; ++cs)
            for (int w = 0; w < NW; ++w) {
                const int k = cs * NW + w;
                if (k >= b) break;
                const int bf = k & 1;
                if (warp == w) {
                    unsigned key = 0;
                    int br = lane;
                    C best = {(T)1, (T)0};
#pragma unroll
                    for (int rs = 0; rs < RS; ++rs) {
                        s_col[bf][lane + 32 * rs] = m[rs][cs];
                        const unsigned a = (used >> rs & 1) ? 0u : pivot_key<T>(abs2(m[rs][cs]));
                        if (a > key) { key = a; br = lane + 32 * rs; best = m[rs][cs]; }
                    }
                    const unsigned kmax = __reduce_max_sync(0xffffffffu, key);
                    const T a2 = abs2(best);
                    const bool bad = !(a2 > (T)0) || !isfinite(a2);
                    if (bad) best = C{(T)1, (T)0};
                    const C ip = cinv(best);
                    if (lane == __ffs(__ballot_sync(0xffffffffu, key == kmax)) - 1) {
                        s_p[k] = br;
                        s_ip[bf] = ip;
                        if (bad) atomicExch(err, DEV_BREAKDOWN);
                    }
                }
                __syncthreads();
                const int p = s_p[k], pl = p & 31, ps = p >> 5;
                const C ip = s_ip[bf];
                C f[RS], fi[RS];
#pragma unroll
                for (int rs = 0; rs < RS; ++rs) {
                    f[rs] = s_col[bf][lane + 32 * rs];
                    fi[rs] = -(f[rs] * ip);
                    if (ps == rs && lane == pl) { used |= 1u << rs; kk[rs] = k; fi[rs] = ip; }
                }
#pragma unroll
                for (int c2 = 0; c2 < CS; ++c2) {
                    if (warp + NW * c2 >= b) break;
                    C v = m[0][c2];
#pragma unroll
                    for (int rs = 1; rs < RS; ++rs)
                        if (ps == rs) v = m[rs][c2];
                    v.re = __shfl_sync(0xffffffffu, v.re, pl);
                    v.im = __shfl_sync(0xffffffffu, v.im, pl);
                    v = v * ip;
                    const bool own = c2 == cs && warp == w;
#pragma unroll
                    for (int rs = 0; rs < RS; ++rs) {
                        const bool pr = ps == rs && lane == pl;
                        m[rs][c2] = own ? fi[rs] : pr ? v : m[rs][c2] - f[rs] * v;
                    }
                }
            }
#pragma unroll
        for (int cs = 0; cs < CS; ++cs) {
            const int c = warp + NW * cs;
            const int pc = c < b ? s_p[c] : 0;
#pragma unroll
            for (int rs = 0; rs < RS; ++rs)
                if (lane + 32 * rs < b && c < b) sx[kk[rs] * ld + pc] = m[rs][cs];
        }
        __syncthreads();
        C* Xi = X + (size_t)i * step;
        for (int r = warp; r < b; r += NW)
            for (int c = lane; c < ldx; c += 32) Xi[(size_t)r * ldx + c] = c < b ? sx[r * ld + c] : C{0, 0};
    }
}

// ---------------------------------------------------------- factorisation (1D)
template <typename T>
__global__ void k_factor1d(const LeafTask* __restrict__ tasks, int ntasks, double kh, int* err) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntasks) return;
    const LeafTask tk = tasks[t];
    cplx<T>* X = (cplx<T>*)tk.X;
    const OpGeom g{tk.b, 1, kh, tk.khr};
    cplx<double> prev_inv = {0.0, 0.0};
    for (int j = 0; j < tk.b; ++j) {
        // S_j = D_j - (-1) S_{j-1}^{-1} (-1)
        const c128 s = op_diag(j, 0, g) - prev_inv;
        if (!(abs2(s) > 0.0)) atomicExch(err, DEV_BREAKDOWN);
        prev_inv = cinv(s);
        X[j] = cvt<T>(prev_inv);
    }
}

// Tallest band whose b x b inverse and pivot workspace fit one block's shared memory
// (227 KiB) in k_factor2d: 119 rows in complex128, 169 in complex64.
int leaf_block_bmax(int elem_bytes) {
    const long long cap = 227 * 1024;
    int b = 1;
    while ((long long)elem_bytes * ((long long)(b + 1) * (b + 1) + 2 * (b + 1)) + 4ll * (b + 1) <= cap) ++b;
    return b;
}

template <typename T, int RS, int NW>
static void factor_reg(const LeafTask* d_tasks, int ntasks, int b_max, int Sx, double kh, int* err, cudaStream_t s) {
    const size_t sm = sizeof(cplx<T>) * (size_t)b_max * (b_max | 1);
    // (a kernel's limit is set once, to its own maximum: problems are set up from several host
    // threads, and one with shorter bands must not lower another's)
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(attr, k_factor2d_reg<T, RS, NW>, (int)sizeof(cplx<T>) * RS * 32 * (RS * 32 | 1));
    for (int mid = 0; mid < 2; ++mid) {       // the two chains, then the middle column
        k_factor2d_reg<T, RS, NW><<<dim3(ntasks, 2 - mid), NW * 32, sm, s>>>(d_tasks, Sx, kh, mid, err);
        note_launch();
    }
}

template <typename T>
void launch_factor(const LeafTask* d_tasks, int ntasks, int b_max, int Sx, double kh, int* err, cudaStream_t s) {
    if (Sx == 1) {
        k_factor1d<T><<<(ntasks + 31) / 32, 32, 0, s>>>(d_tasks, ntasks, kh, err);
        note_launch();
        return;
    }
    // in registers up to 128 rows (complex64) or 96 (complex128): 32 of a thread's 64 registers
    // (36) hold the block there, and taller blocks would spill
    if (b_max <= 32) factor_reg<T, 1, 8>(d_tasks, ntasks, b_max, Sx, kh, err, s);
    else if (b_max <= 64) factor_reg<T, 2, 16>(d_tasks, ntasks, b_max, Sx, kh, err, s);
    else if (b_max <= 96) factor_reg<T, 3, 32>(d_tasks, ntasks, b_max, Sx, kh, err, s);
    else if (sizeof(T) == 4 && b_max <= 128) {
        if constexpr (sizeof(T) == 4) factor_reg<T, 4, 32>(d_tasks, ntasks, b_max, Sx, kh, err, s);
    } else {
        const size_t sm = sizeof(cplx<T>) * ((size_t)b_max * b_max + 2 * b_max) + sizeof(int) * b_max;
        static std::atomic<unsigned long long> attr{0};
        const int bm = leaf_block_bmax((int)sizeof(cplx<T>));
        smem_limit_once(attr, k_factor2d<T>, (int)sizeof(cplx<T>) * (bm * bm + 2 * bm) + (int)sizeof(int) * bm);
        for (int mid = 0; mid < 2; ++mid) {
            k_factor2d<T><<<dim3(ntasks, 2 - mid), 256, sm, s>>>(d_tasks, Sx, kh, mid, err);
            note_launch();
        }
    }
}

// ------------------------------------------------------------------ sweep (2D)
// One pair of CTAs (a cluster) per (leaf, chunk of NC right-hand sides), one for each chain;
// both form the middle column after an exchange through the cluster's shared memory.  X_i
// pieces (row blocks of a column's inverse; NP of them at most) stream through a ring of
// shared-memory slots by 1D bulk copies (TMA engine) completing on mbarriers; the chain vector
// lives in shared memory.  SW_G lanes split every row's dot product.  The latency of a column
// (the dot products, their reduction, one barrier) bounds it, so nothing else stands on that
// chain: f, y and x pass through registers in groups of SW_G columns, lane g holding
// column g of the group, loaded a group ahead.  4 bands of 37 rows x 129 columns, complex64, one
// right-hand side: 0.61 ms with one chain and loads on it, 0.077 ms here.
static constexpr int SW_G = 8;
// threads of a CTA at most: the rows of which three slots fit shared memory, eight lanes a row
template <typename T, int NP> constexpr int sweep_threads() {
    return sizeof(T) == 4 ? (NP == 1 ? 800 : 576) : (NP == 1 ? 576 : 416);
}
template <typename T, int NC, int NP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(sweep_threads<T, NP>(), 1)
    k_sweep2d(const LeafTask* __restrict__ tasks, int Sx, int nrhs, int nslot, int prow, size_t slot_elems, int* err) {
    using C = cplx<T>;
    constexpr int G = SW_G, VE = 16 / (int)sizeof(C);       // VE: entries of a 16-byte load
    namespace cg = cooperative_groups;
    const LeafTask tk = tasks[blockIdx.y];
    const int b = tk.b, ldx = tk.ldx, side = blockIdx.x & 1;
    const int c0 = (int)(blockIdx.x >> 1) * NC, ncol = min(NC, nrhs - c0);
    const C* X = (const C*)tk.X;
    const C* F = (const C*)tk.F;
    C* W = (C*)tk.W;
    const size_t ldrow = (size_t)Sx * nrhs;   // stride between rows of F / W
    const size_t step = (size_t)b * ldx;
    const int n = chain_len(Sx, side), mid = chain_mid(Sx);

    extern __shared__ __align__(128) unsigned char sms[];
    C* slots = (C*)sms;
    C* vbuf = slots + (size_t)nslot * slot_elems;           // [2][NC][ldx]
    C* xbuf = vbuf + 2 * (size_t)ldx * NC;                  // the other chain's W y, [NC][ldx]
    uint64_t* bars = (uint64_t*)(xbuf + (size_t)ldx * NC);
    const int npiece = (b + prow - 1) / prow;
    const int nsteps = 2 * n + 1;                           // inwards, middle, outwards
    const int total = nsteps * npiece;
    auto step_col = [&](int s) { return s == n ? mid : chain_col(Sx, side, s < n ? s : 2 * n - s); };
    // the producer's place (thread 0): the next piece's step, piece and slot; the consumers'
    // slot and its phase (counted on: a division a piece would stand on the chain)
    int i_s = 0, i_p = 0, i_slot = 0, slot = 0;
    uint32_t parity = 0;
    auto issue = [&] {
        const int r0 = i_p * prow;
        const uint32_t bytes = (uint32_t)(min(prow, b - r0) * ldx * sizeof(C));
        mbar_arrive_expect_tx(&bars[i_slot], bytes);
        bulk_g2s(slots + (size_t)i_slot * slot_elems, X + (size_t)step_col(i_s) * step + (size_t)r0 * ldx, bytes,
                 &bars[i_slot]);
        if (++i_p == npiece) { i_p = 0; ++i_s; }
        if (++i_slot == nslot) i_slot = 0;
    };

    if (threadIdx.x == 0) {
        for (int k = 0; k < nslot; ++k) mbar_init(&bars[k], 1);
        fence_barrier_init();
    }
    // (the padding entries of the vectors stay zero)
    for (int e = threadIdx.x; e < 3 * ldx * NC; e += blockDim.x) vbuf[e] = C{0, 0};
    cg::this_cluster().sync();                              // the other CTA's shared memory exists
    if (threadIdx.x == 0)
        for (int q = 0; q < nslot && q < total; ++q) issue();

    const int lr = threadIdx.x / G, g = threadIdx.x % G;
    auto col_of = [&](int t) { return (size_t)chain_col(Sx, side, t) * nrhs + c0; };
    // a group's entries of this lane: columns t0 + g of the chain (f, or y as written below)
    auto load = [&](const C* src, int t0, C (&v)[NP][NC]) {
        const int t = t0 + g;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const int a = p * prow + lr;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                v[p][c] = lr < prow && a < b && t >= 0 && t < n && c < ncol ? src[a * ldrow + col_of(t) + c] : C{0, 0};
        }
    };
    auto store = [&](int t0, const C (&v)[NP][NC]) {
        const int t = t0 + g;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const int a = p * prow + lr;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (lr < prow && a < b && t < n && c < ncol) W[a * ldrow + col_of(t) + c] = v[p][c];
        }
    };
    auto pick = [&](C v, int t) {                           // lane t of the row's group
        const int src = (threadIdx.x & (31 & ~(G - 1))) + (t & (G - 1));
        return C{__shfl_sync(0xffffffffu, v.re, src), __shfl_sync(0xffffffffu, v.im, src)};
    };
    C in[NP][NC], nx[NP][NC], out[NP][NC], fm[NP][NC];
    load(F, 0, in);
    load(F, G, nx);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const int a = p * prow + lr;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            out[p][c] = C{0, 0};
            // f of the middle column joins the left chain's part
            fm[p][c] = !side && lr < prow && a < b && c < ncol ? F[a * ldrow + (size_t)mid * nrhs + c0 + c] : C{0, 0};
            if (g == 0 && lr < prow && a < b) vbuf[c * ldx + a] = in[p][c];
        }
    }
    __syncthreads();
    int q = 0;
    bool ok = true, bad = false;
    // rows of piece p of step s: X_i v, in every lane of the row
    auto product = [&](int s, int p, C (&acc)[NC]) {
        if (!mbar_wait_bounded(&bars[slot], parity, WAIT_LIMIT)) {
            atomicExch(err, DEV_TIMEOUT);
            bad = true;
        }
        const C* v = vbuf + (size_t)(s & 1) * ldx * NC;
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = C{0, 0};
        if (lr < min(prow, b - p * prow)) {
            const C* xr = slots + (size_t)slot * slot_elems + (size_t)lr * ldx;
            for (int k = g * VE; k < ldx; k += G * VE) {
                struct alignas(16) V { C e[VE]; };
                const V xv = *(const V*)(xr + k);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const V vv = *(const V*)(v + c * ldx + k);
#pragma unroll
                    for (int e = 0; e < VE; ++e) cfma(acc[c], xv.e[e], vv.e[e]);
                }
            }
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                acc[c].re += __shfl_xor_sync(0xffffffffu, acc[c].re, o);
                acc[c].im += __shfl_xor_sync(0xffffffffu, acc[c].im, o);
            }
    };
    // after a piece: its slot is free for the piece nslot further on
    auto turn = [&] {
        if (__syncthreads_or(bad)) return false;
        if (threadIdx.x == 0 && q + nslot < total) issue();
        ++q;
        if (++slot == nslot) { slot = 0; parity ^= 1; }
        return true;
    };
    // inwards; the last column's W y (the left one's with f_m) goes to both CTAs
    C* peer = cg::this_cluster().map_shared_rank(xbuf, side ^ 1);
    for (int t = 0; ok && t < n; ++t) {
        const bool last = t + 1 == n;
        if (((t + 1) & (G - 1)) == 0 && !last) {
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int c = 0; c < NC; ++c) in[p][c] = nx[p][c];
            load(F, t + 1 + G, nx);
        }
        C* vn = vbuf + (size_t)((t + 1) & 1) * ldx * NC;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (!ok || p >= npiece) break;
            C y[NC];
            product(t, p, y);
            const int a = p * prow + lr;
            const T wa = (T)wrow(a, b);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const C fn = pick(in[p][c], t + 1);
                if (g == (t & (G - 1))) out[p][c] = y[c];
                const C nv = wa * y[c] + (last ? fm[p][c] : fn);
                if (g == 0 && lr < prow && a < b) {
                    vn[c * ldx + a] = nv;
                    if (last) peer[c * ldx + a] = nv;
                }
            }
            ok = turn();
        }
        if ((t & (G - 1)) == G - 1 || last) store(t & ~(G - 1), out);
    }
    cg::this_cluster().sync();
    // the middle column, in both CTAs alike
    if (ok) {
        C* v = vbuf + (size_t)(n & 1) * ldx * NC;
        for (int e = threadIdx.x; e < ldx * NC; e += blockDim.x) v[e] = (n > 0 ? v[e] : C{0, 0}) + xbuf[e];
        __syncthreads();
        C* vn = vbuf + (size_t)((n + 1) & 1) * ldx * NC;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (!ok || p >= npiece) break;
            C x[NC];
            product(n, p, x);
            const int a = p * prow + lr;
            if (g == 0 && lr < prow && a < b)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (!side && c < ncol) W[a * ldrow + (size_t)mid * nrhs + c0 + c] = x[c];
                    vn[c * ldx + a] = (T)wrow(a, b) * x[c];
                }
            ok = turn();
        }
    }
    // outwards: y of the group in work is still in `out`
    if (n > 0) load(W, ((n - 1) & ~(G - 1)) - G, nx);
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int c = 0; c < NC; ++c) in[p][c] = out[p][c];
    for (int t = n - 1; ok && t >= 0; --t) {
        const int s = 2 * n - t;
        C* vn = vbuf + (size_t)((s + 1) & 1) * ldx * NC;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (!ok || p >= npiece) break;
            C x[NC];
            product(s, p, x);
            const int a = p * prow + lr;
            const T wa = (T)wrow(a, b);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                x[c] = x[c] + pick(in[p][c], t);
                if (g == (t & (G - 1))) out[p][c] = x[c];
                if (g == 0 && lr < prow && a < b) vn[c * ldx + a] = wa * x[c];
            }
            ok = turn();
        }
        if (ok && (t & (G - 1)) == 0) {
            store(t, out);
#pragma unroll
            for (int p = 0; p < NP; ++p)
#pragma unroll
                for (int c = 0; c < NC; ++c) in[p][c] = nx[p][c];
            load(W, t - 2 * G, nx);
        }
    }
    if (!ok && threadIdx.x == 0) {
        // drain copies still in flight before the CTA's shared memory is released
        for (int k = q; k < total && k < q + nslot; ++k)
            mbar_wait_bounded(&bars[k % nslot], (uint32_t)((k / nslot) & 1), WAIT_LIMIT);
    }
}

// --------------------------------------------------------------------- sweep (1D)
// One block per (leaf, right-hand side).  Both recursions are affine, y_j = X_j (f_j +
// y_{j-1}) and x_j = y_j + X_j x_{j+1}: each thread composes the maps of a contiguous chunk,
// the block scans the chunks' maps, and each thread runs its chunk from its entering value.
// What bounds it is the FP64 multiply-add's latency along a chain: one thread's chain over
// 502 rows took 137 us, the scan 4.
static constexpr int S1_THREADS = 256;
template <typename T>
__device__ __forceinline__ cplx<T> s1_scan(cplx<T> A, cplx<T> B, bool up, cplx<T> (*sw)[2]) {
    // the value entering this thread's chunk: the maps (A, B): v -> A v + B of the threads
    // before it (up) or after it, composed in order and applied to zero
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = 1; d < 32; d <<= 1) {
        cplx<T> A2, B2;
        affine_shfl(A, B, d, up, A2, B2);
        if (up ? lane >= d : lane + d < 32) { B = A * B2 + B; A = A * A2; }
    }
    if (lane == (up ? 31 : 0)) { sw[warp][0] = A; sw[warp][1] = B; }
    cplx<T> Ap, Bp;                          // the map of the lanes before (after) this one
    affine_shfl(A, B, 1, up, Ap, Bp);
    __syncthreads();
    cplx<T> v = {0, 0};                      // entering this warp
    if (up) for (int w = 0; w < warp; ++w) v = sw[w][0] * v + sw[w][1];
    else for (int w = S1_THREADS / 32 - 1; w > warp; --w) v = sw[w][0] * v + sw[w][1];
    __syncthreads();
    if (lane == (up ? 0 : 31)) return v;
    return Ap * v + Bp;
}
template <typename T>
__global__ void __launch_bounds__(S1_THREADS) k_sweep1d(const LeafTask* __restrict__ tasks, int nrhs) {
    using C = cplx<T>;
    __shared__ C sw[S1_THREADS / 32][2];
    const LeafTask tk = tasks[blockIdx.y];
    const int c = blockIdx.x, b = tk.b, n = (b + S1_THREADS - 1) / S1_THREADS;
    const C* X = (const C*)tk.X;
    const C* F = (const C*)tk.F + c;
    C* W = (C*)tk.W + c;
    const int s = min(b, (int)threadIdx.x * n), e = min(b, s + n);
    C A = {1, 0}, B = {0, 0};
    for (int j = s; j < e; ++j) {
        A = X[j] * A;
        B = X[j] * (F[(size_t)j * nrhs] + B);
    }
    C y = s1_scan(A, B, true, sw);
    for (int j = s; j < e; ++j) {
        y = X[j] * (F[(size_t)j * nrhs] + y);
        W[(size_t)j * nrhs] = y;
    }
    A = {1, 0};
    B = {0, 0};
    for (int j = e - 1; j >= s; --j) {
        const C a = j == b - 1 ? C{0, 0} : X[j];
        B = W[(size_t)j * nrhs] + a * B;
        A = a * A;
    }
    C x = s1_scan(A, B, false, sw);
    for (int j = e - 1; j >= s; --j) {
        x = j == b - 1 ? W[(size_t)j * nrhs] : W[(size_t)j * nrhs] + X[j] * x;
        W[(size_t)j * nrhs] = x;
    }
}

template <typename T, int NC, int NP>
static void sweep_go(const LeafTask* d_tasks, int ntasks, int Sx, int nrhs, int nslot, int prow, size_t slot_bytes,
                     size_t sm, int* err, cudaStream_t s) {
    const int threads = ((prow * SW_G + 31) / 32) * 32;
    static std::atomic<unsigned long long> attr{0};
    smem_limit_once(attr, k_sweep2d<T, NC, NP>, SW_SMEM);
    k_sweep2d<T, NC, NP><<<dim3(2 * ((nrhs + NC - 1) / NC), ntasks), threads, sm, s>>>(
        d_tasks, Sx, nrhs, nslot, prow, slot_bytes / sizeof(cplx<T>), err);
    note_launch();
}
template <typename T, int NC>
static void sweep_cfg(const LeafTask* d_tasks, int ntasks, int b_max, int Sx, int nrhs, int* err, cudaStream_t s) {
    const int esz = (int)sizeof(cplx<T>);
    const int ldx = leaf_ldx(b_max, esz);
    const size_t budget = SW_SMEM;
    const size_t vbytes = 3 * (size_t)ldx * NC * esz + 8 * SW_SLOTS + 128;
    int prow = std::min(b_max, 1024 / SW_G), nslot = 3;
    size_t slot_bytes = align_up((size_t)prow * ldx * esz, 128);
    auto over = [&] {
        const int cap = prow == b_max ? sweep_threads<T, 1>() : sweep_threads<T, MAXP>();
        return nslot * slot_bytes + vbytes > budget || prow * SW_G > cap;
    };
    while (over() && prow > 8) {
        prow = (prow + 1) / 2;
        slot_bytes = align_up((size_t)prow * ldx * esz, 128);
    }
    // Halving overshoots on the tallest complex64 bands (143 rows and more: five or six pieces of
    // about 36 rows, where four of 36 to 43 fit): take the largest pieces the kernel needs.  With
    // that every band leaf_block_bmax accepts has a sweep (169 rows: three slots of 57 KB).
    if ((b_max + prow - 1) / prow > MAXP) {
        prow = (b_max + MAXP - 1) / MAXP;
        slot_bytes = align_up((size_t)prow * ldx * esz, 128);
        if (over()) {
            int one = DEV_BADARG;
            cudaMemcpyAsync(err, &one, sizeof(int), cudaMemcpyHostToDevice, s);
            return;
        }
    }
    while ((nslot + 1) * slot_bytes + vbytes <= budget && nslot < SW_SLOTS) ++nslot;
    const size_t sm = nslot * slot_bytes + vbytes;
    const int np = (b_max + prow - 1) / prow;
    if (np == 1) sweep_go<T, NC, 1>(d_tasks, ntasks, Sx, nrhs, nslot, prow, slot_bytes, sm, err, s);
    else sweep_go<T, NC, MAXP>(d_tasks, ntasks, Sx, nrhs, nslot, prow, slot_bytes, sm, err, s);
}

template <typename T>
void launch_sweep(const LeafTask* d_tasks, int ntasks, int b_max, int Sx, int nrhs, int* err, cudaStream_t s) {
    if (Sx == 1) {
        k_sweep1d<T><<<dim3(nrhs, ntasks), S1_THREADS, 0, s>>>(d_tasks, nrhs);
        note_launch();
        return;
    }
    // prow * G threads must fit in one CTA; rows beyond are handled as further pieces
    if (nrhs == 1) sweep_cfg<T, 1>(d_tasks, ntasks, b_max, Sx, nrhs, err, s);
    else sweep_cfg<T, 2>(d_tasks, ntasks, b_max, Sx, nrhs, err, s);
}

template void launch_factor<float>(const LeafTask*, int, int, int, double, int*, cudaStream_t);
template void launch_factor<double>(const LeafTask*, int, int, int, double, int*, cudaStream_t);
template void launch_sweep<float>(const LeafTask*, int, int, int, int, int*, cudaStream_t);
template void launch_sweep<double>(const LeafTask*, int, int, int, int, int*, cudaStream_t);

}  // namespace hh
