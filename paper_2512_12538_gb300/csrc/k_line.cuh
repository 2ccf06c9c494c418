// k_line.cuh -- the two scalar recursions of one line of a leaf sweep, by one warp.
#pragma once
#include "hh_core.cuh"

namespace hh {

// Both recursions are affine, y_i = xi_i y_{i-1} + xi_i f_i and
// x_i = xi_i x_{i+1} + y_i (with x_{n-1} = y_{n-1}), so each lane composes the maps of a
// contiguous chunk of the line, a warp scan (shuffles) composes the chunks, and each lane
// then replays its chunk from its entering value.
template <typename T>
__device__ __forceinline__ void affine_shfl(cplx<T>& A, cplx<T>& B, int d, bool up, cplx<T>& A2, cplx<T>& B2) {
    if (up) {
        A2.re = __shfl_up_sync(0xffffffffu, A.re, d); A2.im = __shfl_up_sync(0xffffffffu, A.im, d);
        B2.re = __shfl_up_sync(0xffffffffu, B.re, d); B2.im = __shfl_up_sync(0xffffffffu, B.im, d);
    } else {
        A2.re = __shfl_down_sync(0xffffffffu, A.re, d); A2.im = __shfl_down_sync(0xffffffffu, A.im, d);
        B2.re = __shfl_down_sync(0xffffffffu, B.re, d); B2.im = __shfl_down_sync(0xffffffffu, B.im, d);
    }
}

// Both recursions of one line, in place: on entry fs = f^ (Sx values) and as = xi; on
// exit fs = x^.  One warp; lane l owns the contiguous chunk [l L, (l + 1) L).
template <typename T>
__device__ __forceinline__ void warp_line_solve(const cplx<T>* as, cplx<T>* fs, int Sx, int lane) {
    using C = cplx<T>;
    const int L = (Sx + 31) / 32;
    const int s = lane * L, e = min(Sx, s + L);
    // forward: y_i = a_i (y_{i-1} + f_i)
    C A = {1, 0}, B = {0, 0};
    for (int i = s; i < e; ++i) { A = as[i] * A; B = as[i] * (B + fs[i]); }
    for (int d = 1; d < 32; d <<= 1) {
        C A2, B2;
        affine_shfl(A, B, d, true, A2, B2);
        if (lane >= d) { B = A * B2 + B; A = A * A2; }
    }
    C y;
    y.re = __shfl_up_sync(0xffffffffu, B.re, 1);
    y.im = __shfl_up_sync(0xffffffffu, B.im, 1);
    if (lane == 0) y = {0, 0};
    for (int i = s; i < e; ++i) { y = as[i] * (fs[i] + y); fs[i] = y; }
    __syncwarp();
    // backward: x_i = y_i + a'_i x_{i+1}, a'_{n-1} = 0
    A = {1, 0};
    B = {0, 0};
    for (int i = e - 1; i >= s; --i) {
        const C ap = (i == Sx - 1) ? C{0, 0} : as[i];
        B = ap * B + fs[i];
        A = ap * A;
    }
    for (int d = 1; d < 32; d <<= 1) {
        C A2, B2;
        affine_shfl(A, B, d, false, A2, B2);
        if (lane + d < 32) { B = A * B2 + B; A = A * A2; }
    }
    C x;
    x.re = __shfl_down_sync(0xffffffffu, B.re, 1);
    x.im = __shfl_down_sync(0xffffffffu, B.im, 1);
    if (lane == 31) x = {0, 0};
    for (int i = e - 1; i >= s; --i) {
        const C ap = (i == Sx - 1) ? C{0, 0} : as[i];
        x = fs[i] + ap * x;
        fs[i] = x;
    }
    __syncwarp();
}


// The same recursions with everything that depends on xi alone given (line_scan_init): the
// products of the lanes' coefficients at every stage of the two scans.  12 multiply-adds an
// element and a scan of one value instead of 28 and two.  Lane chunks are of odd length, so
// that the lanes' strided shared-memory accesses fall in distinct banks.
template <typename T>
struct LineScan {
    cplx<T> f[5], b[5];
};
template <typename T>
__device__ __forceinline__ cplx<T> shfl_c(cplx<T> v, int d, bool up) {
    cplx<T> o;
    if (up) { o.re = __shfl_up_sync(0xffffffffu, v.re, d); o.im = __shfl_up_sync(0xffffffffu, v.im, d); }
    else { o.re = __shfl_down_sync(0xffffffffu, v.re, d); o.im = __shfl_down_sync(0xffffffffu, v.im, d); }
    return o;
}
template <typename T>
__device__ __forceinline__ void line_scan_init(const cplx<T>* as, int Sx, int lane, LineScan<T>& sc) {
    using C = cplx<T>;
    const int L = ((Sx + 31) / 32) | 1, s = min(Sx, lane * L), e = min(Sx, s + L);
    C a = {1, 0};
    for (int i = s; i < e; ++i) a = as[i] * a;
    C f = a, b = e == Sx && s < e ? C{0, 0} : a;   // nothing enters from past the line's end
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const int d = 1 << k;
        sc.f[k] = f;
        sc.b[k] = b;
        const C f2 = shfl_c(f, d, true), b2 = shfl_c(b, d, false);
        if (lane >= d) f = f * f2;
        if (lane + d < 32) b = b * b2;
    }
}
template <typename T>
__device__ __forceinline__ void line_solve(const cplx<T>* as, cplx<T>* fs, int Sx, int lane, const LineScan<T>& sc) {
    using C = cplx<T>;
    const int L = ((Sx + 31) / 32) | 1;
    const int s = min(Sx, lane * L), n = min(Sx - s, L);
    const C* a = as + s;
    C* x = fs + s;
    C v = {0, 0};
#pragma unroll 4
    for (int i = 0; i < n; ++i) v = a[i] * (v + x[i]);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const C u = shfl_c(v, 1 << k, true);
        if (lane >= (1 << k)) cfma(v, sc.f[k], u);
    }
    v = shfl_c(v, 1, true);
    if (lane == 0) v = {0, 0};
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
        v = a[i] * (x[i] + v);
        x[i] = v;
    }
    // backward over the lane's own chunk; the recursion starts from zero past the line's end,
    // so the last element needs no case of its own
    v = {0, 0};
#pragma unroll 4
    for (int i = n - 1; i >= 0; --i) {
        C t = x[i];
        cfma(t, a[i], v);
        v = t;
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const C u = shfl_c(v, 1 << k, false);
        if (lane + (1 << k) < 32) cfma(v, sc.b[k], u);
    }
    v = shfl_c(v, 1, false);
    if (lane == 31) v = {0, 0};
#pragma unroll 4
    for (int i = n - 1; i >= 0; --i) {
        C t = x[i];
        cfma(t, a[i], v);
        x[i] = t;
        v = t;
    }
    __syncwarp();
}

}  // namespace hh
