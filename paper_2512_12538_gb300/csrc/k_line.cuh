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


// The same recursions with the products of each lane's coefficients, which depend on xi
// alone, given (line_products): 20 multiply-adds an element instead of 28.  Lane chunks are of odd
// length, so that the lanes' strided shared-memory accesses fall in distinct banks.
template <typename T>
__device__ __forceinline__ void line_products(const cplx<T>* as, int Sx, int lane, cplx<T>& pf, cplx<T>& pb) {
    using C = cplx<T>;
    const int L = ((Sx + 31) / 32) | 1, s = lane * L, e = min(Sx, s + L);
    C a = {1, 0}, b = {1, 0};
    for (int i = s; i < e; ++i) {
        a = as[i] * a;
        b = (i == Sx - 1 ? C{0, 0} : as[i]) * b;
    }
    pf = a;
    pb = b;
}
template <typename T>
__device__ __forceinline__ void line_solve(const cplx<T>* as, cplx<T>* fs, int Sx, int lane, cplx<T> pf, cplx<T> pb) {
    using C = cplx<T>;
    const int L = ((Sx + 31) / 32) | 1;
    const int s = lane * L, e = min(Sx, s + L);
    C A = pf, B = {0, 0};
    for (int i = s; i < e; ++i) B = as[i] * (B + fs[i]);
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
    // backward over the lane's own chunk
    A = pb;
    B = {0, 0};
    for (int i = e - 1; i >= s; --i) B = i == Sx - 1 ? fs[i] : as[i] * B + fs[i];
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
        x = i == Sx - 1 ? fs[i] : fs[i] + as[i] * x;
        fs[i] = x;
    }
    __syncwarp();
}

}  // namespace hh
