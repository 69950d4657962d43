// Dot products that a thread forms over its entries of one column.
#pragma once

#include "heom_ff.cuh"
#include "heom_internal.h"
#include "heom_kernels.cuh"

namespace heom {

// c = sum conj(a) b and n = sum |b|^2. FP64 vectors in FP64; FP32 vectors in FP32 sums of more bits than FP64's
// (Sum3). Those have FP32's exponents only: a product beyond 3.4e38 turns the sums into infinity or NaN; the block's
// sums are then formed again by wide_dots, whose products do not overflow. (Products
// below 2^-101 lose bits and below 2^-149 vanish: the solvers scale their right-hand sides to one, so that is beneath
// 2^-50 of the sums that decide anything.)
template <class R>
struct ColDots;
template <>
struct ColDots<double> {
    double re = 0, im = 0, nn = 0;
    __device__ __forceinline__ void cross(cx<double> a, cx<double> b) {
        re += a.re * b.re + a.im * b.im;
        im += a.re * b.im - a.im * b.re;
    }
    __device__ __forceinline__ void norm(cx<double> b) { nn += norm2(b); }
    __device__ __forceinline__ double c_re() const { return re; }
    __device__ __forceinline__ double c_im() const { return im; }
    __device__ __forceinline__ double n() const { return nn; }
};
template <>
struct ColDots<float> {
    Sum3 c, q;
    __device__ __forceinline__ void cross(cx<float> a, cx<float> b) {
        c.mac(make_float2(a.re, a.re), make_float2(b.re, b.im));
        c.mac(make_float2(a.im, a.im), make_float2(b.im, -b.re));
    }
    __device__ __forceinline__ void norm(cx<float> b) {
        const float2 x = make_float2(b.re, b.im);
        q.mac(x, x);
    }
    __device__ __forceinline__ double c_re() const { return c.x(); }
    __device__ __forceinline__ double c_im() const { return c.y(); }
    __device__ __forceinline__ double n() const { return q.x() + q.y(); }
};
// A block's dot products of one column again in FP64: (w, y) or with conj_y (y, w), and (y, y), over the rows that its
// threads visited: nrun runs of ne rows from each of q, q + step, ... on.
template <class R>
__device__ __forceinline__ void wide_dots(double (&val)[3], const cx<R> *y, const cx<R> *w, int64_t B, int64_t q,
                                          int64_t q_end, int64_t step, int nrun, int ne, int d2, const Kept &kept,
                                          bool conj_y) {
    ColDots<double> wide;
#pragma unroll 1
    for (; q < q_end; q += step)
#pragma unroll 1
        for (int64_t row = q * ne, end = min(q + nrun, q_end) * ne; row < end; ++row) {
            if (!kept(row / d2)) continue;
            const cx<double> yv = cast<double>(y[row * B]), wv = cast<double>(w[row * B]);
            wide.cross(conj_y ? yv : wv, conj_y ? wv : yv);
            wide.norm(yv);
        }
    val[0] = wide.c_re();
    val[1] = wide.c_im();
    val[2] = wide.n();
}

}  // namespace heom
