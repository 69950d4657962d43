// Dot products that a thread forms over its entries of one column.
#pragma once

#include "heom_ff.cuh"
#include "heom_internal.h"

namespace heom {

// c = sum conj(a) b and n = sum |b|^2. FP64 vectors in FP64; FP32 vectors in FP32 sums of more bits than FP64's
// (Sum3). Those have FP32's exponents only: a product beyond 3.4e38 turns the sums into infinity or NaN, which
// overflowed() tells; the caller then forms them again in ColDots<double>, whose products do not overflow. (Products
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
    __device__ __forceinline__ bool overflowed() const { return false; }
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
    // once a product or a sum has overflowed its error term is NaN and stays so
    __device__ __forceinline__ bool overflowed() const {
        return !(isfinite(c.h.x + c.m.x) && isfinite(c.h.y + c.m.y) && isfinite(q.h.x + q.m.x) && isfinite(q.h.y + q.m.y));
    }
};
// the column's values of a thread
struct DotVals {
    double re, im, n;
    template <class R>
    __device__ __forceinline__ explicit DotVals(const ColDots<R> &d) : re(d.c_re()), im(d.c_im()), n(d.n()) {}
};

}  // namespace heom
