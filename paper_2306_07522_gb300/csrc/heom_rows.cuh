// The matrix-free HEOM apply row by row: one thread forms CW neighbouring elements (r, c0 ..
// c0 + CW - 1) of one ADO's d x d block in one batch column.
//
// Why rows. Everything that is not a multiply-add -- the neighbour entry, its exponent's
// coefficients, the operator's row list -- is the same for the CW elements, so it is decoded
// once for all of them; per element it used to cost more than the arithmetic (FP32: 68 % of
// the issue slots at 5 % of the memory rate; FP64: the pipe 87 % busy, most of it with
// products by 0, 1 and -1 and with integer conversions). The left product O X reads CW
// neighbouring elements of row l (one vector load each at one column); the right product X O
// reads elements of row r, column by column of O. Consecutive threads hold consecutive
// columns of one row (batches) or consecutive rows of one ADO (one column), so every load of a
// warp falls into whole 32-byte sectors, and neighbour blocks are re-read from L1 and L2.
//
// What FP64 saves: GB300 retires two FP64 multiply-adds per clock and SM, so only those that
// change the result are issued: operator values +-1 and entry signs flip sign bits, a
// coefficient's zero half (raising terms with a real operator are imaginary, Pade terms
// beyond the first real or imaginary) is skipped. FP32 keeps the sums over the coefficients'
// real and imaginary parts in packed f32x2 pairs: two instructions per complex multiply-add.
#pragma once

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "heom_ff.cuh"
#include "heom_kernels.cuh"

namespace heom {

// whether a double is not +-0, on the integer pipe
__device__ __forceinline__ bool nonzero(double a) {
    return ((((unsigned)__double2hiint(a)) << 1) | (unsigned)__double2loint(a)) != 0u;
}

// Coefficient of one operator nonzero O: -i m O (raised neighbour), or m a' O with a' = -i a the
// exponent's coefficient (lowered); m is +-1 but for bosonic multiplicities.
template <class R>
__device__ __noinline__ cx<R> term_coef_general(R re, R im, bool raised, int m, cx<R> a) {
    const cx<R> c = raised ? cx<R>{im, -re} : a * cx<R>{re, im};
    return cx<R>{R(m) * c.re, R(m) * c.im};
}
__device__ __forceinline__ double flip(double x, int sign) {
    return __hiloint2double(__double2hiint(x) ^ sign, __double2loint(x));
}
// FP64: O = +-1 and m = +-1 (every fermionic term) flip sign bits; anything else is a call, so that
// its FP64 instructions are not executed speculatively.
__device__ __forceinline__ cx<double> term_coef(const OpRec<double> &o, bool raised, int m, cx<double> a) {
    if (o.kind != OK_UNIT || (m != 1 && m != -1)) return term_coef_general<double>(o.re, o.im, raised, m, a);
    const int sign = (m ^ __double2hiint(o.re)) & (int)0x80000000;
    if (raised) return cx<double>{0.0, __hiloint2double(0x3ff00000 ^ (sign ^ (int)0x80000000), 0)};
    return cx<double>{flip(a.re, sign), flip(a.im, sign)};
}
__device__ __forceinline__ cx<float> term_coef(const OpRec<float> &o, bool raised, int m, cx<float> a) {
    if (o.kind == OK_COMPLEX) return term_coef_general<float>(o.re, o.im, raised, m, a);
    const float f = (float)m * o.re;
    return raised ? cx<float>{0.f, -f} : cx<float>{f * a.re, f * a.im};
}

template <class R>
__device__ __forceinline__ OpRec<R> ld_rec(const OpRec<R> *p) {
    OpRec<R> o;
    if constexpr (sizeof(R) == 4) {
        const int4 t = __ldg(reinterpret_cast<const int4 *>(p));
        o.re = __int_as_float(t.x);
        o.im = __int_as_float(t.y);
        o.idx = t.z;
        o.kind = t.w;
    } else {
        const double2 t = __ldg(reinterpret_cast<const double2 *>(p));
        const int2 k = __ldg(reinterpret_cast<const int2 *>(p) + 2);
        o.re = t.x;
        o.im = t.y;
        o.idx = k.x;
        o.kind = k.y;
    }
    return o;
}

// Times a block of FP64 multiply-adds runs: 0 or 1, opaque to the compiler. A predicated-off
// DFMA still takes its 64 cycles of a sub-partition's FP64 pipe, and the compiler predicates
// short branches, so a half of a coefficient that may be zero is left out by a loop that runs zero
// times (measured on one apply of 396,607 ADOs of 4 x 4: 8.2M FP64 warp instructions with
// predication).
__device__ __forceinline__ int once(bool on) {
    int n = on ? 1 : 0;
    asm volatile("" : "+r"(n));
    return n;
}

// accumulators of N complex output elements
template <class R, int N>
struct RowAcc;
template <int N>
struct RowAcc<double, N> {
    cx<double> s[N];
    __device__ __forceinline__ RowAcc() {
#pragma unroll
        for (int u = 0; u < N; ++u) s[u] = cx<double>{0.0, 0.0};
    }
    // s[U0 + i * ST] += c x[i] for i < M, without the zero halves of c
    template <int U0, int M, int ST>
    __device__ __forceinline__ void mac(cx<double> c, const cx<double> (&x)[M]) {
#pragma unroll 1
        for (int k = once(nonzero(c.re)); k > 0; --k)
#pragma unroll
            for (int i = 0; i < M; ++i) {
                s[U0 + i * ST].re = fma(c.re, x[i].re, s[U0 + i * ST].re);
                s[U0 + i * ST].im = fma(c.re, x[i].im, s[U0 + i * ST].im);
            }
#pragma unroll 1
        for (int k = once(nonzero(c.im)); k > 0; --k)
#pragma unroll
            for (int i = 0; i < M; ++i) {
                s[U0 + i * ST].re = fma(-c.im, x[i].im, s[U0 + i * ST].re);
                s[U0 + i * ST].im = fma(c.im, x[i].re, s[U0 + i * ST].im);
            }
    }
    __device__ __forceinline__ cx<double> value(int u) const { return s[u]; }
};
template <int N>
struct RowAcc<float, N> {
    float2 a[N], b[N];  // sums of c.re (x.re, x.im) and of c.im (x.re, x.im)
    __device__ __forceinline__ RowAcc() {
#pragma unroll
        for (int u = 0; u < N; ++u) a[u] = b[u] = make_float2(0.f, 0.f);
    }
    template <int U0, int M, int ST>
    __device__ __forceinline__ void mac(cx<float> c, const cx<float> (&x)[M]) {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const float2 xv = make_float2(x[i].re, x[i].im);
            a[U0 + i * ST] = f2_fma(make_float2(c.re, c.re), xv, a[U0 + i * ST]);
            b[U0 + i * ST] = f2_fma(make_float2(c.im, c.im), xv, b[U0 + i * ST]);
        }
    }
    __device__ __forceinline__ cx<float> value(int u) const {
        return cx<float>{a[u].x - b[u].y, a[u].y + b[u].x};
    }
};
// compile-time loop f(integral_constant<int, 0 .. N-1>)
template <int N, class F, int I = 0>
__device__ __forceinline__ void static_for(F &&f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<N, F, I + 1>(static_cast<F &&>(f));
    }
}


// CW neighbouring elements at p, stride B; VEC: B == 1, CW even and p 16-byte aligned
template <class R, int CW, bool VEC>
__device__ __forceinline__ void ld_row(const cx<R> *__restrict__ p, int64_t B, cx<R> (&x)[CW]) {
    if constexpr (VEC && sizeof(R) == 4 && CW % 2 == 0) {
#pragma unroll
        for (int u = 0; u < CW; u += 2) {
            const float4 t = __ldg(reinterpret_cast<const float4 *>(p + u));
            x[u] = cx<R>{t.x, t.y};
            x[u + 1] = cx<R>{t.z, t.w};
        }
    } else {
#pragma unroll
        for (int u = 0; u < CW; ++u) x[u] = ldc(p + (VEC ? (int64_t)u : u * B));
    }
}

template <class R, int CW, bool VEC>
__device__ __forceinline__ void st_row(cx<R> *p, int64_t B, const cx<R> (&y)[CW]) {
    if constexpr (VEC && sizeof(R) == 4 && CW % 2 == 0) {
#pragma unroll
        for (int u = 0; u < CW; u += 2)
            *reinterpret_cast<float4 *>(p + u) = make_float4(y[u].re, y[u].im, y[u + 1].re, y[u + 1].im);
    } else {
#pragma unroll
        for (int u = 0; u < CW; ++u) p[VEC ? (int64_t)u : u * B] = y[u];
    }
}

// y[u] = (M X)[n][r][c0 + u][b], x0[u] = X[n][r][c0 + u][b] (Eq. HEOM). Term order per element:
// damping with the element's own system term, the other system terms, then every neighbour
// entry (left products before right ones). The caller leaves out ADOs beyond the truncation of
// the column's parameter set (heom_set_truncation: held at zero); neighbours beyond it are not
// read here, so this is the apply of that set's own, shallower hierarchy, whose couplings into
// the dropped tiers do not exist.
template <class R, int CW>
__device__ __forceinline__ void apply_rows(const DevView<R> &v, const cx<R> *__restrict__ X,
                                           int64_t n, int r, int c0, int64_t b, int64_t B, int set,
                                           cx<R> (&x0)[CW], cx<R> (&y)[CW]) {
    const int d = v.d, d2 = v.d2, ns = v.n_sets;
    const cx<R> *Xn = X + n * d2 * B + b;
    const int e0 = r * d + c0;
    ld_row<R, CW, false>(Xn + e0 * B, B, x0);
    RowAcc<R, CW> acc;
    {
        const cx<R> dmp = ldc(v.damp + n * ns + set);
        static_for<CW>([&](auto U) {
            constexpr int u = U.value;
            cx<R> own{-dmp.re, -dmp.im};
            for (int j = __ldg(v.s_ptr + e0 + u), j1 = __ldg(v.s_ptr + e0 + u + 1); j < j1; ++j) {
                const cx<R> cf = ldc(v.s_val + (int64_t)j * ns + set);
                const int src = __ldg(v.s_src + j);
                const cx<R> x[1] = {ldc(Xn + src * B)};
                if (src == e0 + u) own = own + cf;
                else acc.template mac<u, 1, 1>(cf, x);
            }
            const cx<R> x[1] = {x0[u]};
            acc.template mac<u, 1, 1>(own, x);
        });
    }
    const Kept kept(v, set);
    const int t1 = __ldg(v.row_ptr + n + 1);
    for (int t = __ldg(v.row_ptr + n); t < t1; ++t) {
        const int4 raw = __ldg(reinterpret_cast<const int4 *>(v.ent) + t);
        const int nb = raw.x;
        if (!kept(nb)) continue;  // beyond the set's tiers: not in its hierarchy
        const bool raised = (int16_t)(raw.z & 0xffff) > 0;
        const int ml = (int)(int16_t)(raw.z >> 16), mr = (int)(int16_t)(raw.w & 0xffff);
        const cx<R> *Xb = X + (int64_t)nb * d2 * B + b;
        cx<R> al{R(0), R(0)}, ar{R(0), R(0)};
        if (!raised) {
            const int64_t pk = (int64_t)(raw.y >> 16) * ns + set;
            al = mul_mi(ldc(v.coefL + pk));
            ar = mul_mi(ldc(v.coefR + pk));
        }
        const int base = (int)(int16_t)(raw.y & 0xffff) * (d + 1);
        for (int j = __ldg(v.op_rptr + base + r), j1 = __ldg(v.op_rptr + base + r + 1); j < j1; ++j) {
            const OpRec<R> o = ld_rec(v.op_rrec + j);
            const cx<R> cf = term_coef(o, raised, ml, al);
            cx<R> x[CW];
            ld_row<R, CW, false>(Xb + (o.idx * d + c0) * B, B, x);
            acc.template mac<0, CW, 1>(cf, x);
        }
        int j0 = __ldg(v.op_cptr + base + c0);
        static_for<CW>([&](auto U) {
            constexpr int u = U.value;
            const int j1 = __ldg(v.op_cptr + base + c0 + u + 1);
            for (; j0 < j1; ++j0) {
                const OpRec<R> o = ld_rec(v.op_crec + j0);
                const cx<R> x[1] = {ldc(Xb + (r * d + o.idx) * B)};
                acc.template mac<u, 1, 1>(term_coef(o, raised, mr, ar), x);
            }
        });
    }
#pragma unroll
    for (int u = 0; u < CW; ++u) y[u] = acc.value(u);
}

// rows beyond a set's truncation: a zero apply; x0 is the input (null: not needed)
template <class R, int CW>
__device__ __forceinline__ void zero_rows(const cx<R> *x, int64_t B, cx<R> (&x0)[CW], cx<R> (&y)[CW]) {
#pragma unroll
    for (int u = 0; u < CW; ++u) {
        y[u] = cx<R>{R(0), R(0)};
        x0[u] = x ? x[u * B] : cx<R>{R(0), R(0)};
    }
}
// y += shift x0, and the trace augmentation of the (0, (0, 0)) equation; e0 = first element
template <class R, int CW>
__device__ __forceinline__ void apply_mods(const ApplyMods<R> &mods, const DevView<R> &v, const cx<R> *__restrict__ X,
                                           int64_t n, int e0, int64_t b, int64_t B, const cx<R> (&x0)[CW],
                                           cx<R> (&y)[CW]) {
    if (mods.shift) {
        const cx<R> sh = mods.shift[b];
#pragma unroll
        for (int u = 0; u < CW; ++u) fma_to(y[u], sh, x0[u]);
    }
    if (mods.aug != R(0) && n == 0 && e0 == 0) {
        cx<R> tr{R(0), R(0)};
        for (int k = 0; k < v.d; ++k) tr = tr + X[(int64_t)(k * v.d + k) * B + b];
        y[0] = y[0] + mods.aug * tr;
    }
}

// Run q of CW elements of a vector. 32-bit arithmetic where the launch allows it (a 64-bit
// division costs as much as a dozen multiply-adds).
struct RowPos {
    int64_t n;
    int r, c0;
};
template <int CW>
__device__ __forceinline__ RowPos row_of(int64_t q, int d, bool small) {
    const int per = d / CW, pa = d * per;  // runs per row, per ADO
    RowPos p;
    int rem;
    if (small) {
        const uint32_t n = (uint32_t)q / (uint32_t)pa;
        p.n = n;
        rem = (int)((uint32_t)q - n * (uint32_t)pa);
    } else {
        p.n = q / pa;
        rem = (int)(q - p.n * pa);
    }
    p.r = rem / per;
    p.c0 = (rem - p.r * per) * CW;
    return p;
}
// Elements per thread: a run of four (two) where d allows it and the launch still gives every
// SM about eight warps, else one (small hierarchies are latency-bound and want the threads).
constexpr double kRowFill = 152.0 * 256.0;
inline int row_width(int64_t N, int d, int64_t B) {
    const int cw = d % 4 == 0 ? 4 : d % 2 == 0 ? 2 : 1;
    return (double)N * d * d * (double)B / cw >= kRowFill ? cw : 1;
}
// Whether single-column launches can use 16-byte loads and stores on these buffers.
template <class R>
inline bool row_vec(int64_t B, const void *a, const void *b, const void *c = nullptr, const void *e = nullptr) {
    return B == 1 && (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)e) & 15) == 0;
}
// Flat launch over `total` threads. Small launches use blocks of 64: the ADOs of the lowest tiers
// have an entry for every exponent and stand first, so large blocks would gather them on a few
// SMs.
inline Geom flat_geom(int64_t total) {
    const int bd = total >= 152 * 2048 ? 256 : 64;
    Geom g;
    g.block = dim3(bd, 1, 1);
    g.grid = dim3((unsigned)std::min<int64_t>(std::max<int64_t>((total + bd - 1) / bd, 1), 1 << 30), 1, 1);
    return g;
}

}  // namespace heom
