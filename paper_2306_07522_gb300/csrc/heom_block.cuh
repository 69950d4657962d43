// The matrix-free HEOM apply for small blocks (d = 2, 4), laid out so that the lanes of a warp
// agree on what they do. The operators of these systems have two to four nonzeros; decoding
// them per output element costs several times the multiply-adds, and lanes that hold different
// elements of different ADOs walk each other's branches (measured on the 56-exponent Anderson
// model: 300 warp instructions per neighbour entry and warp, the FP64 pipe 85 % busy with half
// of its lanes idle). Two layouts avoid that:
//
// * one column (apply_warp): a warp owns 32 ADOs, a lane one whole block, its accumulators in
//   registers. The ADOs are taken in an order in which neighbours use the same operators in
//   the same entries (DevView::perm), so a warp nearly always needs one pass per entry (it
//   makes one pass per distinct operator). Neighbour blocks are copied by the warp together
//   (whole lines, cp.async, kWarpDepth deep) into shared memory, where a lane picks rows and
//   columns of its neighbour by index.
// * many columns (apply_cols): lanes hold neighbouring columns of one ADO (and rows), so the
//   operator is the same for the warp: its nonzeros are tested once, accumulators stay in
//   registers, elements are read straight from global memory, coalesced over the columns.
#pragma once

#include "heom_rows.cuh"
#include "heom_staged.cuh"

namespace heom {

// ---------------------------------------------------------------- one column
constexpr int kWarpDepth = 3;  // neighbour blocks in flight per lane
constexpr int kWarpWarps = 4;  // warps per block

// elements between two lanes' blocks in shared memory (padded by 16 bytes: the same element of
// neighbouring lanes falls into different banks)
template <class R, int D>
__host__ __device__ constexpr int warp_slot() {
    return D * D + 16 / (int)(2 * sizeof(R));
}
template <class R, int D>
__host__ __device__ constexpr size_t warp_smem() {  // ring of one warp
    return (size_t)kWarpDepth * 32 * warp_slot<R, D>() * sizeof(cx<R>);
}

// s = the lane's D x D block of M X for ADO n (n < 0: none, zero); every lane of the warp calls
// this. ring: the warp's shared memory.
template <class R, int D, int W>
__device__ __forceinline__ void apply_warp(const DevView<R> &v, const OpRec<R> *s_ops, cx<R> *ring,
                                           const cx<R> *__restrict__ X, int n, cx<R> (&s)[D * D]) {
    constexpr int D2 = D * D, SL = warp_slot<R, D>(), LPB = D2 * (int)sizeof(cx<R>) / 16, BPI = 32 / LPB;
    const int lane = threadIdx.x & 31;
    RowAcc<R, D2> acc;
    int t0 = 0, cnt = -1;
    if (n >= 0 && !beyond_cap(v, n, 0)) {
        t0 = __ldg(v.row_ptr + n);
        cnt = __ldg(v.row_ptr + n + 1) - t0;
    }
    const int last = __reduce_max_sync(0xffffffffu, cnt);
    const Kept kept(v, 0);
    auto block_of = [&](int i) {  // ADO of the lane's block i (own, then neighbours), -1: none
        if (i > cnt) return -1;
        if (i == 0) return n;
        const int nb = __ldg(reinterpret_cast<const int *>(v.ent) + 4 * (int64_t)(t0 + i - 1));
        return kept(nb) ? nb : -1;
    };
    auto issue = [&](int nb, int i) {  // the warp copies its lanes' blocks line by line
        char *dst = reinterpret_cast<char *>(ring + (i % kWarpDepth) * 32 * SL + (lane / LPB) * SL) + 16 * (lane % LPB);
        const char *src = reinterpret_cast<const char *>(X) + 16 * (lane % LPB);
#pragma unroll
        for (int k = 0; k < LPB; ++k) {
            const int from = __shfl_sync(0xffffffffu, nb, k * BPI + lane / LPB);
            if (from >= 0) stage_copy(dst + (size_t)k * BPI * SL * sizeof(cx<R>), src + (int64_t)from * (D2 * sizeof(cx<R>)), 1);
        }
    };
    __syncwarp();  // the ring is free again
#pragma unroll
    for (int i = 0; i < kWarpDepth - 1; ++i) {
        issue(block_of(i), i);
        stage_commit();
    }
    int nb_next = block_of(kWarpDepth - 1);
    for (int i = 0; i <= last; ++i) {
        int4 raw = make_int4(-1, 0, 0, 0);
        cx<R> al{R(0), R(0)}, ar{R(0), R(0)};
        bool use = i <= cnt, raised = false;
        if (use && i > 0) {
            raw = __ldg(reinterpret_cast<const int4 *>(v.ent) + t0 + i - 1);
            if (v.set_cap) use = block_of(i) >= 0;
            raised = (int16_t)(raw.z & 0xffff) > 0;
            if (!raised) {
                const int k = raw.y >> 16;
                al = mul_mi(ldc(v.coefL + k));
                ar = mul_mi(ldc(v.coefR + k));
            }
        }
        stage_wait<kWarpDepth - 2>();
        __syncwarp();
        issue(nb_next, i + kWarpDepth - 1);  // into the slot of block i - 1, used by every lane
        stage_commit();
        nb_next = block_of(i + kWarpDepth);
        const cx<R> *xs = ring + ((i % kWarpDepth) * 32 + lane) * SL;
        if (i == 0) {
            if (!use) continue;
            const cx<R> dmp = ldc(v.damp + n);
            static_for<D2>([&](auto E) {
                constexpr int e = E.value;
                cx<R> own{-dmp.re, -dmp.im};
                for (int j = __ldg(v.s_ptr + e), j1 = __ldg(v.s_ptr + e + 1); j < j1; ++j) {
                    const cx<R> cf = ldc(v.s_val + j);
                    const int src = __ldg(v.s_src + j);
                    const cx<R> x[1] = {xs[src]};
                    if (src == e) own = own + cf;
                    else acc.template mac<e, 1, 1>(cf, x);
                }
                const cx<R> x[1] = {xs[e]};
                acc.template mac<e, 1, 1>(own, x);
            });
            continue;
        }
        const int ml = (int)(int16_t)(raw.z >> 16), mr = (int)(int16_t)(raw.w & 0xffff);
        const int op = use ? (int)(int16_t)(raw.y & 0xffff) : -1;
        for (unsigned left = __ballot_sync(0xffffffffu, use); left;) {
            const int cur = __shfl_sync(0xffffffffu, op, __ffs(left) - 1);  // one operator of the warp
            const bool mine = op == cur;
            left &= ~__ballot_sync(0xffffffffu, mine);
            if (!mine) continue;
            const OpRec<R> *ol = s_ops + cur * 2 * D * W, *oc = ol + D * W;
            static_for<D>([&](auto K) {  // row k of O X and column k of X O
                constexpr int k = K.value;
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const OpRec<R> o = ol[k * W + w], p = oc[k * W + w];
                    if (o.idx >= 0) {
                        cx<R> x[D];
#pragma unroll
                        for (int c = 0; c < D; ++c) x[c] = xs[o.idx * D + c];
                        acc.template mac<k * D, D, 1>(term_coef(o, raised, ml, al), x);
                    }
                    if (p.idx >= 0) {
                        cx<R> x[D];
#pragma unroll
                        for (int q = 0; q < D; ++q) x[q] = xs[q * D + p.idx];
                        acc.template mac<k, D, D>(term_coef(p, raised, mr, ar), x);
                    }
                }
            });
        }
    }
    stage_wait<0>();
#pragma unroll
    for (int e = 0; e < D2; ++e) s[e] = acc.value(e);
}

// ---------------------------------------------------------------- one column, FP32
// FP32 issues multiply-adds 64 times as fast as FP64, so here decoding and latency decide: a lane
// takes four elements (r, c0 .. c0 + 3) and every step is free of branches. With real operators
// (v.op_real) the lane takes its terms from fixed-width records {offset, value} -- where there is no
// nonzero, value 0 and a neighbour element that is loaded and left out by a predicate; nothing
// depends on which lane holds which operator, so all loads of an entry are in flight together.
// Blocks are read straight from global memory: the lanes of a block share its lines in L1.
// 396,607 ADOs of 4 x 4: 381 us (one thread per element) -> 119 us, bound by L1 wavefronts (75 %);
// a charge-cavity RK4 stage (790 ADOs of 24 x 24): 36 us -> 25 us. Two entries at a time (111
// registers) 154 us, loads predicated off where there is no nonzero 142 us, whole blocks staged
// through shared memory 182 us.

// records [op][side][i][w] as {offset, value}: left records give l d (the row's start), right
// records l, relative to the neighbour's block; missing ones value 0
template <int W>
__device__ __forceinline__ void stage_quads(const DevView<float> &v, float2 *s_rec) {
    const int total = v.n_ops * 2 * v.d * W;
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const OpRec<float> o = ld_rec(v.op_ell + i);
        const int side = i / W / v.d & 1;
        const int l = max(o.idx, 0);
        s_rec[i] = make_float2(__int_as_float(side ? l : l * v.d), o.idx < 0 ? 0.f : o.re);
    }
    __syncthreads();
}

template <int W>
__device__ __forceinline__ void apply_quad(const DevView<float> &v, const float2 *s_rec,
                                           const cx<float> *__restrict__ X, int64_t n, int e0,
                                           cx<float> (&x0)[4], cx<float> (&y)[4]) {
    const int d = v.d, d2 = v.d2, r = e0 / d, c0 = e0 - r * d;
    const cx<float> *Xn = X + n * d2;
    const int t0 = __ldg(v.row_ptr + n), t1 = __ldg(v.row_ptr + n + 1);
    ld_row<float, 4, true>(Xn + e0, 1, x0);
    RowAcc<float, 4> acc;
    {
        const cx<float> dmp = ldc(v.damp + n);
        static_for<4>([&](auto E) {
            constexpr int u = E.value;
            cx<float> own{-dmp.re, -dmp.im};
            for (int j = __ldg(v.s_ptr + e0 + u), j1 = __ldg(v.s_ptr + e0 + u + 1); j < j1; ++j) {
                const cx<float> cf = ldc(v.s_val + j);
                const int src = __ldg(v.s_src + j);
                const cx<float> x[1] = {ldc(Xn + src)};
                if (src == e0 + u) own = own + cf;
                else acc.template mac<u, 1, 1>(cf, x);
            }
            const cx<float> x[1] = {x0[u]};
            acc.template mac<u, 1, 1>(own, x);
        });
    }
    const Kept kept(v, 0);
    for (int t = t0; t < t1; ++t) {
        cx<float> al, ar, xl[W][4], xr[W][4];
        float fl[W], fr[W][4];
        // every load of the entry
        const int4 raw = __ldg(reinterpret_cast<const int4 *>(v.ent) + t);
        if (!kept(raw.x)) continue;  // beyond the set's tiers: not in its hierarchy
        const float ml = (float)(int16_t)(raw.z >> 16), mr = (float)(int16_t)(raw.w & 0xffff);
        if ((int16_t)(raw.z & 0xffff) > 0) {
            al = ar = cx<float>{0.f, -1.f};
        } else {
            al = mul_mi(ldc(v.coefL + (raw.y >> 16)));
            ar = mul_mi(ldc(v.coefR + (raw.y >> 16)));
        }
        const cx<float> *Xb = X + (int64_t)raw.x * d2;
        const float2 *ol = s_rec + (int)(int16_t)(raw.y & 0xffff) * 2 * d * W + r * W;
        const float2 *oc = s_rec + ((int)(int16_t)(raw.y & 0xffff) * 2 * d + d + c0) * W;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const float2 o = ol[w];
            fl[w] = ml * o.y;
            ld_row<float, 4, true>(Xb + __float_as_int(o.x) + c0, 1, xl[w]);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float2 p = oc[u * W + w];
                fr[w][u] = mr * p.y;
                xr[w][u] = ldc(Xb + r * d + __float_as_int(p.x));
            }
        }
        // an element that is not coupled adds nothing, whatever it holds
#pragma unroll
        for (int w = 0; w < W; ++w) {
            if (fl[w] != 0.f) acc.template mac<0, 4, 1>(fl[w] * al, xl[w]);
            static_for<4>([&](auto E) {
                constexpr int u = E.value;
                const cx<float> x[1] = {xr[w][u]};
                if (fr[w][u] != 0.f) acc.template mac<u, 1, 1>(fr[w][u] * ar, x);
            });
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) y[u] = acc.value(u);
}

// ---------------------------------------------------------------- many columns
// s[q * D + c] = (M X)[n][r0 + q][c][b] for RP rows (RP = D: the whole block, r0 = 0), x0 likewise
// the input; s_ops as staged by stage_ops (fixed width W). Term order as in apply_rows.
template <class R, int D, int RP, int W>
__device__ __forceinline__ void apply_cols(const DevView<R> &v, const OpRec<R> *s_ops, const cx<R> *__restrict__ X,
                                           int64_t n, int r0, int64_t b, int64_t B, int set,
                                           cx<R> (&x0)[RP * D], cx<R> (&s)[RP * D]) {
    constexpr int D2 = D * D;
    const int ns = v.n_sets;
    const cx<R> *Xn = X + n * D2 * B + b;
    const int t0 = __ldg(v.row_ptr + n), t1 = __ldg(v.row_ptr + n + 1);
    const cx<R> dmp = ldc(v.damp + n * ns + set);
#pragma unroll
    for (int u = 0; u < RP * D; ++u) x0[u] = ldc(Xn + (r0 * D + u) * B);
    const Kept kept(v, set);
    RowAcc<R, RP * D> acc;
    static_for<RP * D>([&](auto U) {
        constexpr int u = U.value;
        const int e = r0 * D + u;
        cx<R> own{-dmp.re, -dmp.im};
        for (int j = __ldg(v.s_ptr + e), j1 = __ldg(v.s_ptr + e + 1); j < j1; ++j) {
            const cx<R> cf = ldc(v.s_val + (int64_t)j * ns + set);
            const int src = __ldg(v.s_src + j);
            const cx<R> x[1] = {ldc(Xn + src * B)};
            if (src == e) own = own + cf;
            else acc.template mac<u, 1, 1>(cf, x);
        }
        const cx<R> x[1] = {x0[u]};
        acc.template mac<u, 1, 1>(own, x);
    });
    int4 next = t0 < t1 ? __ldg(reinterpret_cast<const int4 *>(v.ent) + t0) : make_int4(0, 0, 0, 0);
    for (int t = t0; t < t1; ++t) {
        const int4 raw = next;
        if (t + 1 < t1) next = __ldg(reinterpret_cast<const int4 *>(v.ent) + t + 1);
        if (!kept(raw.x)) continue;  // beyond the set's tiers: not in its hierarchy
        const bool raised = (int16_t)(raw.z & 0xffff) > 0;
        const int ml = (int)(int16_t)(raw.z >> 16), mr = (int)(int16_t)(raw.w & 0xffff);
        const cx<R> *Xb = X + (int64_t)raw.x * D2 * B + b;
        const OpRec<R> *ol = s_ops + (int)(int16_t)(raw.y & 0xffff) * 2 * D * W, *oc = ol + D * W;
        cx<R> al{R(0), R(0)}, ar{R(0), R(0)};
        if (!raised) {
            const int64_t pk = (int64_t)(raw.y >> 16) * ns + set;
            al = mul_mi(ldc(v.coefL + pk));
            ar = mul_mi(ldc(v.coefR + pk));
        }
        static_for<RP>([&](auto Q) {
            constexpr int q = Q.value;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const OpRec<R> o = ol[(r0 + q) * W + w];
                if (o.idx >= 0) {
                    cx<R> x[D];
#pragma unroll
                    for (int c = 0; c < D; ++c) x[c] = ldc(Xb + (o.idx * D + c) * B);
                    acc.template mac<q * D, D, 1>(term_coef(o, raised, ml, al), x);
                }
            }
        });
        static_for<D>([&](auto C) {
            constexpr int c = C.value;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const OpRec<R> o = oc[c * W + w];
                if (o.idx >= 0) {
                    cx<R> x[RP];
#pragma unroll
                    for (int q = 0; q < RP; ++q) x[q] = ldc(Xb + ((r0 + q) * D + o.idx) * B);
                    acc.template mac<c, RP, D>(term_coef(o, raised, mr, ar), x);
                }
            }
        });
    }
#pragma unroll
    for (int u = 0; u < RP * D; ++u) s[u] = acc.value(u);
}

// ---------------------------------------------------------------- one element per thread
// y = (M X)[n][e][b] term by term, one element per thread, every coefficient multiplied as a whole. Most threads and
// least bookkeeping per thread: the fastest layout of FP32 launches that do not fill the chip, and in both precisions
// of operators with more than two non-zeros per row. Term order as in apply_rows.
template <class R>
__device__ __forceinline__ cx<R> apply_point(const DevView<R> &v, const cx<R> *__restrict__ X, int64_t n, int e,
                                             int64_t b, int64_t B, int set, cx<R> &x0) {
    const int d = v.d, ns = v.n_sets, r = e / d, c = e - r * d;
    const cx<R> *Xn = X + n * v.d2 * B + b;
    x0 = ldc(Xn + e * B);
    const cx<R> dmp = ldc(v.damp + n * ns + set);
    cx<R> acc{-(dmp.re * x0.re - dmp.im * x0.im), -(dmp.re * x0.im + dmp.im * x0.re)};
    for (int j = __ldg(v.s_ptr + e), j1 = __ldg(v.s_ptr + e + 1); j < j1; ++j)
        fma_to(acc, ldc(v.s_val + (int64_t)j * ns + set), ldc(Xn + __ldg(v.s_src + j) * B));
    const Kept kept(v, set);
    const int t1 = __ldg(v.row_ptr + n + 1);
    for (int t = __ldg(v.row_ptr + n); t < t1; ++t) {
        const int4 raw = __ldg(reinterpret_cast<const int4 *>(v.ent) + t);
        if (!kept(raw.x)) continue;  // beyond the set's tiers: not in its hierarchy
        const R ml = R((int16_t)(raw.z >> 16)), mr = R((int16_t)(raw.w & 0xffff));
        cx<R> cl{R(0), -ml}, cr{R(0), -mr};
        if ((int16_t)(raw.z & 0xffff) <= 0) {
            const int64_t pk = (int64_t)(raw.y >> 16) * ns + set;
            cl = mul_mi(ml * ldc(v.coefL + pk));
            cr = mul_mi(mr * ldc(v.coefR + pk));
        }
        const cx<R> *Xb = X + (int64_t)raw.x * v.d2 * B + b;
        const int base = (int)(int16_t)(raw.y & 0xffff) * (d + 1);
        for (int j = __ldg(v.op_rptr + base + r), j1 = __ldg(v.op_rptr + base + r + 1); j < j1; ++j) {
            const OpRec<R> o = ld_rec(v.op_rrec + j);
            fma_to(acc, cl * cx<R>{o.re, o.im}, ldc(Xb + (o.idx * d + c) * B));
        }
        for (int j = __ldg(v.op_cptr + base + c), j1 = __ldg(v.op_cptr + base + c + 1); j < j1; ++j) {
            const OpRec<R> o = ld_rec(v.op_crec + j);
            fma_to(acc, cr * cx<R>{o.re, o.im}, ldc(Xb + (r * d + o.idx) * B));
        }
    }
    return acc;
}

// ---------------------------------------------------------------- choice
// Whether an FP32 launch runs one element per thread in (32 columns x 8 elements) blocks. Operators with at most
// two non-zeros per row, several columns: the wider layouts need enough threads to pay off
// (d = 4, 16 and more columns: 25 ADOs x 17 columns 17.3 against 24.4
// us, 2,325 x 16 29.5 against 25.4; fewer columns: 2,325 x 8 23.2 against 27.9, 12,951 x 3 48 against 32);
// larger blocks have them only where 32-column blocks stand half empty (charge-cavity model, 790 ADOs of
// 24 x 24: 16 columns 327 against 345 us, 17 columns 627 against 382). One column of larger blocks: the smallest
// launches (13 ADOs of 6 x 6 13 against 16 us, 4 of 24 x 24 10 against 12). The lines lie between the sizes measured
// (elements x columns: 6,800, 297,600, 595,200 and 621,648 at d = 4), not at a measured crossing.
inline bool point_ok(const DevView<float> &v, int64_t B) {
    const double el = (double)v.N * v.d2 * (double)B;
    if (el >= 2147483647.0 || (v.d > 4 && v.op_width > 2)) return false;
    if (B == 1) return v.d > 4 && el < 2500;
    if (v.d <= 4) return el < (B >= 16 ? 430e3 : 590e3);
    return B <= 16 || el < 800e3 || (double)((B + 31) / 32 * 32) < 1.5 * (double)B;
}
// Whether the FP32 one-column kernel runs a launch: d a multiple of four, real operators with at
// most two nonzeros per row and column, 16-byte aligned buffers.
inline bool quad_ok(const DevView<float> &v, int64_t B, const void *a, const void *b, const void *c = nullptr,
                    const void *e = nullptr) {
    return B == 1 && v.d % 4 == 0 && v.op_ell && v.op_real &&
           (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)e) & 15) == 0 &&
           (size_t)v.n_ops * 2 * v.d * v.op_width * sizeof(float2) <= kStageOps;
}
inline bool quad_ok(const DevView<double> &, int64_t, const void *, const void *, const void * = nullptr,
                    const void * = nullptr) {
    return false;
}

// Whether the one-column layout runs a launch: FP64, small blocks, 16-byte aligned buffers, an ADO order
// (built from kWarpMinAdos ADOs on, one warp of 32 per SM sub-partition; below that, groups of
// d^2 / 4 threads per ADO use more of the chip (heom_staged.cuh), and below kStageMin64 elements
// one thread per element).
template <class R>
inline bool warp_ok(const DevView<R> &v, int64_t B, const void *a, const void *b, const void *c = nullptr,
                    const void *e = nullptr) {
    return sizeof(R) == 8 && B == 1 && (v.d == 2 || v.d == 4) && v.perm && v.op_ell &&
           (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)e) & 15) == 0 &&
           (size_t)v.n_ops * 2 * v.d * v.op_width * sizeof(OpRec<R>) <= kStageOps;
}
// dynamic shared memory of a one-column launch
template <class R, int D>
inline size_t warp_launch_smem(const DevView<R> &v) {
    return (size_t)v.n_ops * 2 * v.d * v.op_width * sizeof(OpRec<R>) + kWarpWarps * warp_smem<R, D>();
}

// ---------------------------------------------------------------- layouts
// What a thread of the flat and per-column-sum kernels forms: run q of NE neighbouring elements
// (ADO n, elements e0 .. e0 + NE - 1) of one column, and the function that forms it.
template <class R, int CW>
struct RowsLayout {  // runs of a row, operator lists from global memory
    static constexpr int NE = CW, MINB = 1;
    static constexpr bool VEC = false;
    static __host__ __device__ int per_ado(const DevView<R> &v) { return v.d2 / CW; }
    static __device__ __forceinline__ const OpRec<R> *stage(const DevView<R> &) { return nullptr; }
    static __device__ __forceinline__ void pos(const DevView<R> &v, int64_t q, bool small, int64_t &n, int &e0) {
        const RowPos p = row_of<CW>(q, v.d, small);
        n = p.n;
        e0 = p.r * v.d + p.c0;
    }
    static __device__ __forceinline__ void apply(const DevView<R> &v, const OpRec<R> *, const cx<R> *__restrict__ X,
                                                 int64_t n, int e0, int64_t b, int64_t B, int set, cx<R> (&x0)[NE],
                                                 cx<R> (&y)[NE]) {
        const int r = e0 / v.d;
        apply_rows<R, CW>(v, X, n, r, e0 - r * v.d, b, B, set, x0, y);
    }
};
template <int W>
struct QuadLayout {  // FP32, one column: four elements, branch-free
    static constexpr int NE = 4;
    static constexpr bool VEC = true;  // one column, 16-byte loads and stores
    static __host__ __device__ int per_ado(const DevView<float> &v) { return v.d2 / 4; }
    static __device__ __forceinline__ const float2 *stage(const DevView<float> &v) {
        extern __shared__ __align__(16) unsigned char quad_smem[];
        float2 *s = reinterpret_cast<float2 *>(quad_smem);
        stage_quads<W>(v, s);
        return s;
    }
    static __device__ __forceinline__ void pos(const DevView<float> &v, int64_t q, bool small, int64_t &n, int &e0) {
        const int pa = v.d2 / 4;
        n = small ? (int64_t)((uint32_t)q / (uint32_t)pa) : q / pa;
        e0 = (int)(q - n * pa) * 4;
    }
    static __device__ __forceinline__ void apply(const DevView<float> &v, const float2 *s_rec,
                                                 const cx<float> *__restrict__ X, int64_t n, int e0, int64_t, int64_t,
                                                 int, cx<float> (&x0)[4], cx<float> (&y)[4]) {
        apply_quad<W>(v, s_rec, X, n, e0, x0, y);
    }
};
template <class R, int D, int RP, int W>
struct ColsLayout {  // RP rows of a small block, operators in shared memory
    static constexpr int NE = RP * D, PA = D / RP;
    // blocks of 256 per SM that kernels with per-column sums are compiled for: the FP32 row waits for loads and
    // wants the warps (32 sets of uneven depth, 12,951 ADOs: stationary states 111 -> 98 ms)
    static constexpr int MINB = sizeof(R) == 4 && RP == 1 ? 3 : 1;
    static constexpr bool VEC = false;
    static __host__ __device__ int per_ado(const DevView<R> &) { return PA; }
    static __device__ __forceinline__ const OpRec<R> *stage(const DevView<R> &v) {
        extern __shared__ __align__(16) unsigned char cols_smem[];
        OpRec<R> *s = reinterpret_cast<OpRec<R> *>(cols_smem);
        stage_ops<R, W>(v, s);
        return s;
    }
    static __device__ __forceinline__ void pos(const DevView<R> &, int64_t q, bool, int64_t &n, int &e0) {
        n = q / PA;
        e0 = (int)(q - n * PA) * NE;
    }
    static __device__ __forceinline__ void apply(const DevView<R> &v, const OpRec<R> *s_ops,
                                                 const cx<R> *__restrict__ X, int64_t n, int e0, int64_t b, int64_t B,
                                                 int set, cx<R> (&x0)[NE], cx<R> (&y)[NE]) {
        apply_cols<R, D, RP, W>(v, s_ops, X, n, e0 / D, b, B, set, x0, y);
    }
};

template <class R>
struct PointLayout {  // one element
    static constexpr int NE = 1, MINB = 1;
    static constexpr bool VEC = false;
    static __host__ __device__ int per_ado(const DevView<R> &v) { return v.d2; }
    static __device__ __forceinline__ const OpRec<R> *stage(const DevView<R> &) { return nullptr; }
    static __device__ __forceinline__ void pos(const DevView<R> &v, int64_t q, bool small, int64_t &n, int &e0) {
        n = small ? (int64_t)((uint32_t)q / (uint32_t)v.d2) : q / v.d2;
        e0 = (int)(q - n * v.d2);
    }
    static __device__ __forceinline__ void apply(const DevView<R> &v, const OpRec<R> *, const cx<R> *__restrict__ X,
                                                 int64_t n, int e0, int64_t b, int64_t B, int set, cx<R> (&x0)[1],
                                                 cx<R> (&y)[1]) {
        y[0] = apply_point(v, X, n, e0, b, B, set, x0[0]);
    }
};

// Layout of a launch: cw > 0 the row layout (point: one element per thread with whole coefficients), quad the FP32
// one-column layout, else rows/w of the many-column one.
struct LayoutPick {
    int cw = 1, d = 0, rows = 0, w = 0, ne = 1;
    bool quad = false, point = false;
    size_t smem = 0;
};
constexpr int64_t kColsMinB = 16;
// FP64: the whole block per thread from eight warps per SM sub-partition on, else one row; FP32: one
// row (the whole block's accumulators take 150 registers)
constexpr int64_t kColsWhole = 608 * 32 * 8;
template <class R>
inline LayoutPick pick_layout(const DevView<R> &v, int64_t B, bool quad = false, int64_t min_b = kColsMinB) {
    LayoutPick p;
    if (quad) {
        p.quad = true;
        p.cw = 0;
        p.ne = 4;
        p.w = v.op_width;
        p.smem = (size_t)v.n_ops * 2 * v.d * v.op_width * sizeof(float2);
        return p;
    }
    const size_t ops = (size_t)v.n_ops * 2 * v.d * v.op_width * sizeof(OpRec<R>);
    if ((v.d == 2 || v.d == 4) && B >= min_b && v.op_width >= 1 && v.op_width <= 2 && ops <= kStageOps) {
        p.cw = 0;
        p.d = v.d;
        p.rows = v.d == 2 || (sizeof(R) == 8 && v.N * B >= kColsWhole) ? v.d : 1;
        p.w = v.op_width;
        p.ne = p.rows * v.d;
        p.smem = ops;
        return p;
    }
    p.cw = p.ne = row_width(v.N, v.d, B);
    // More than two non-zeros per row: decoding shared by a run no longer pays, one element per thread with every
    // coefficient multiplied as a whole does. RK4, three steps, in rows, in 32 x 8 blocks of elements, so: 222 ADOs of
    // 16 x 16, 20 columns FP32 5.3, 4.0, 2.7 ms; 27 of 24 x 24 FP64, two columns 4.4, 3.4, 2.3 ms, 15 columns 16.2, 9.7, 8.7
    // ms, 32 columns 25.9, 14.9, 14.8 ms. An iteration's FP64 apply of 27 ADOs of 8 x 8, five columns: 160 us in rows.
    if (v.op_width > 2) {
        p.cw = p.ne = 1;
        p.point = true;
    }
    return p;
}
// one element per thread: FP64 leaves out the zero halves of coefficients
template <class R>
using OneLayout = std::conditional_t<sizeof(R) == 8, RowsLayout<R, 1>, PointLayout<R>>;

// CALL(Layout) of a pick
#define HEOM_COLS_W(R, D, RP, w, CALL)                                                          \
    do {                                                                                        \
        if ((w) == 1) { using Ly = ColsLayout<R, D, RP, 1>; CALL(Ly); }                         \
        else { using Ly = ColsLayout<R, D, RP, 2>; CALL(Ly); }                                  \
    } while (0)
#define HEOM_LAYOUT_DISPATCH(R, p, CALL)                                                        \
    do {                                                                                        \
        if ((p).cw == 4) { using Ly = RowsLayout<R, 4>; CALL(Ly); }                             \
        else if ((p).cw == 2) { using Ly = RowsLayout<R, 2>; CALL(Ly); }                        \
        else if ((p).cw == 1 && (p).point) { using Ly = PointLayout<R>; CALL(Ly); }             \
        else if ((p).cw == 1) { using Ly = OneLayout<R>; CALL(Ly); }                            \
        else if ((p).d == 2) HEOM_COLS_W(R, 2, 2, (p).w, CALL);                                 \
        else if ((p).rows == 4) HEOM_COLS_W(R, 4, 4, (p).w, CALL);                              \
        else HEOM_COLS_W(R, 4, 1, (p).w, CALL);                                                 \
    } while (0)

// the same with the FP32 one-column layout among the choices (CALLs of double ignore it)
#define HEOM_FLAT_DISPATCH(R, p, CALL)                                                          \
    do {                                                                                        \
        if constexpr (sizeof(R) == 4) {                                                         \
            if ((p).quad) {                                                                     \
                if ((p).w == 1) { using Ly = QuadLayout<1>; CALL(Ly); }                         \
                else { using Ly = QuadLayout<2>; CALL(Ly); }                                    \
                break;                                                                          \
            }                                                                                   \
        }                                                                                       \
        HEOM_LAYOUT_DISPATCH(R, p, CALL);                                                       \
    } while (0)

// (run, column) of flat index i, columns fastest
__device__ __forceinline__ void run_col(int64_t i, int64_t B, bool small, int64_t &q, int64_t &b) {
    if (B == 1) {
        q = i;
        b = 0;
        return;
    }
    q = small ? (int64_t)((uint32_t)i / (uint32_t)B) : i / B;
    b = i - q * B;
}

}  // namespace heom
