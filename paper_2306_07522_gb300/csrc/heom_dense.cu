// FP32 apply of operators with few zeros (d = 8, 16, 24, 32): block products from shared memory.
//
// Term by term (heom_tile.cuh) a dense operator costs 2 d complex multiply-adds per neighbour and
// element, each with its own load from L1 or L2. Here a CTA owns one ADO and BT columns and works operator
// by operator: the neighbours coupled by one operator O are first summed, S = sum a X_nb and
// T = sum b X_nb, into shared memory (two multiply-adds per neighbour and element, each block read
// once per CTA), then Y += O S + T O: d x d products whose operands come from shared memory. A
// thread forms RT = d / 4 rows of one block column for four batch columns, so a step of the
// inner loop is 4 RT complex multiply-adds on packed FP32 pairs for RT + 2 (left) or 2 RT + 1 (right)
// 16-byte shared-memory loads, most of them broadcasts. Real and imaginary parts lie in separate planes: a
// pair holds two columns, and one accumulator pair takes the real, one the imaginary part. Zero entries of the
// operators are multiplied like the others; a thread whose results are not all finite forms them again without
// (infinities and NaN spread over couplings only).
//
// 222 ADOs of 24 x 24: 64 columns 2,595 us (term by term) -> 352 us, bound by shared-memory wavefronts (61 %) with two
// CTAs per SM (12.6 GFLOP of block products, FMA pipe half busy); one column 133 -> 50 us, bound by a CTA's chain of products. 16 x 16: 748 -> 118 us at 64
// columns, 99 -> 25 us at one.
#include <cstdint>

#include "heom_ff.cuh"
#include "heom_kernels.cuh"

namespace heom {

namespace {

struct DenseEntry {
    int32_t nb, op;
    cx<float> a, b;
};
constexpr int kDenseMaxEntries = 256;

__device__ __forceinline__ float2 lo(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 neg(float4 v) { return make_float4(-v.x, -v.y, -v.z, -v.w); }

// four columns of one row, planes re and im; cols: columns that exist; vec: 16-byte loads allowed
__device__ __forceinline__ void ld_cols(const cx<float> *__restrict__ p, int cols, bool vec, float4 &re, float4 &im) {
    if (vec && cols >= 4) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(p)), b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
        re = make_float4(a.x, a.z, b.x, b.z);
        im = make_float4(a.y, a.w, b.y, b.w);
    } else {
        const cx<float> none{0.f, 0.f};
        const cx<float> a = cols > 0 ? ldc(p) : none, b = cols > 1 ? ldc(p + 1) : none, c = cols > 2 ? ldc(p + 2) : none,
                        e = cols > 3 ? ldc(p + 3) : none;
        re = make_float4(a.re, b.re, c.re, e.re);
        im = make_float4(a.im, b.im, c.im, e.im);
    }
}
// (sr, si) += c (xr, xi)
__device__ __forceinline__ void cmac4(cx<float> c, float4 xr, float4 xi, float2 (&sr)[2], float2 (&si)[2]) {
    const float2 cr = make_float2(c.re, c.re), ci = make_float2(c.im, c.im), nc = make_float2(-c.im, -c.im);
    sr[0] = f2_fma(nc, lo(xi), f2_fma(cr, lo(xr), sr[0]));
    sr[1] = f2_fma(nc, hi(xi), f2_fma(cr, hi(xr), sr[1]));
    si[0] = f2_fma(ci, lo(xr), f2_fma(cr, lo(xi), si[0]));
    si[1] = f2_fma(ci, hi(xr), f2_fma(cr, hi(xi), si[1]));
}
__device__ __forceinline__ void st_planes(float *re, float *im, const float2 (&sr)[2], const float2 (&si)[2]) {
    *reinterpret_cast<float4 *>(re) = make_float4(sr[0].x, sr[0].y, sr[1].x, sr[1].y);
    *reinterpret_cast<float4 *>(im) = make_float4(si[0].x, si[0].y, si[1].x, si[1].y);
}

template <int D, int BT>
constexpr size_t dense_smem() {
    return (size_t)D * D * (4 * BT * sizeof(float) + sizeof(float4)) + kDenseMaxEntries * sizeof(DenseEntry);
}

// The results of a thread again without the zero entries of the operators, for a thread whose results are not all
// finite: a zero entry couples nothing, whatever the block sums hold. The same operations in the same order
// otherwise, so the results that are finite do not change; one by one, and out of line, so that the products above
// keep their registers.
template <int D>
__device__ __noinline__ void masked_results(const DevView<float> &v, const DenseEntry *ent, int cnt,
                                            const cx<float> *__restrict__ X, cx<float> *__restrict__ Y, int64_t n, int r0,
                                            int c, int64_t b0, int cols, int64_t B) {
    constexpr int D2 = D * D;
    const cx<float> dmp = ldc(v.damp + n);
    for (int r = r0; r < r0 + D / 4; ++r)
        for (int64_t b = b0; b < b0 + min(cols, 4); ++b) {
            cx<float> y{0.f, 0.f};
            fma_to(y, cx<float>{-dmp.re, -dmp.im}, ldc(X + (n * D2 + r * D + c) * B + b));
            for (int o = 0; o <= v.n_ops; ++o)
                for (int right = 0; right < 2; ++right)
                    for (int l = 0; l < D; ++l) {
                        const cx<float> q = ldc(v.dense + (int64_t)o * D2 + (right ? l * D + c : r * D + l));
                        if (q.re == 0.f && q.im == 0.f) continue;
                        const int64_t at = right ? r * D + l : l * D + c;
                        cx<float> sum{0.f, 0.f};
                        if (o == v.n_ops) {
                            fma_to(sum, cx<float>{0.f, right ? 1.f : -1.f}, ldc(X + (n * D2 + at) * B + b));
                        } else {
                            for (int t = 0; t < cnt; ++t)
                                if (ent[t].op == o)
                                    fma_to(sum, right ? ent[t].b : ent[t].a, ldc(X + (ent[t].nb * (int64_t)D2 + at) * B + b));
                        }
                        fma_to(y, q, sum);
                    }
            Y[(n * D2 + r * D + c) * B + b] = y;
        }
}

template <int D, int BT>
__global__ void __launch_bounds__(D *BT, 2) k_apply_dense(const __grid_constant__ DevView<float> v,
                                                          const cx<float> *__restrict__ X, cx<float> *__restrict__ Y,
                                                          int64_t B, bool vec) {
    constexpr int D2 = D * D, RT = D / 4, Q = BT / 4, T = D * BT;
    extern __shared__ __align__(16) unsigned char dense_sm[];
    float4 *rec = reinterpret_cast<float4 *>(dense_sm);  // operator (re, re, im, im)
    float *Lr = reinterpret_cast<float *>(rec + D2), *Li = Lr + D2 * BT, *Rr = Li + D2 * BT, *Ri = Rr + D2 * BT;
    DenseEntry *ent = reinterpret_cast<DenseEntry *>(Ri + D2 * BT);
    const int tid = threadIdx.x;
    const int64_t n = blockIdx.x % v.N, b0 = blockIdx.x / v.N * BT;
    const int t0 = __ldg(v.row_ptr + n), cnt = __ldg(v.row_ptr + n + 1) - t0;
    for (int t = tid; t < cnt; t += T) {
        const int4 raw = __ldg(reinterpret_cast<const int4 *>(v.ent) + t0 + t);
        const float ml = (float)(int16_t)(raw.z >> 16), mr = (float)(int16_t)(raw.w & 0xffff);
        DenseEntry q{raw.x, (int)(int16_t)(raw.y & 0xffff), {0.f, -ml}, {0.f, -mr}};
        if ((int16_t)(raw.z & 0xffff) <= 0) {
            q.a = ml * mul_mi(ldc(v.coefL + (raw.y >> 16)));
            q.b = mr * mul_mi(ldc(v.coefR + (raw.y >> 16)));
        }
        ent[t] = q;
    }
    // the thread's output: rows r0 .. r0 + RT - 1 of block column c, columns b0 + 4 bq .. + 3
    const int bq = tid % Q, c = tid / Q % D, r0 = tid / (Q * D) * RT;
    const int cols = (int)min((int64_t)4, B - b0 - 4 * bq);
    const cx<float> *Xb = X + b0;
    float2 are[RT][2], aim[RT][2];
    {
        const cx<float> dmp = ldc(v.damp + n);
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            float4 xr, xi;
            ld_cols(Xb + (n * D2 + (r0 + r) * D + c) * B + 4 * bq, cols, vec, xr, xi);
            are[r][0] = are[r][1] = aim[r][0] = aim[r][1] = make_float2(0.f, 0.f);
            cmac4(cx<float>{-dmp.re, -dmp.im}, xr, xi, are[r], aim[r]);
        }
    }
    for (int o = 0; o <= v.n_ops; ++o) {  // the last one is H: -i H X + i X H
        __syncthreads();                  // entries are there; the last products have been formed
        bool any = o == v.n_ops;
        for (int t = 0; t < cnt && !any; ++t) any = ent[t].op == o;
        if (!any) continue;
        for (int e = tid; e < D2; e += T) {
            const cx<float> w = ldc(v.dense + (int64_t)o * D2 + e);
            rec[e] = make_float4(w.re, w.re, w.im, w.im);
        }
#pragma unroll 1
        for (int i = 0; i < RT; i += 2) {  // two runs of four columns at a time
            float2 lr[2][2], li[2][2], rr[2][2], ri[2][2];
            int at[2], have[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int idx = tid + (i + u) * T, q = idx % Q;
                at[u] = idx / Q;
                have[u] = (int)min((int64_t)4, B - b0 - 4 * q);
                lr[u][0] = lr[u][1] = li[u][0] = li[u][1] = make_float2(0.f, 0.f);
                rr[u][0] = rr[u][1] = ri[u][0] = ri[u][1] = make_float2(0.f, 0.f);
            }
            const auto add = [&](int64_t nb, cx<float> a, cx<float> b) {
                float4 xr[2], xi[2];
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    ld_cols(Xb + (nb * D2 + at[u]) * B + 4 * ((tid + (i + u) * T) % Q), have[u], vec, xr[u], xi[u]);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    cmac4(a, xr[u], xi[u], lr[u], li[u]);
                    cmac4(b, xr[u], xi[u], rr[u], ri[u]);
                }
            };
            if (o == v.n_ops) {
                add(n, cx<float>{0.f, -1.f}, cx<float>{0.f, 1.f});
            } else {
                for (int t = 0; t < cnt; ++t)
                    if (ent[t].op == o) add(ent[t].nb, ent[t].a, ent[t].b);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int w = (tid + (i + u) * T) * 4;
                st_planes(Lr + w, Li + w, lr[u], li[u]);
                st_planes(Rr + w, Ri + w, rr[u], ri[u]);
            }
        }
        __syncthreads();
#pragma unroll 2
        for (int l = 0; l < D; ++l) {  // O S
            const int w = (l * D + c) * BT + 4 * bq;
            const float4 xr = *reinterpret_cast<const float4 *>(Lr + w), xi = *reinterpret_cast<const float4 *>(Li + w),
                         nx = neg(xi);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const float4 q = rec[(r0 + r) * D + l];
                are[r][0] = f2_fma(hi(q), lo(nx), f2_fma(lo(q), lo(xr), are[r][0]));
                are[r][1] = f2_fma(hi(q), hi(nx), f2_fma(lo(q), hi(xr), are[r][1]));
                aim[r][0] = f2_fma(hi(q), lo(xr), f2_fma(lo(q), lo(xi), aim[r][0]));
                aim[r][1] = f2_fma(hi(q), hi(xr), f2_fma(lo(q), hi(xi), aim[r][1]));
            }
        }
#pragma unroll 2
        for (int l = 0; l < D; ++l) {  // T O
            const float4 q = rec[l * D + c], nq = neg(q);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const int w = ((r0 + r) * D + l) * BT + 4 * bq;
                const float4 xr = *reinterpret_cast<const float4 *>(Rr + w), xi = *reinterpret_cast<const float4 *>(Ri + w);
                are[r][0] = f2_fma(hi(nq), lo(xi), f2_fma(lo(q), lo(xr), are[r][0]));
                are[r][1] = f2_fma(hi(nq), hi(xi), f2_fma(lo(q), hi(xr), are[r][1]));
                aim[r][0] = f2_fma(hi(q), lo(xr), f2_fma(lo(q), lo(xi), aim[r][0]));
                aim[r][1] = f2_fma(hi(q), hi(xr), f2_fma(lo(q), hi(xi), aim[r][1]));
            }
        }
    }
    float2 tot = make_float2(0.f, 0.f);
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        cx<float> *p = Y + (n * D2 + (r0 + r) * D + c) * B + b0 + 4 * bq;
        const float re[4] = {are[r][0].x, are[r][0].y, are[r][1].x, are[r][1].y};
        const float im[4] = {aim[r][0].x, aim[r][0].y, aim[r][1].x, aim[r][1].y};
        if (vec && cols >= 4) {
            reinterpret_cast<float4 *>(p)[0] = make_float4(re[0], im[0], re[1], im[1]);
            reinterpret_cast<float4 *>(p)[1] = make_float4(re[2], im[2], re[3], im[3]);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (u < cols) p[u] = cx<float>{re[u], im[u]};
        }
        tot = f2_add(tot, f2_add(f2_add(are[r][0], are[r][1]), f2_add(aim[r][0], aim[r][1])));
    }
    if (!(isfinite(tot.x) && isfinite(tot.y)) && cols > 0) masked_results<D>(v, ent, cnt, X, Y, n, r0, c, b0 + 4 * bq, cols, B);
}

template <int D, int BT>
cudaError_t launch_bt(const DevView<float> &v, const cx<float> *x, cx<float> *y, int64_t B, cudaStream_t s) {
    constexpr size_t sm = dense_smem<D, BT>();
    const cudaError_t e = cudaFuncSetAttribute(k_apply_dense<D, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const bool vec = B % 2 == 0 && (((uintptr_t)x | (uintptr_t)y) & 15) == 0;
    k_apply_dense<D, BT><<<(unsigned)(v.N * ((B + BT - 1) / BT)), D * BT, sm, s>>>(v, x, y, B, vec);
    return cudaGetLastError();
}

}  // namespace

// columns of a CTA
static int dense_columns(int d, int64_t B) { return B > 4 && d < 32 ? 8 : 4; }

bool dense_ok(const DevView<float> &v, int64_t B) {
    if (!v.dense || v.n_sets != 1 || v.set_cap || v.max_entries > kDenseMaxEntries) return false;
    const int bt = dense_columns(v.d, B);
    const double ctas = (double)v.N * (double)((B + bt - 1) / bt);
    return ctas >= v.dense_min && ctas < 2147483647.0;
}

cudaError_t launch_apply_dense(const DevView<float> &v, const cx<float> *x, cx<float> *y, int64_t B, cudaStream_t s) {
    const bool wide = dense_columns(v.d, B) == 8;
    switch (v.d) {
    case 8: return wide ? launch_bt<8, 8>(v, x, y, B, s) : launch_bt<8, 4>(v, x, y, B, s);
    case 16: return wide ? launch_bt<16, 8>(v, x, y, B, s) : launch_bt<16, 4>(v, x, y, B, s);
    case 24: return wide ? launch_bt<24, 8>(v, x, y, B, s) : launch_bt<24, 4>(v, x, y, B, s);
    default: return launch_bt<32, 4>(v, x, y, B, s);
    }
}

}  // namespace heom
