// The matrix-free HEOM apply of a few columns, block by block: a group of T = d^2 / CW threads
// owns one ADO of one column and streams the neighbour blocks it needs through shared memory.
//
// Why. In one column an ADO's block is 128 bytes (d = 4, FP32) to a few kilobytes, and every
// neighbour entry starts a chain of dependent loads -- entry, operator record, element -- of
// which the last comes from L2 or HBM. Followed one after the other these chains, and not bytes or
// multiply-adds, set the time (13 entries for a charge-cavity ADO, 24 to 53 for the low
// tiers of the Anderson model). Here the group copies whole neighbour blocks asynchronously
// (cp.async, each thread its own CW elements) kStageDepth deep, so the block of an entry is in
// shared memory when its turn comes and the operator's row and column lists, which sit there
// too, index it at shared-memory latency. A group inside one warp needs no block barrier.
// Operators: at most W (1 or 2) nonzeros per row and column (annihilators, number operators,
// Pauli matrices, a + a^dag); others run one element per thread (PointLayout, heom_block.cuh).
#pragma once

#include "heom_rows.cuh"

namespace heom {

constexpr int kStageDepth = 4;     // blocks in flight per group (a power of two)
constexpr int kStageThreads = 128; // block size when groups fit into warps

// Operator records (DevView::op_ell) into shared memory. All threads of the block.
template <class R, int W>
__device__ __forceinline__ void stage_ops(const DevView<R> &v, OpRec<R> *s_ops) {
    const int total = v.n_ops * 2 * v.d * W;
    for (int i = threadIdx.y * blockDim.x + threadIdx.x; i < total; i += blockDim.x * blockDim.y)
        s_ops[i] = ld_rec(v.op_ell + i);
    __syncthreads();
}

__device__ __forceinline__ void stage_copy(void *smem, const void *gmem, int bytes16) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if (bytes16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Elements of one ring slot, padded by 16 bytes so that neighbouring groups' rows fall into
// different banks.
template <class R>
__host__ __device__ inline int stage_slot(int d2) { return d2 + 16 / (int)(2 * sizeof(R)); }

// y[u] = (M X)[n][e0 + u][b] and x0[u] = X[n][e0 + u][b], e0 = g CW, for the group's ADO n and
// column b; called by every thread of the sync domain (the warp, or with BLOCK the block: one
// group, whose threads past the last element only synchronise), with on = false where a group
// has no ADO, or one beyond its set's truncation (the same for a whole block): it then only
// takes part in the synchronisation. ring: the group's kStageDepth slots. vec: B == 1 and X 16-byte
// aligned (FP32 copies of two elements at once). Term order as in apply_rows.
template <class R, int CW, bool BLOCK, int W>
__device__ __forceinline__ void apply_staged(const DevView<R> &v, const OpRec<R> *s_ops, cx<R> *ring,
                                             const cx<R> *__restrict__ X, bool on, int64_t n, int g, int64_t b,
                                             int64_t B, int set, bool vec, cx<R> (&x0)[CW], cx<R> (&y)[CW]) {
    constexpr int D = kStageDepth;
    const int d = v.d, d2 = v.d2, ns = v.n_sets, slot = stage_slot<R>(d2);
    const bool el = !BLOCK || g < d2 / CW;  // the thread has elements
    const int e0 = g * CW, r = e0 / d, c0 = e0 - r * d;
    int t0 = 0, cnt = -1;
    if (on) {
        t0 = __ldg(v.row_ptr + n);
        cnt = __ldg(v.row_ptr + n + 1) - t0;
    }
    const int last = BLOCK ? cnt : __reduce_max_sync(0xffffffffu, cnt);
    const Kept kept(v, set);  // inside the tiers of the column's parameter set
    auto issue = [&](int i) {  // block i of the group: its own ADO, then its neighbours in entry order
        if (i > cnt || !el) return;
        int64_t nb = n;
        if (i > 0) {
            nb = __ldg(reinterpret_cast<const int *>(v.ent) + 4 * (int64_t)(t0 + i - 1));
            if (!kept((int)nb)) return;
        }
        cx<R> *dst = ring + (i & (D - 1)) * slot + e0;
        const cx<R> *src = X + (nb * d2 + e0) * B + b;
        if constexpr (sizeof(R) == 8) {
#pragma unroll
            for (int u = 0; u < CW; ++u) stage_copy(dst + u, src + u * B, 1);
        } else {
            if (vec && CW % 2 == 0) {
#pragma unroll
                for (int u = 0; u < CW; u += 2) stage_copy(dst + u, src + u, 1);
            } else {
#pragma unroll
                for (int u = 0; u < CW; ++u) stage_copy(dst + u, src + u * B, 0);
            }
        }
    };
    if (BLOCK) __syncthreads();  // the ring is free again (previous ADO)
    else __syncwarp();
#pragma unroll
    for (int i = 0; i < D - 1; ++i) {
        issue(i);
        stage_commit();
    }
    RowAcc<R, CW> acc;
    for (int i = 0; i <= last; ++i) {
        int4 raw = make_int4(0, 0, 0, 0);
        cx<R> al{R(0), R(0)}, ar{R(0), R(0)};
        bool use = i <= cnt && el, raised = false;
        if (use && i > 0) {
            raw = __ldg(reinterpret_cast<const int4 *>(v.ent) + t0 + i - 1);
            use = kept(raw.x);
            raised = (int16_t)(raw.z & 0xffff) > 0;
            if (!raised) {
                const int64_t pk = (int64_t)(raw.y >> 16) * ns + set;
                al = mul_mi(ldc(v.coefL + pk));
                ar = mul_mi(ldc(v.coefR + pk));
            }
        }
        stage_wait<D - 2>();  // this thread's part of block i has landed
        if (BLOCK) __syncthreads();
        else __syncwarp();
        issue(i + D - 1);     // into the slot of block i - 1, which every thread has used
        stage_commit();
        if (!use) continue;
        const cx<R> *xs = ring + (i & (D - 1)) * slot;
        if (i == 0) {
            const cx<R> dmp = ldc(v.damp + n * ns + set);
            static_for<CW>([&](auto U) {
                constexpr int u = U.value;
                x0[u] = xs[e0 + u];
                cx<R> own{-dmp.re, -dmp.im};
                for (int j = __ldg(v.s_ptr + e0 + u), j1 = __ldg(v.s_ptr + e0 + u + 1); j < j1; ++j) {
                    const cx<R> cf = ldc(v.s_val + (int64_t)j * ns + set);
                    const int src = __ldg(v.s_src + j);
                    const cx<R> x[1] = {xs[src]};
                    if (src == e0 + u) own = own + cf;
                    else acc.template mac<u, 1, 1>(cf, x);
                }
                const cx<R> x[1] = {x0[u]};
                acc.template mac<u, 1, 1>(own, x);
            });
            continue;
        }
        const int ml = (int)(int16_t)(raw.z >> 16), mr = (int)(int16_t)(raw.w & 0xffff);
        const OpRec<R> *ol = s_ops + ((int)(int16_t)(raw.y & 0xffff) * 2 * d) * W, *oc = ol + d * W;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const OpRec<R> o = ol[r * W + w];
            if (o.idx >= 0) {
                cx<R> x[CW];
#pragma unroll
                for (int u = 0; u < CW; ++u) x[u] = xs[o.idx * d + c0 + u];
                acc.template mac<0, CW, 1>(term_coef(o, raised, ml, al), x);
            }
        }
        static_for<CW>([&](auto U) {
            constexpr int u = U.value;
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const OpRec<R> o = oc[(c0 + u) * W + w];
                if (o.idx >= 0) {
                    const cx<R> x[1] = {xs[r * d + o.idx]};
                    acc.template mac<u, 1, 1>(term_coef(o, raised, mr, ar), x);
                }
            }
        });
    }
    stage_wait<0>();
#pragma unroll
    for (int u = 0; u < CW; ++u) y[u] = acc.value(u);
}

// Geometry of a staged launch: cw elements per thread, T threads per group, groups per block
// (several inside warps, or one that fills the block), operator width; cw = 0: not applicable.
struct StageGeom {
    int cw = 0, T = 0, groups = 0, threads = 0, w = 0;
    bool block = false;
    size_t smem = 0;
    unsigned grid = 1;
};
constexpr size_t kStageOps = 24 * 1024;   // largest operator table
constexpr int64_t kStageMaxB = 15;        // wider batches read whole sectors column by column
// FP64: elements from which staging pays. Below them its groups leave most of the chip idle and one element per thread
// (RowsLayout) is faster, us: 13 ADOs of 24 x 24 39 against 18, 130 of 8 x 8 53 against 28, 301 of 4 x 4 with 24
// exponents 44 against 32, 2,325 46 against 30; 316 of 16 x 16, two columns (161,792 elements) 65 against 66.
constexpr double kStageMin64 = 160e3;
template <class R>
inline StageGeom stage_geom(const DevView<R> &v, int64_t B) {
    StageGeom g;
    if (v.d < 2 || v.d % 2 || v.op_width < 1 || v.op_width > 2 || B > kStageMaxB) return g;
    if (sizeof(R) == 8 && (double)v.N * v.d2 * (double)B < kStageMin64) return g;
    const size_t ops = (size_t)v.n_ops * 2 * v.d * v.op_width * sizeof(OpRec<R>);
    if (ops > kStageOps) return g;
    const int cw = v.d % 4 == 0 ? 4 : 2, T = v.d2 / cw;
    if (T > 512) return g;  // the launch bound of the staged kernels
    g.block = T > 32 || 32 % T != 0;
    g.threads = g.block ? (T + 31) / 32 * 32 : kStageThreads;
    g.groups = g.block ? 1 : kStageThreads / T;
    g.smem = ops + (size_t)g.groups * kStageDepth * stage_slot<R>(v.d2) * sizeof(cx<R>);
    if (g.smem > 200 * 1024) return g;
    g.cw = cw;
    g.T = T;
    g.w = v.op_width;
    g.grid = (unsigned)std::min<int64_t>((v.N * B + g.groups - 1) / g.groups, 1 << 30);
    return g;
}
// CALL(CW, BLOCK, W) of a staged geometry
#define HEOM_STAGE_DISPATCH(g, CALL)                                            \
    do {                                                                        \
        if ((g).cw == 4 && !(g).block) {                                        \
            if ((g).w == 1) { CALL(4, false, 1); } else { CALL(4, false, 2); }  \
        } else if ((g).cw == 4) {                                               \
            if ((g).w == 1) { CALL(4, true, 1); } else { CALL(4, true, 2); }    \
        } else if (!(g).block) {                                                \
            if ((g).w == 1) { CALL(2, false, 1); } else { CALL(2, false, 2); }  \
        } else {                                                                \
            if ((g).w == 1) { CALL(2, true, 1); } else { CALL(2, true, 2); }    \
        }                                                                       \
    } while (0)

// Launch of a staged kernel (its dynamic shared memory may exceed the default limit).
template <class... P, class... A>
inline cudaError_t launch_staged(void (*k)(P...), const StageGeom &g, cudaStream_t s, A... args) {
    if (g.smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem);
        if (e != cudaSuccess) return e;
    }
    k<<<g.grid, g.threads, g.smem, s>>>(args...);
    return cudaGetLastError();
}

// The (ADO, column) items of a staged kernel: body(in, n, b, set, g, ring, s_ops) with all
// threads of the block in step; in = false in the groups past the last item. In a block-wide
// group the threads g >= T have no elements.
template <class R, int CW, bool BLOCK, int W, class F>
__device__ __forceinline__ void staged_items(const DevView<R> &v, int64_t B, ColSets cps, F &&body) {
    extern __shared__ __align__(16) unsigned char stage_smem[];
    OpRec<R> *s_ops = reinterpret_cast<OpRec<R> *>(stage_smem);
    stage_ops<R, W>(v, s_ops);
    const int T = v.d2 / CW, groups = BLOCK ? 1 : (int)blockDim.x / T;
    const int slot = BLOCK ? 0 : threadIdx.x / T, g = BLOCK ? threadIdx.x : threadIdx.x - slot * T;
    cx<R> *ring = reinterpret_cast<cx<R> *>(s_ops + v.n_ops * 2 * v.d * W) + slot * kStageDepth * stage_slot<R>(v.d2);
    const int64_t total = v.N * B;
    for (int64_t base = (int64_t)blockIdx.x * groups; base < total; base += (int64_t)gridDim.x * groups) {
        const int64_t i = base + slot;
        const bool in = i < total;
        const int64_t n = !in ? 0 : B == 1 ? i : i / B, b = in ? i - n * B : 0;
        body(in, n, b, cps.set(b), g, ring, s_ops);
    }
}

}  // namespace heom
