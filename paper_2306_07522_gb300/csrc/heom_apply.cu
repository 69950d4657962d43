// The hot path: y = M x over all ADOs and batch columns (Eq. HEOM), matrix-free.
//
// By size, batch and operators (launch_apply): block products of dense FP32 operators (heom_dense.cu), the
// tiled kernel for many columns of one parameter set (heom_tile.cuh), a block per lane for one FP64 column of many
// ADOs and one element per thread for small FP32 launches (heom_block.cuh), neighbour blocks staged through shared
// memory for a few columns, in FP64 of large hierarchies only (heom_staged.cuh), and the flat kernel below over rows,
// quads of elements, whole blocks or, where operators have more than two non-zeros per row, single elements
// (heom_rows.cuh, heom_block.cuh) for everything else.
#include <algorithm>
#include <cstdint>

#include "heom_block.cuh"
#include "heom_tile.cuh"

namespace heom {

Geom make_geom(int64_t rows, int64_t B, int max_blocks_x) {
    Geom g;
    int bx = 1;
    while (bx < B && bx < 32) bx <<= 1;
    int by = 256 / bx;
    g.block = dim3(bx, by, 1);
    int64_t gy = (B + bx - 1) / bx;
    int64_t gx = (rows + by - 1) / by;
    if (max_blocks_x > 0 && gx > max_blocks_x) gx = max_blocks_x;
    if (gx < 1) gx = 1;
    g.grid = dim3((unsigned)gx, (unsigned)gy, 1);
    g.rows = rows;
    g.B = B;
    return g;
}

// y = M x (+ shift, trace augmentation), one thread per run of elements and column
template <class R, class Ly>
__global__ void __launch_bounds__(256, Ly::VEC ? 3 : 1) k_apply(DevView<R> v, const cx<R> *__restrict__ x,
                                               cx<R> *__restrict__ y, int64_t B, ColSets cps,
                                               ApplyMods<R> mods) {
    constexpr int NE = Ly::NE;
    const auto s_ops = Ly::stage(v);
    const int64_t total = v.N * Ly::per_ado(v) * B;
    const bool small = total < (int64_t(1) << 31);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        int64_t q, b, n;
        int e0;
        run_col(i, B, small, q, b);
        Ly::pos(v, q, small, n, e0);
        const int set = cps.set(b);
        const int64_t i0 = (n * v.d2 + e0) * B + b;
        cx<R> x0[NE], o[NE];
        if (beyond_cap(v, n, set)) zero_rows<R, NE>(mods.shift ? x + i0 : nullptr, B, x0, o);
        else Ly::apply(v, s_ops, x, n, e0, b, B, set, x0, o);
        apply_mods<R, NE>(mods, v, x, n, e0, b, B, x0, o);
        st_row<R, NE, Ly::VEC>(y + i0, B, o);
    }
}

// y = M x for the launches of point_ok: threadIdx.x over columns, threadIdx.y over elements
template <class R>
__global__ void __launch_bounds__(256) k_apply_point(DevView<R> v, const cx<R> *__restrict__ x, cx<R> *__restrict__ y,
                                                     int64_t B, ColSets cps, ApplyMods<R> mods) {
    const int b = blockIdx.y * blockDim.x + threadIdx.x, rows = (int)v.N * v.d2;
    const int row = blockIdx.x * blockDim.y + threadIdx.y;
    if (b >= B || row >= rows) return;
    const int n = row / v.d2, e = row - n * v.d2, set = cps.set(b);
    const int64_t i0 = (int64_t)row * B + b;
    cx<R> x0[1], o[1];
    if (beyond_cap(v, n, set)) zero_rows<R, 1>(mods.shift ? x + i0 : nullptr, B, x0, o);
    else o[0] = apply_point(v, x, n, e, b, B, set, x0[0]);
    apply_mods<R, 1>(mods, v, x, n, e, b, B, x0, o);
    y[i0] = o[0];
}

// One column of a large hierarchy of small blocks: 32 ADOs per warp (heom_block.cuh). The warp
// hands its blocks through shared memory and writes whole lines.
template <class R, int D, int W>
__global__ void __launch_bounds__(kWarpWarps * 32) k_apply_warp(DevView<R> v, const cx<R> *__restrict__ x,
                                                                cx<R> *__restrict__ y, ApplyMods<R> mods) {
    constexpr int D2 = D * D, SL = warp_slot<R, D>();
    extern __shared__ __align__(16) unsigned char warp_sm[];
    OpRec<R> *s_ops = reinterpret_cast<OpRec<R> *>(warp_sm);
    stage_ops<R, W>(v, s_ops);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cx<R> *ring = reinterpret_cast<cx<R> *>(s_ops + v.n_ops * 2 * D * W) +
                  (size_t)warp * (warp_smem<R, D>() / sizeof(cx<R>));
    for (int64_t n0 = ((int64_t)blockIdx.x * kWarpWarps + warp) * 32; n0 < v.N;
         n0 += (int64_t)gridDim.x * kWarpWarps * 32) {
        const int n = n0 + lane < v.N ? __ldg(v.perm + n0 + lane) : -1;
        cx<R> s[D2];
        apply_warp<R, D, W>(v, s_ops, ring, x, n, s);
        if (n >= 0) {
            if (mods.shift) {
                const cx<R> sh = mods.shift[0];
#pragma unroll
                for (int e = 0; e < D2; ++e) fma_to(s[e], sh, x[(int64_t)n * D2 + e]);
            }
            if (mods.aug != R(0) && n == 0) {
                cx<R> tr{R(0), R(0)};
                for (int k = 0; k < D; ++k) tr = tr + x[k * D + k];
                s[0] = s[0] + mods.aug * tr;
            }
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < D2; ++e) ring[lane * SL + e] = s[e];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < D2; ++k) {
            const int i = k * 32 + lane, blk = i / D2, e = i % D2;
            const int to = __shfl_sync(0xffffffffu, n, blk);
            if (to >= 0) y[(int64_t)to * D2 + e] = ring[blk * SL + e];
        }
    }
}

// The same for a few columns, neighbour blocks staged through shared memory (heom_staged.cuh)
template <class R, int CW, bool BLOCK, int W>
__global__ void __launch_bounds__(512) k_apply_staged(DevView<R> v, const cx<R> *__restrict__ x, cx<R> *__restrict__ y, int64_t B,
                               ColSets cps, ApplyMods<R> mods, bool vec) {
    staged_items<R, CW, BLOCK, W>(v, B, cps, [&](bool in, int64_t n, int64_t b, int set, int g, cx<R> *ring,
                                                 const OpRec<R> *s_ops) {
        const bool cut = beyond_cap(v, n, set);
        const int64_t i0 = (n * v.d2 + g * CW) * B + b;
        cx<R> x0[CW], o[CW];
        apply_staged<R, CW, BLOCK, W>(v, s_ops, ring, x, in && !cut, n, g, b, B, set, vec, x0, o);
        if (!in || (BLOCK && g >= v.d2 / CW)) return;
        if (cut) zero_rows<R, CW>(mods.shift ? x + i0 : nullptr, B, x0, o);
        apply_mods<R, CW>(mods, v, x, n, g * CW, b, B, x0, o);
        if (vec) st_row<R, CW, true>(y + i0, B, o);
        else st_row<R, CW, false>(y + i0, B, o);
    });
}

template <class R>
cudaError_t launch_apply(const DevView<R> &v, const cx<R> *x, cx<R> *y, int64_t B,
                         const ApplyMods<R> &mods, cudaStream_t s) {
    // the tiled kernel reads and writes 16-byte vectors: both buffers must be 16-byte aligned
    const bool tiled = tile_ok(v, B) && (((uintptr_t)x | (uintptr_t)y) & 15) == 0;
    if constexpr (sizeof(R) == 4)
        if (!(tiled && v.tile_pinned) && !mods.shift && mods.aug == 0.f && dense_ok(v, B))
            return launch_apply_dense(v, x, y, B, s);
    if (tiled) {
        TileArgs<R> a{};
        a.v = v;
        a.x = x;
        a.out = y;
        a.shift = mods.shift;
        a.aug = mods.aug;
        a.B = B;
        return launch_tile<R, TM_STORE>(a, s);
    }
    const ColSets cps(B / v.n_sets);
    const bool quad = quad_ok(v, B, x, y);
    if (warp_ok(v, B, x, y)) {
        const unsigned grid = (unsigned)((v.N + 32 * kWarpWarps - 1) / (32 * kWarpWarps));
#define CALL(D, W)                                                                                       \
    do {                                                                                                 \
        const size_t sm = warp_launch_smem<R, D>(v);                                                     \
        const cudaError_t e =                                                                            \
            cudaFuncSetAttribute(k_apply_warp<R, D, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm); \
        if (e != cudaSuccess) return e;                                                                  \
        k_apply_warp<R, D, W><<<grid, kWarpWarps * 32, sm, s>>>(v, x, y, mods);                          \
    } while (0)
        if (v.d == 4 && v.op_width == 1) CALL(4, 1);
        else if (v.d == 4) CALL(4, 2);
        else if (v.op_width == 1) CALL(2, 1);
        else CALL(2, 2);
#undef CALL
        return cudaGetLastError();
    }
    const StageGeom sg = stage_geom(v, B);
    if constexpr (sizeof(R) == 4)
        if (point_ok(v, B)) {
            const Geom g = make_geom(v.N * v.d2, B, 1 << 30);
            k_apply_point<R><<<g.grid, g.block, 0, s>>>(v, x, y, B, cps, mods);
            return cudaGetLastError();
        }
    if (sg.cw && !quad) {
        const bool vec = row_vec<R>(B, x, y);
#define CALL(CW, BLOCK, W) \
    return launch_staged(k_apply_staged<R, CW, BLOCK, W>, sg, s, v, x, y, B, cps, mods, vec)
        HEOM_STAGE_DISPATCH(sg, CALL);
#undef CALL
    }
    const LayoutPick p = pick_layout(v, B, quad);
    const Geom g = flat_geom(v.N * v.d2 / p.ne * B);
#define CALL(Ly) k_apply<R, Ly><<<g.grid, g.block, p.smem, s>>>(v, x, y, B, cps, mods)
    HEOM_FLAT_DISPATCH(R, p, CALL);
#undef CALL
    return cudaGetLastError();
}

// damp[n][set] = sum_k count_k rate_k over the occupied exponents of ADO n, in FP64 and rounded
// to FP32 (one table entry per ADO and set, read by every element of the ADO's block)
__global__ void k_damping(int64_t N, int n_sets, const int32_t *__restrict__ occ_ptr, const OccEntry *__restrict__ occ,
                          const cx<double> *__restrict__ rate, cx<double> *__restrict__ d64, cx<float> *__restrict__ d32) {
    const int64_t total = N * n_sets;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t n = i / n_sets;
        const int set = (int)(i - n * n_sets);
        cx<double> a{0.0, 0.0};
        for (int o = occ_ptr[n]; o < occ_ptr[n + 1]; ++o)
            a = a + (double)occ[o].count * rate[(int64_t)occ[o].k * n_sets + set];
        d64[i] = a;
        d32[i] = cast<float>(a);
    }
}

heom_status fill_damping(heom_hier *h, int n_sets, cudaStream_t s) {
    const int64_t total = h->N * n_sets;
    heom_status st = HEOM_OK;
    // tables of the same size stay (the uploads before this have waited for the device)
    if (h->d_damp64.bytes != total * sizeof(cx<double>)) st = dalloc(h->d_damp64, total * sizeof(cx<double>));
    if (st == HEOM_OK && h->d_damp32.bytes != total * sizeof(cx<float>)) st = dalloc(h->d_damp32, total * sizeof(cx<float>));
    if (st != HEOM_OK) return st;
    const Geom g = flat_geom(std::min<int64_t>(total, 152 * 16 * 256));
    k_damping<<<g.grid, g.block, 0, s>>>(h->N, n_sets, (const int32_t *)h->d_occ_ptr.p, (const OccEntry *)h->d_occ.p,
                                         (const cx<double> *)h->d_rate64.p, (cx<double> *)h->d_damp64.p,
                                         (cx<float> *)h->d_damp32.p);
    HEOM_CUDA(cudaGetLastError());
    return HEOM_OK;
}

template cudaError_t launch_apply<double>(const DevView<double> &, const cx<double> *,
                                          cx<double> *, int64_t, const ApplyMods<double> &,
                                          cudaStream_t);
template cudaError_t launch_apply<float>(const DevView<float> &, const cx<float> *, cx<float> *,
                                         int64_t, const ApplyMods<float> &, cudaStream_t);

}  // namespace heom

extern "C" heom_status heom_apply(const heom_hier *h, const void *x, void *y, int64_t batch,
                                  int prec, heom_stream s) {
    if (!h || !x || !y || batch < 1 || batch % h->n_sets != 0 ||
        (prec != HEOM_FP64 && prec != HEOM_FP32)) {
        heom::set_error("heom_apply: need a hierarchy, x, y, batch >= 1 (multiple of n_sets) and "
                        "prec FP64 or FP32");
        return HEOM_EINVAL;
    }
    if (batch > 65535LL * 32) {
        heom::set_error("heom_apply: batch larger than 2097120");
        return HEOM_EINVAL;
    }
    const size_t elt = prec == HEOM_FP64 ? 16 : 8;
    const size_t bytes = (size_t)h->N * h->d2 * batch * elt;
    const char *xs = (const char *)x, *ys = (const char *)y;
    if (xs < ys + bytes && ys < xs + bytes) {
        heom::set_error("heom_apply: x and y overlap");
        return HEOM_EINVAL;
    }
    HEOM_DEVICE(h->device);
    cudaError_t e;
    // accounted here, not in launch_apply: the solvers that call launch_apply account the
    // launch under their own kernel class
    heom::Prof pr(HEOM_KC_APPLY, (cudaStream_t)s, (double)h->N * batch, 2.0 * bytes);
    if (prec == HEOM_FP64) {
        heom::ApplyMods<double> m{nullptr, 0.0};
        e = heom::launch_apply(h->view64(), (const heom::cx<double> *)x, (heom::cx<double> *)y,
                               batch, m, (cudaStream_t)s);
    } else {
        heom::ApplyMods<float> m{nullptr, 0.0f};
        e = heom::launch_apply(h->view32(), (const heom::cx<float> *)x, (heom::cx<float> *)y,
                               batch, m, (cudaStream_t)s);
    }
    if (e != cudaSuccess) return heom::cuda_fail(e, "heom_apply launch");
    return HEOM_OK;
}

// ------------------------------------------------------------------ autotuner
namespace heom {
namespace {

// deterministic bounded input: re, im of x[i] from a 64-bit mix of i, in [-1, 1)
template <class R>
__global__ void k_tune_fill(int64_t total, cx<R> *x) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t z = (uint64_t)i * 0x9e3779b97f4a7c15ULL;
        z = (z ^ (z >> 31)) * 0xbf58476d1ce4e5b9ULL;
        z ^= z >> 29;
        const double a = (double)(z >> 40) * (1.0 / 8388608.0) - 1.0;
        const double b = (double)((z >> 16) & 0xffffffULL) * (1.0 / 8388608.0) - 1.0;
        x[i] = cx<R>{R(a), R(b)};
    }
}

// average device time of `reps` applies of the hierarchy's current configuration
template <class R>
heom_status tune_time(heom_hier *h, const cx<R> *x, cx<R> *y, int64_t B, cudaStream_t s, double *us) {
    const ApplyMods<R> m{nullptr, R(0)};
    auto view = [&]() {
        if constexpr (sizeof(R) == 8) return h->view64();
        else return h->view32();
    };
    const DevView<R> cur = view();
    cudaEvent_t e0, e1;
    HEOM_CUDA(cudaEventCreate(&e0));
    HEOM_CUDA(cudaEventCreate(&e1));
    const int reps = 5;
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = launch_apply(cur, x, y, B, m, s);  // warm-up
    if (e == cudaSuccess) e = cudaEventRecord(e0, s);
    for (int k = 0; k < reps && e == cudaSuccess; ++k) e = launch_apply(cur, x, y, B, m, s);
    if (e == cudaSuccess) e = cudaEventRecord(e1, s);
    if (e == cudaSuccess) e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) return cuda_fail(e, "heom_autotune");
    *us = 1e3 * ms / reps;
    return HEOM_OK;
}

template <class R>
heom_status autotune(heom_hier *h, int64_t B, double *cand, int *tiled, int *per_sm, int *variant,
                     double *best, cudaStream_t s) {
    const int64_t total = h->N * h->d2 * B;
    DBuf buf;
    heom_status st = dalloc(buf, 2 * total * sizeof(cx<R>));
    if (st != HEOM_OK) return st;
    cx<R> *x = (cx<R> *)buf.p, *y = x + total;
    k_tune_fill<R><<<(unsigned)std::min<int64_t>((total + 255) / 256, 152 * 16), 256, 0, s>>>(total, x);
    const int per_sm0 = h->tile_per_sm, var0 = h->tile_var, pinned0 = h->tile_pinned;
    const int64_t min_b0 = h->tile_min_b;
    // candidate 0: what runs with the tiled kernel switched off
    h->tile_min_b = INT64_MAX;
    double t0 = 0.0;
    st = tune_time<R>(h, x, y, B, s, &t0);
    cand[0] = t0;
    int best_p = 0, best_v = var0;
    double best_t = t0;
    // candidates 1..5: the tiled kernel with 1..5 ADO ranges per SM, each with every FP32
    // variant (FP64 has one); cand[p] keeps the fastest variant at p ranges per SM
    const bool tile_possible = B >= 16 && h->n_sets == 1 && !(sizeof(R) == 4 && (B & 1));
    const int n_var = sizeof(R) == 4 ? kTileVariants : 1;
    for (int p = 1; p <= 5 && st == HEOM_OK; ++p) {
        cand[p] = -1.0;
        if (!tile_possible) continue;
        if ((st = set_tile_partition(h, p)) != HEOM_OK) break;
        h->tile_min_b = 16;
        h->tile_pinned = 1;
        for (int var = 0; var < n_var && st == HEOM_OK; ++var) {
            h->tile_var = var;
            bool ok;
            if constexpr (sizeof(R) == 8) ok = tile_ok(h->view64(), B);
            else ok = tile_ok(h->view32(), B) && tile_var_of(h->view32(), B) == var;
            if (!ok) continue;  // ranges exceed the shared-memory budget, or B too narrow
            double t = 0.0;
            if ((st = tune_time<R>(h, x, y, B, s, &t)) != HEOM_OK) break;
            if (cand[p] < 0 || t < cand[p]) cand[p] = t;
            if (t < best_t) { best_t = t; best_p = p; best_v = var; }
        }
    }
    dfree(buf);
    if (st != HEOM_OK) {  // leave the configuration as it was
        set_tile_partition(h, per_sm0);
        h->tile_min_b = min_b0;
        h->tile_var = var0;
        h->tile_pinned = pinned0;
        return st;
    }
    // keep the winner: tiled with best_p ranges per SM and variant best_v, or no tiling
    // for batches up to this width (wider batches keep the tiled kernel at its default
    // granularity). The dense kernel is FP32's.
    h->tile_pinned = sizeof(R) == 4 ? (best_p > 0 ? 1 : 0) : std::min(pinned0, 1);
    if (best_p > 0) {
        st = set_tile_partition(h, best_p);
        h->tile_min_b = 16;
        if (sizeof(R) == 4) h->tile_var = best_v;
    } else {
        st = set_tile_partition(h, per_sm0 > 0 ? per_sm0 : 2);
        h->tile_min_b = B + 1;
        h->tile_var = var0;
    }
    *tiled = best_p > 0;
    *per_sm = best_p;
    *variant = best_p > 0 ? (sizeof(R) == 4 ? best_v : 0) : -1;
    *best = best_t;
    return st;
}

}  // namespace
}  // namespace heom

extern "C" heom_status heom_autotune(heom_hier *h, int64_t batch, int prec, double *candidates_us,
                                     int *tiled, int *ctas_per_sm, double *best_us, int *variant,
                                     heom_stream s) {
    if (!h || batch < 1 || batch > 65535LL * 32 || (prec != HEOM_FP64 && prec != HEOM_FP32)) {
        heom::set_error("heom_autotune: need a hierarchy, 1 <= batch <= 2097120, prec FP64 or FP32");
        return HEOM_EINVAL;
    }
    HEOM_DEVICE(h->device);
    double cand[6], best = 0.0;
    int t = 0, p = 0, var = -1;
    const heom_status st = prec == HEOM_FP64
                               ? heom::autotune<double>(h, batch, cand, &t, &p, &var, &best, (cudaStream_t)s)
                               : heom::autotune<float>(h, batch, cand, &t, &p, &var, &best, (cudaStream_t)s);
    if (st != HEOM_OK) return st;
    if (candidates_us) for (int i = 0; i < 6; ++i) candidates_us[i] = cand[i];
    if (tiled) *tiled = t;
    if (ctas_per_sm) *ctas_per_sm = p;
    if (best_us) *best_us = best;
    if (variant) *variant = var;
    return HEOM_OK;
}

extern "C" heom_status heom_set_tile_config(heom_hier *h, int ctas_per_sm, int variant) {
    if (!h || ctas_per_sm < 1 || ctas_per_sm > 5 || variant < 0 ||
        variant >= heom::kTileVariants) {
        heom::set_error("heom_set_tile_config: need a hierarchy, 1 <= ctas_per_sm <= 5 and "
                        "0 <= variant < %d", heom::kTileVariants);
        return HEOM_EINVAL;
    }
    HEOM_DEVICE(h->device);
    const heom_status st = heom::set_tile_partition(h, ctas_per_sm);
    if (st != HEOM_OK) return st;
    h->tile_var = variant;
    h->tile_min_b = 16;
    h->tile_pinned = 2;
    return HEOM_OK;
}
