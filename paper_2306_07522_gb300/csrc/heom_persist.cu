// Persistent cooperative BiCGStab for one right-hand side (batch 1): the whole solve is one
// launch. Each CTA owns one ADO range (one per SM), builds that range's term programs of
// Eq. HEOM in shared memory once (from the neighbour tables, never stored elsewhere) and
// keeps them for every iteration. Vector updates touch only the CTA's own rows; the apply
// reads neighbour rows of the whole vector after a grid-wide barrier. Dot products are
// block sums exchanged by the barriers and added in a fixed order by every CTA, so every CTA
// derives the same Krylov scalars and the same convergence decision without any host round trip. Five grid barriers per iteration; the host reads the result
// once, at the end. In the FP64 solve the two applies of an iteration run in float-float (the
// Krylov vectors, dot products and scalars stay FP64).
#include <algorithm>
#include <cmath>

#include "heom_ff.cuh"
#include "heom_grid.cuh"
#include "heom_tile.cuh"

namespace heom {

struct PersistOut {
    int iterations;
    int status;
    double nr;   // ||r||^2 at exit
    double bn;   // ||b||^2
};

template <class R>
struct PersistArgs {
    DevView<R> v;
    const cx<R> *b;  // columns col of [rows][B]
    cx<R> *x;
    int64_t B, col;
    int set;         // the column's parameter set
    const cx<R> *shift;  // [1] or null
    R aug;
    int precond;
    cx<R> *r, *rh, *p, *vv, *ph, *sh, *t, *xw;
    float4 *phf, *shf;  // FP64 solve: float-float copies of ph and sh (the apply operands)
    GridBar *bar;
    long long wait_cycles;  // bound of every grid-barrier wait (SM clock cycles)
    double tol;
    int max_iter, stall_iters;
    int local;         // own rows of the vectors in shared memory, local_off bytes from its start
    int local_off;
    PersistOut *out;
};

namespace {

constexpr int kPersThreads = 512;
constexpr size_t kPersSmem = 224 * 1024;  // of 227 KB: the kernel has static arrays too
constexpr int kPersVals = 3;  // numbers a barrier exchanges

// Load written earlier in this launch by another CTA: through L2 (ld.global.cg), never the
// non-coherent read-only path.
template <class R>
__device__ __forceinline__ cx<R> ld_l2(const cx<R> *p) {
    if constexpr (sizeof(R) == 8) {
        const double2 t = __ldcg(reinterpret_cast<const double2 *>(p));
        return cx<R>{t.x, t.y};
    } else {
        const float2 t = __ldcg(reinterpret_cast<const float2 *>(p));
        return cx<R>{t.x, t.y};
    }
}

// y = (M + shift) X at one item (single column), from the item's program
template <class R>
__device__ __forceinline__ cx<R> prog_apply(const ProgSmem<R> &ps, int it, const cx<R> *X,
                                            cx<R> shift) {
    const int j0 = ps.item[it], j1 = ps.item[it + 1];
    cx<R> acc = (ps.coef[j0] + shift) * ld_l2(X + ps.src[j0]);
    for (int jj = j0 + 1; jj < j1; jj += 8) {
        cx<R> cf[8], xv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool ok = jj + u < j1;
            const int idx = ok ? jj + u : j1 - 1;
            cf[u] = ok ? ps.coef[idx] : cx<R>{R(0), R(0)};
            xv[u] = ld_l2(X + ps.src[idx]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) fma_to(acc, cf[u], xv[u]);
    }
    return acc;
}

// The same apply in float-float for the FP64 solve: float-float coefficients (the shift
// already folded into each item's first term) and a float-float copy of X, so that the
// multiply-adds run on the FP32 pipe instead of GB300's 1/64-rate FP64 pipe; about 48
// significant bits per product and sum.
// Terms from j0 on, up to j1, of an item; unevaluated {re hi, im hi, re lo, im lo}.
__device__ __forceinline__ float4 prog_apply_ff(const ProgSmem<double> &ps, int j0, int j1, const float4 *X) {
    const float4 *coef = reinterpret_cast<const float4 *>(ps.coef);
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    for (int jj = j0; jj < j1; jj += 8) {
        float4 c[8], x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool ok = jj + u < j1;
            const int idx = ok ? jj + u : j1 - 1;
            c[u] = ok ? coef[idx] : make_float4(0.f, 0.f, 0.f, 0.f);
            x[u] = __ldcg(X + ps.src[idx]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            ff_mac(rh, rl, c[u].x, c[u].z, x[u].x, x[u].z);
            ff_mac(rh, rl, -c[u].y, -c[u].w, x[u].y, x[u].w);
            ff_mac(ih, il, c[u].x, c[u].z, x[u].y, x[u].w);
            ff_mac(ih, il, c[u].y, c[u].w, x[u].x, x[u].z);
        }
    }
    return make_float4(rh, ih, rl, il);
}

// body(it, y) for every item of the block with y = its apply to X, the FP64 solve's in float-float. Where the block
// has two threads per item, each takes half of its terms (an item of a low tier has 25 and more, each load
// a trip to L2: the ranges that hold them set the pace of the whole grid).
template <class R, class F>
__device__ __forceinline__ void apply_items(const ProgSmem<R> &ps, int items, const cx<R> *X, const float4 *Xf, cx<R> shift,
                                            float4 *s_half, F &&body) {
    if constexpr (sizeof(R) == 8) {
        if (2 * items <= (int)blockDim.x) {
            const int half = blockDim.x / 2, hf = threadIdx.x >= half, it = threadIdx.x - hf * half;
            float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
            if (it < items) {
                const int j0 = ps.item[it], j1 = ps.item[it + 1], mid = (j0 + j1 + 1) / 2;
                q = hf ? prog_apply_ff(ps, mid, j1, Xf) : prog_apply_ff(ps, j0, mid, Xf);
                if (hf) s_half[it] = q;
            }
            __syncthreads();
            if (!hf && it < items) {
                const float4 o = s_half[it];
                ff_norm(q.x, q.z);
                ff_norm(q.y, q.w);
                ff_add(q.x, q.z, o.x, o.z);
                ff_add(q.y, q.w, o.y, o.w);
                body(it, ff_join(q));
            }
            return;
        }
        for (int it = threadIdx.x; it < items; it += blockDim.x)
            body(it, ff_join(prog_apply_ff(ps, ps.item[it], ps.item[it + 1], Xf)));
    } else {
        for (int it = threadIdx.x; it < items; it += blockDim.x) body(it, prog_apply(ps, it, X, shift));
    }
}

// Grid-wide sum of NV doubles: block sums, exchanged by the barrier. Only the first nw warps hold
// values. One warp per value adds them (each FP64 addition of a warp occupies its sub-partition's pipe for
// 64 cycles: a shuffle tree in every warp took more of them than everything else here).
template <int NV>
__device__ __forceinline__ bool grid_sum(double (&val)[NV], double *s_red, double *s_tot, GridBar *bar, BarState &gen,
                                         int nw, long long limit) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < nw) {
#pragma unroll
        for (int k = 0; k < NV; ++k) s_red[k * kPersThreads + threadIdx.x] = val[k];
    }
    __syncthreads();
    double mine = 0.0;
    if (warp < NV) {  // warp k adds value k: its warps' values lane by lane, then the lanes
        for (int w = 0; w < nw; ++w) mine += s_red[warp * kPersThreads + w * 32 + lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
        if (lane == 0) s_tot[warp] = mine;
    }
    __syncthreads();
    mine = threadIdx.x < NV ? s_tot[threadIdx.x] : 0.0;
    if (!grid_exchange(bar, gen, kPersVals, limit, NV, mine, s_tot, RedSum{})) return false;
#pragma unroll
    for (int k = 0; k < NV; ++k) val[k] = s_tot[k];
    return true;
}

// 1/x by Newton-Raphson (r <- r (2 - x r), written r + r (1 - x r)) from the FP32 reciprocal
// as seed: the seed's relative error (<= 2^-23) squares at each step, so two steps reach FP64
// rounding. An FP64 division is a long instruction sequence on GB300's narrow FP64 pipe; this
// is six FP64-pipe instructions. Outside the seed's range (and for 0, inf, NaN) the plain
// division is used.
__device__ __forceinline__ double nr_rcp(double x) {
    const double ax = fabs(x);
    if (!(ax > 1e-30 && ax < 1e30)) return 1.0 / x;
    double r = (double)__frcp_rn((float)x);
    double e = fma(-x, r, 1.0);
    r = fma(r, e, r);
    e = fma(-x, r, 1.0);
    return fma(r, e, r);
}
__device__ __forceinline__ cx<double> cplx_div(cx<double> a, cx<double> b) {
    const double inv = nr_rcp(b.re * b.re + b.im * b.im);
    return cx<double>{(a.re * b.re + a.im * b.im) * inv, (a.im * b.re - a.re * b.im) * inv};
}
__device__ __forceinline__ bool finite_c(cx<double> a) { return isfinite(a.re) && isfinite(a.im); }

template <class R>
__global__ void __launch_bounds__(kPersThreads) k_persist_bicg(PersistArgs<R> a) {
    BarState gen;
    // Krylov scalars are computed once per CTA by thread 0 and broadcast (every CTA derives
    // the same values from the same grid sums); redundant FP64 divisions in all 16 warps
    // would queue on the FP64 pipe
    __shared__ double s_sc[9];
    const DevView<R> &v = a.v;
    const int d2 = v.d2;
    const int n0 = __ldg(v.pers_ado + blockIdx.x), n1 = __ldg(v.pers_ado + blockIdx.x + 1);
    extern __shared__ __align__(16) unsigned char smem[];
    double *s_red = reinterpret_cast<double *>(smem);   // [kPersVals][threads]
    double *s_tot = s_red + kPersVals * kPersThreads;   // [4]
    float4 *s_half = reinterpret_cast<float4 *>(s_tot + 4);  // [threads / 2]
    cx<R> *s_pinv = reinterpret_cast<cx<R> *>(s_half + kPersThreads / 2);
    ProgSmem<R> ps = prog_layout<R>(v.pers_terms, v.pers_slots, v.pers_ados, d2,
                                    reinterpret_cast<unsigned char *>(s_pinv + (size_t)v.pers_ados * d2));
    build_programs<R, true>(v, ps, n0, n1, a.aug, a.set);
    const cx<R> shift = a.shift ? a.shift[a.col] : cx<R>{R(0), R(0)};
    const int items = (n1 - n0) * d2;
    const int64_t row0 = (int64_t)n0 * d2;
    // warps that hold elements (thread t takes items t, t + blockDim.x, ...)
    const int nw_act = max(1, min((int)(blockDim.x >> 5), (items + 31) >> 5));
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const int pp = it / d2, e = it - pp * d2;
        const int64_t n = n0 + pp;
        s_pinv[it] = a.precond ? precond_inv(v, n, e, a.set, damping_of(v, n, a.set), shift)
                               : cx<R>{R(1), R(0)};
    }
    __syncthreads();

    // The CTA's own rows of the vectors: in shared memory where they fit (a.local), so that the updates wait
    // for no load from L2; the operands of the applies, which other CTAs read, are global too.
    cx<R> *const loc = reinterpret_cast<cx<R> *>(smem + a.local_off);
    const auto own = [&](int k, cx<R> *g) { return a.local ? loc + (size_t)k * v.pers_ados * d2 : g + row0; };
    cx<R> *const r = own(0, a.r), *const rh = own(1, a.rh), *const p = own(2, a.p), *const vv = own(3, a.vv),
                *const t = own(4, a.t), *const x = own(5, a.xw),
                *const ph = sizeof(R) == 8 ? own(6, a.ph) : a.ph + row0,
                *const sh = sizeof(R) == 8 ? own(7, a.sh) : a.sh + row0;

    // ---- x = 0, r = b, rh = r, p = v = 0
    double val1[1] = {0.0};
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
        const cx<R> ri = a.b[(row0 + it) * a.B + a.col];
        x[it] = cx<R>{R(0), R(0)};
        r[it] = ri;
        rh[it] = ri;
        p[it] = cx<R>{R(0), R(0)};
        vv[it] = cx<R>{R(0), R(0)};
        val1[0] += (double)norm2(ri);
    }
    if constexpr (sizeof(R) == 8) {
        // float-float programs for the iteration: fold the shift into every item's first
        // (damping) term, then split the coefficients in place (16 bytes either way)
        __syncthreads();
        if (a.shift)
            for (int it = threadIdx.x; it < items; it += blockDim.x) {
                cx<R> &c0 = ps.coef[ps.item[it]];
                c0 = c0 + shift;
            }
        __syncthreads();
        float4 *cf = reinterpret_cast<float4 *>(ps.coef);
        for (int t = threadIdx.x; t < ps.item[items]; t += blockDim.x) cf[t] = ff_split(ps.coef[t]);
        __syncthreads();
    }
    const bool started = grid_sum<1>(val1, s_red, s_tot, a.bar, gen, nw_act, a.wait_cycles);
    // Thread 0 holds the scalars and takes the decisions, the same ones in every CTA (redundant FP64 operations of
    // 16 warps queue on the FP64 pipe); s_st < 0: go on
    __shared__ int s_st;
    double nr = val1[0];
    const double bn = nr, stop2 = a.tol * a.tol * bn;
    cx<double> rho{nr, 0.0}, rho_old{1.0, 0.0}, alpha{1.0, 0.0}, omega{1.0, 0.0};
    double best = nr, rhn = nr;  // rhn = ||rh||^2
    int best_it = 0, it_done = 0;
    // restart when rh has become nearly orthogonal to r: rh = r, p = r; beta = (rho / rho_old)(alpha / omega)
    const auto next_scalars = [&](int iter) {
        const bool rs = iter > 1 && norm2(rho) < kRestartTau2 * rhn * nr;
        if (rs) {
            rho = cx<double>{nr, 0.0};
            rhn = nr;
        }
        const cx<double> bb = cplx_div(rho, rho_old) * cplx_div(alpha, omega), bo = bb * omega;
        s_sc[0] = rs ? 1.0 : 0.0;
        s_sc[1] = bb.re;
        s_sc[2] = bb.im;
        s_sc[3] = -bo.re;
        s_sc[4] = -bo.im;
    };
    if (threadIdx.x == 0) {
        s_st = !started ? HEOM_ETIMEOUT : nr <= stop2 ? 0 : -1;
        if (s_st < 0) next_scalars(1);
    }
    __syncthreads();
    int status = s_st;
    for (int iter = 1; status < 0 && iter <= a.max_iter; ++iter) {
        const bool restart = __double2hiint(s_sc[0]) != 0;
        // ---- p = r + beta (p - omega v), ph = P^-1 p
        const cx<R> bt{R(s_sc[1]), R(s_sc[2])}, nbo{R(s_sc[3]), R(s_sc[4])};
        for (int it = threadIdx.x; it < items; it += blockDim.x) {
            const int64_t i = row0 + it;
            const cx<R> ri = r[it];
            cx<R> pi = ri;
            if (!restart) {
                fma_to(pi, bt, p[it]);
                fma_to(pi, nbo, vv[it]);
            }
            if (restart) rh[it] = ri;
            p[it] = pi;
            const cx<R> phi = pi * s_pinv[it];
            ph[it] = phi;
            if constexpr (sizeof(R) == 8) a.phf[i] = ff_split(phi);
        }
        if (!grid_barrier(a.bar, gen, kPersVals, a.wait_cycles)) { status = HEOM_ETIMEOUT; break; }
        // ---- v = A ph, (rh, v)
        double d1[2] = {0.0, 0.0};
        apply_items<R>(ps, items, a.ph, a.phf, shift, s_half, [&](int it, cx<R> y) {
            vv[it] = y;
            const cx<double> yd = cast<double>(y), wd = cast<double>(rh[it]);
            d1[0] = fma(wd.re, yd.re, fma(wd.im, yd.im, d1[0]));
            d1[1] = fma(wd.re, yd.im, fma(-wd.im, yd.re, d1[1]));
        });
        if (!grid_sum<2>(d1, s_red, s_tot, a.bar, gen, nw_act, a.wait_cycles)) { status = HEOM_ETIMEOUT; break; }
        if (threadIdx.x == 0) {
            const cx<double> rv{d1[0], d1[1]};
            s_st = norm2(rv) == 0.0 ? HEOM_EBREAKDOWN : -1;
            alpha = cplx_div(rho, rv);
            s_sc[5] = alpha.re;
            s_sc[6] = alpha.im;
        }
        __syncthreads();
        if (s_st >= 0) { status = s_st; it_done = iter; break; }
        const cx<R> al{R(s_sc[5]), R(s_sc[6])}, nal{-al.re, -al.im};
        for (int it = threadIdx.x; it < items; it += blockDim.x) {
            const int64_t i = row0 + it;
            cx<R> si = r[it];
            fma_to(si, nal, vv[it]);
            r[it] = si;
            const cx<R> shi = si * s_pinv[it];
            sh[it] = shi;
            if constexpr (sizeof(R) == 8) a.shf[i] = ff_split(shi);
        }
        if (!grid_barrier(a.bar, gen, kPersVals, a.wait_cycles)) { status = HEOM_ETIMEOUT; break; }
        // ---- t = A sh, (t, s), (t, t)
        double d2v[3] = {0.0, 0.0, 0.0};
        apply_items<R>(ps, items, a.sh, a.shf, shift, s_half, [&](int it, cx<R> y) {
            t[it] = y;
            const cx<double> yd = cast<double>(y), wd = cast<double>(r[it]);
            d2v[0] = fma(yd.re, wd.re, fma(yd.im, wd.im, d2v[0]));
            d2v[1] = fma(yd.re, wd.im, fma(-yd.im, wd.re, d2v[1]));
            d2v[2] = fma(yd.re, yd.re, fma(yd.im, yd.im, d2v[2]));
        });
        if (!grid_sum<3>(d2v, s_red, s_tot, a.bar, gen, nw_act, a.wait_cycles)) { status = HEOM_ETIMEOUT; break; }
        if (threadIdx.x == 0) {
            const double it2 = d2v[2] == 0.0 ? 0.0 : nr_rcp(d2v[2]);
            omega = cx<double>{d2v[0] * it2, d2v[1] * it2};
            s_st = finite_c(omega) && finite_c(alpha) ? -1 : HEOM_EBREAKDOWN;
            s_sc[7] = omega.re;
            s_sc[8] = omega.im;
        }
        __syncthreads();
        if (s_st >= 0) { status = s_st; it_done = iter; break; }
        // ---- x += alpha ph + omega sh, r = s - omega t, (rh, r), ||r||^2
        const cx<R> omr{R(s_sc[7]), R(s_sc[8])}, nomr{-omr.re, -omr.im};
        double d3[3] = {0.0, 0.0, 0.0};
        for (int it = threadIdx.x; it < items; it += blockDim.x) {
            const int64_t i = row0 + it;
            cx<R> xi = x[it], ri = r[it];
            fma_to(xi, al, ph[it]);
            fma_to(xi, omr, sh[it]);
            x[it] = xi;
            fma_to(ri, nomr, t[it]);
            r[it] = ri;
            const cx<double> rd = cast<double>(ri), hd = cast<double>(rh[it]);
            d3[0] = fma(hd.re, rd.re, fma(hd.im, rd.im, d3[0]));
            d3[1] = fma(hd.re, rd.im, fma(-hd.im, rd.re, d3[1]));
            d3[2] = fma(rd.re, rd.re, fma(rd.im, rd.im, d3[2]));
        }
        if (!grid_sum<3>(d3, s_red, s_tot, a.bar, gen, nw_act, a.wait_cycles)) { status = HEOM_ETIMEOUT; break; }
        it_done = iter;
        if (threadIdx.x == 0) {
            rho_old = rho;
            rho = cx<double>{d3[0], d3[1]};
            nr = d3[2];
            int next = -1;
            if (!isfinite(nr)) next = HEOM_EBREAKDOWN;
            else if (nr <= stop2) next = 0;
            // no new minimum for stall_iters iterations: stalled (or diverging); the result is
            // usable if it still improved on the start. Single large transients (a near
            // breakdown just after a restart) are allowed: the recursion often recovers.
            else if (nr < best) { best = nr; best_it = iter; }
            else if (iter - best_it >= a.stall_iters) next = nr < bn ? HEOM_ENOCONV : HEOM_EBREAKDOWN;
            s_st = next;
            if (next < 0) next_scalars(iter + 1);
        }
        __syncthreads();
        status = s_st;
    }
    for (int it = threadIdx.x; it < items; it += blockDim.x) a.x[(row0 + it) * a.B + a.col] = x[it];
    if (status < 0) status = HEOM_ENOCONV;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.out = PersistOut{it_done, status, nr, bn};
}

template <class R>
DevView<R> view_of_p(const heom_hier *h) {
    if constexpr (sizeof(R) == 8) return h->view64();
    else return h->view32();
}

template <class R>
size_t persist_smem(const DevView<R> &v) {
    return kPersVals * kPersThreads * sizeof(double) + 4 * sizeof(double) + kPersThreads / 2 * sizeof(float4) + (size_t)v.pers_ados * v.d2 * sizeof(cx<R>) +
           prog_smem_bytes<R>(v.pers_terms, v.pers_slots, v.pers_ados, v.d2) + 64;
}

}  // namespace

template <class R>
bool persist_ok(const heom_hier *h) {
    if (h->pers_ranges < 1 || h->pers_ranges > kBarMaxGrid) return false;
    const DevView<R> v = view_of_p<R>(h);
    return persist_smem(v) <= 200 * 1024;
}
template bool persist_ok<double>(const heom_hier *);
template bool persist_ok<float>(const heom_hier *);

// A persistent iteration takes 25 to 45 us a column whatever the hierarchy (its barriers), a batched one 70 us and
// more for all columns together (five launches, two of them waiting for the longest chain of neighbour entries), so the
// line follows the entries: 6 an ADO in the spin-boson model, 15 in the small charge-cavity model, 24 in the Anderson
// model. Stationary states, ms, one by one against together (FP64; mixed):
//   35 ADOs of 2 x 2:          2 columns 3.0 / 2.8, 3 4.3 / 2.8, 8 11.0 / 3.4; 2 5.5 / 9.6, 3 8.2 / 9.7, 8 21 / 9.7
//   charge-cavity, 60 iter.:   2 4.0 / 5.2, 5 9.6 / 5.4; 2 3.2 / 3.6, 5 7.5 / 3.7
//   25 ADOs of 4 x 4:          3 1.1 / 1.3, 4 1.3 / 1.5, 5 1.7 / 1.5, 8 2.5 / 1.5; 5 4.0 / 5.8, 6 4.8 / 5.8, 8 6.4 / 5.8
//   301 ADOs:                  3 5.2 / 6.8, 4 7.2 / 7.3, 5 8.6 / 8.2, 8 13.2 / 7.3; 5 14.2 / 33, 8 23 / 47
//   2,325 ADOs, uneven depths: 4 9.2 / 12.3, 6 14.4 / 17.5, 8 20.6 / 16.0; 5 24.1 / 28.9, 8 29.5 / 36.5
// Shifted systems (spectra, frequency by frequency) take few iterations together in FP32 too, mixed, two columns a
// frequency: 301 ADOs 6 columns 4.6 / 6.0, 8 6.4 / 6.1; 2,325 6 6.2 / 9.6, 8 8.2 / 6.3.
template <class R>
int64_t persist_max_cols(const heom_hier *h, bool shifted) {
    if (h->max_entries < 20) return 2;
    if (sizeof(R) == 8) return h->N < 1000 ? 4 : 6;
    return h->N < 100 ? 5 : shifted ? 6 : 8;
}
template int64_t persist_max_cols<double>(const heom_hier *, bool);
template int64_t persist_max_cols<float>(const heom_hier *, bool);

// One persistent BiCGStab solve of (M + shift + aug e00 tr) x = b from x = 0 for column col of b and x ([rows][B]).
template <class R>
heom_status bicgstab_persistent(heom_hier *h, const cx<R> *b, cx<R> *x, int64_t B, int64_t col,
                                const cx<R> *shift, R aug, double tol, int max_iter,
                                int stall_iters, int *iters, int *status, double *rel_res,
                                cudaStream_t s) {
    const DevView<R> v = view_of_p<R>(h);
    const int64_t rows = h->N * h->d2;
    const int G = h->pers_ranges;
    const size_t vec = ((size_t)rows * sizeof(cx<R>) + 255) & ~size_t(255);
    const size_t fvec = sizeof(R) == 8 ? (((size_t)rows * sizeof(float4) + 255) & ~size_t(255)) : 0;
    const size_t bytes = 8 * vec + 2 * fvec + 128 + grid_bar_bytes(G, kPersVals);
    heom_status st = ensure_ws(h->ws_pers, bytes);
    if (st != HEOM_OK) return st;
    char *base = (char *)h->ws_pers.p;
    PersistArgs<R> a{};
    a.v = v;
    a.b = b;
    a.x = x;
    a.B = B;
    a.col = col;
    a.set = (int)(col / (B / h->n_sets));
    a.shift = shift;
    a.aug = aug;
    a.precond = 1;
    cx<R> **vecs[8] = {&a.r, &a.rh, &a.p, &a.vv, &a.ph, &a.sh, &a.t, &a.xw};
    for (int i = 0; i < 8; ++i) *vecs[i] = (cx<R> *)(base + i * vec);
    if (fvec) {
        a.phf = (float4 *)(base + 8 * vec);
        a.shf = (float4 *)(base + 8 * vec + fvec);
    }
    a.out = (PersistOut *)(base + 8 * vec + 2 * fvec);
    a.bar = (GridBar *)((char *)a.out + 128);
    HEOM_CUDA(grid_bar_reset(a.bar, G, kPersVals, s));
    a.tol = tol;
    a.max_iter = max_iter;
    a.stall_iters = stall_iters;
    a.wait_cycles = wait_limit_cycles();
    size_t sm = persist_smem(v);
    const size_t loc = (size_t)8 * v.pers_ados * v.d2 * sizeof(cx<R>), off = (sm + 15) & ~size_t(15);
    if (off + loc <= kPersSmem) {
        a.local = 1;
        a.local_off = (int)off;
        sm = off + loc;
    }
    HEOM_CUDA(cudaFuncSetAttribute(k_persist_bicg<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    void *args[] = {&a};
    {
        Prof pr(sizeof(R) == 4 ? HEOM_KC_KRYLOV_APPLY32 : HEOM_KC_KRYLOV_APPLY64, s, 0.0, 0.0);
        HEOM_CUDA(cudaLaunchCooperativeKernel((const void *)k_persist_bicg<R>, dim3(G), dim3(kPersThreads),
                                              args, sm, s));
    }
    PersistOut o{};
    HEOM_CUDA(memcpy_counted(&o, a.out, sizeof(o), cudaMemcpyDeviceToHost, s));
    HEOM_CUDA(cudaStreamSynchronize(s));
    *iters = o.iterations;
    *status = o.status;
    *rel_res = o.bn > 0 ? std::sqrt(o.nr / o.bn) : 0.0;
    if (o.status == HEOM_ETIMEOUT)  // every CTA has left; the caller reports the column
        set_error("persistent BiCGStab: a grid-barrier wait ran out after %lld cycles",
                  (long long)a.wait_cycles);
    // launch accounting: two applies per iteration, ADO-applies as units
    prof_add(sizeof(R) == 4 ? HEOM_KC_KRYLOV_APPLY32 : HEOM_KC_KRYLOV_APPLY64,
             2.0 * o.iterations * (double)h->N, 2.0 * o.iterations * 3.0 * (double)rows * sizeof(cx<R>));
    return HEOM_OK;
}

template heom_status bicgstab_persistent<double>(heom_hier *, const cx<double> *, cx<double> *, int64_t, int64_t,
                                                 const cx<double> *, double, double, int, int, int *,
                                                 int *, double *, cudaStream_t);
template heom_status bicgstab_persistent<float>(heom_hier *, const cx<float> *, cx<float> *, int64_t, int64_t,
                                                const cx<float> *, float, double, int, int, int *,
                                                int *, double *, cudaStream_t);

}  // namespace heom
