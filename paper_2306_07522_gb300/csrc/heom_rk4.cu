// RK4 time stepping (package architecture: dynamics): one fused stage of classical RK4 per launch.
#include "heom_block.cuh"

namespace heom {

// One fused stage of classical RK4: k = M z_in, then
//   stage 1: acc = k,       z_out = y + dt/2 k
//   stage 2: acc += 2k,     z_out = y + dt/2 k
//   stage 3: acc += 2k,     z_out = y + dt k
//   stage 4: y += dt/6 (acc + k)
// The stage's update of the run of CW elements at i0 (column stride B), from k = M z_in.
template <class R, int CW, bool VEC>
__device__ __forceinline__ void rk4_update(int64_t i0, int64_t B, const cx<R> (&k)[CW], cx<R> *z_out, cx<R> *y,
                                           cx<R> *acc, R dt, int stage) {
    cx<R> yv[CW], av[CW];
    if (stage > 1) ld_row<R, CW, VEC>(acc + i0, B, av);
    ld_row<R, CW, VEC>(y + i0, B, yv);
    const R h = stage == 3 ? dt : R(0.5) * dt;
#pragma unroll
    for (int u = 0; u < CW; ++u) {
        if (stage < 4) {
            av[u] = stage == 1 ? k[u] : av[u] + R(2) * k[u];
            yv[u] = yv[u] + h * k[u];
        } else {
            yv[u] = yv[u] + (dt / R(6)) * (av[u] + k[u]);
        }
    }
    if (stage < 4) st_row<R, CW, VEC>(acc + i0, B, av);
    st_row<R, CW, VEC>((stage < 4 ? z_out : y) + i0, B, yv);
}

// one thread per run of elements and column
template <class R, class Ly>
__global__ void __launch_bounds__(256, Ly::VEC ? 3 : 1) k_rk4_stage(DevView<R> v, const cx<R> *__restrict__ z_in, cx<R> *z_out,
                                                   cx<R> *y, cx<R> *acc, int64_t B, ColSets cps, R dt, int stage) {
    constexpr int NE = Ly::NE;
    const auto s_ops = Ly::stage(v);
    const int64_t total = v.N * Ly::per_ado(v) * B;
    const bool small = total < (int64_t(1) << 31);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        int64_t q, b, n;
        int e0;
        run_col(t, B, small, q, b);
        Ly::pos(v, q, small, n, e0);
        const int set = cps.set(b);
        cx<R> x0[NE], k[NE];
        if (beyond_cap(v, n, set)) zero_rows<R, NE>(nullptr, B, x0, k);
        else Ly::apply(v, s_ops, z_in, n, e0, b, B, set, x0, k);
        rk4_update<R, NE, Ly::VEC>((n * v.d2 + e0) * B + b, B, k, z_out, y, acc, dt, stage);
    }
}

// the launches of point_ok: threadIdx.x over columns, threadIdx.y over elements
template <class R>
__global__ void __launch_bounds__(256) k_rk4_point(DevView<R> v, const cx<R> *__restrict__ z_in, cx<R> *z_out, cx<R> *y,
                                                   cx<R> *acc, int64_t B, ColSets cps, R dt, int stage) {
    const int b = blockIdx.y * blockDim.x + threadIdx.x, rows = (int)v.N * v.d2;
    const int row = blockIdx.x * blockDim.y + threadIdx.y;
    if (b >= B || row >= rows) return;
    const int n = row / v.d2, e = row - n * v.d2, set = cps.set(b);
    cx<R> x0[1], k[1];
    if (beyond_cap(v, n, set)) zero_rows<R, 1>(nullptr, B, x0, k);
    else k[0] = apply_point(v, z_in, n, e, b, B, set, x0[0]);
    rk4_update<R, 1, false>((int64_t)row * B + b, B, k, z_out, y, acc, dt, stage);
}

// a few columns: neighbour blocks staged through shared memory (heom_staged.cuh)
template <class R, int CW, bool BLOCK, int W>
__global__ void __launch_bounds__(512) k_rk4_staged(DevView<R> v, const cx<R> *__restrict__ z_in, cx<R> *z_out, cx<R> *y, cx<R> *acc,
                             int64_t B, ColSets cps, R dt, int stage, bool vec) {
    staged_items<R, CW, BLOCK, W>(v, B, cps, [&](bool in, int64_t n, int64_t b, int set, int g, cx<R> *ring,
                                                 const OpRec<R> *s_ops) {
        const bool cut = beyond_cap(v, n, set);
        cx<R> x0[CW], k[CW];
        apply_staged<R, CW, BLOCK, W>(v, s_ops, ring, z_in, in && !cut, n, g, b, B, set, vec, x0, k);
        if (!in || (BLOCK && g >= v.d2 / CW)) return;
        if (cut) zero_rows<R, CW>(nullptr, B, x0, k);
        const int64_t i0 = (n * v.d2 + g * CW) * B + b;
        if (vec) rk4_update<R, CW, true>(i0, B, k, z_out, y, acc, dt, stage);
        else rk4_update<R, CW, false>(i0, B, k, z_out, y, acc, dt, stage);
    });
}

template <class R>
cudaError_t launch_rk4_stage(const DevView<R> &v, const cx<R> *z_in, cx<R> *z_out, cx<R> *y,
                             cx<R> *acc, int64_t B, R dt, int stage, cudaStream_t s) {
    const ColSets cps(B / v.n_sets);
    const bool quad = quad_ok(v, B, z_in, z_out, y, acc);
    const StageGeom sg = stage_geom(v, B);
    if constexpr (sizeof(R) == 4)
        if (point_ok(v, B)) {
            const Geom g = make_geom(v.N * v.d2, B, 1 << 30);
            k_rk4_point<R><<<g.grid, g.block, 0, s>>>(v, z_in, z_out, y, acc, B, cps, dt, stage);
            return cudaGetLastError();
        }
    if (sg.cw && !quad) {
        const bool vec = row_vec<R>(B, z_in, z_out, y, acc);
#define CALL(CW, BLOCK, W) \
    return launch_staged(k_rk4_staged<R, CW, BLOCK, W>, sg, s, v, z_in, z_out, y, acc, B, cps, dt, stage, vec)
        HEOM_STAGE_DISPATCH(sg, CALL);
#undef CALL
    }
    const LayoutPick p = pick_layout(v, B, quad);
    const Geom g = flat_geom(v.N * v.d2 / p.ne * B);
#define CALL(Ly) k_rk4_stage<R, Ly><<<g.grid, g.block, p.smem, s>>>(v, z_in, z_out, y, acc, B, cps, dt, stage)
    HEOM_FLAT_DISPATCH(R, p, CALL);
#undef CALL
    return cudaGetLastError();
}
template cudaError_t launch_rk4_stage<double>(const DevView<double> &, const cx<double> *,
                                              cx<double> *, cx<double> *, cx<double> *, int64_t,
                                              double, int, cudaStream_t);
template cudaError_t launch_rk4_stage<float>(const DevView<float> &, const cx<float> *,
                                             cx<float> *, cx<float> *, cx<float> *, int64_t,
                                             float, int, cudaStream_t);


}  // namespace heom
