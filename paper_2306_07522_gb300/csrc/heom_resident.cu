// RK4 of hierarchies that fit into shared memory: one thread-block cluster integrates one column over
// all steps in a single launch (heom_evolve, heom_evolve_td).
//
// Why. A stage of these systems is a few hundred to a few ten thousand multiply-adds; run as one launch
// per stage it costs a launch, the table walks of the general apply and a pass over four vectors in L2
// whatever its size (14.5 us per stage at 35 ADOs of 2 x 2). Here the stage vector stays in
// shared memory (a full copy in every CTA of the cluster, double-buffered: one cluster barrier per
// stage), y and the RK4 sum stay in registers, and the apply runs from a term program: for every output
// element the list of (source position, coefficient index), four bytes a term. What a term multiplies by
// is one of few values per parameter set (exponent, side, operator value), so the program holds the
// hierarchy's structure only, is built once on the host and serves all sets and both precisions.
//
// Elements are sorted by the kinds of their terms and cut into chunks of 32, a lane per element: the
// lanes of a warp then have lists of the same length and, in FP64, the same zero coefficient
// halves (left out as in RowAcc: the pipe retires two FP64 multiply-adds per clock and SM and is
// what bounds the larger systems). Chunks are spread over the cluster's SM sub-partitions by cost.
// Left and right products of one source element (diagonal operators) are one term.
//
// Measured, 1,000 steps of 35 ADOs of 2 x 2, FP64: 59 ms (one launch per stage) -> 6.8 ms, bound by the latency of
// dependent FP64 instructions; 50 steps of 37 sets of 301 ADOs of 4 x 4, FP64: 16.4 -> 2.3 ms, bound by
// the FP64 pipe; 20 steps of 25 ADOs, FP32: 1.7 -> 0.14 ms.
#include <algorithm>
#include <cstdint>
#include <map>
#include <numeric>
#include <tuple>
#include <vector>

#include "heom_rows.cuh"

namespace heom {

namespace {

constexpr int kResThreads = 512;      // launch bound (16 warps, 128 registers)
constexpr int kResMaxPerWarp = 4;     // chunks of a warp
// Columns of a launch: the grid bounds them, not the speed. 20 steps of 301 ADOs of 4 x 4 take, tiled or
// staged against here, 4.6 and 0.52 ms (FP64, one column), 76 and 21 ms (1,024 columns); 2.1 and 0.22 ms (FP32,
// one column), 9.3 and 5.6 ms (1,024 columns); from a few hundred columns on both sides grow with the columns.
constexpr int64_t kResMaxB = 65535;
constexpr size_t kResSmem = 225 * 1024;
constexpr int64_t kResMaxTerms = 1 << 18;
constexpr int64_t kResSteps = 2048;   // steps of one launch
constexpr int kResBatch = 4;          // terms whose loads are in flight together

__host__ __device__ inline size_t res_align(size_t b) { return (b + 15) & ~size_t(15); }

template <class R>
struct ResArgs {
    const uint32_t *prog;   // [row][32] records: source position | coefficient << 16, chunk by chunk
    const int32_t *elem;    // [chunks][32] element of a position, -1: padding
    const int32_t *sown;    // [chunks][32] coefficient of the element's own system term, 0: none
    const ResCoef *coef;    // [nc] after the zero coefficient; then nS system terms
    const int4 *slot;       // [C][warps][M] {chunk (-1: none), first program row, rows, row in shared memory}
    cx<R> *y;               // [N d2][B]
    cx<R> *traj;            // snapshots (null: none)
    const cx<R> *damp;      // [N][n_sets]
    const cx<R> *coefL, *coefR;  // [K][n_sets]
    const cx<R> *s_val;     // [nS][n_sets], or with a drive [sample][nS][n_sets]
    int64_t B, cps, step0, steps, save, s_stride;  // s_stride: elements from one sample to the next (0: no drive)
    R dt;
    int n_sets, nS, nc, d2, P, C;                  // P: positions
};

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// every thread of the cluster; what was stored before it (also to other CTAs' shared memory) is
// visible after it
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;\n" ::: "memory");
}
// *p of every CTA of the cluster = v
template <class R>
__device__ __forceinline__ void store_all(cx<R> *p, cx<R> v, int C) {
    if (C == 1) {
        *p = v;
        return;
    }
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    for (int r = 0; r < C; ++r) {
        unsigned ra;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(r));
        if constexpr (sizeof(R) == 8)
            asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(ra), "d"(v.re), "d"(v.im) : "memory");
        else
            asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(ra), "f"(v.re), "f"(v.im) : "memory");
    }
}

__device__ __forceinline__ void res_mac(cx<double> &s, cx<double> c, cx<double> x) {
#pragma unroll 1
    for (int k = once(nonzero(c.re)); k > 0; --k) {
        s.re = fma(c.re, x.re, s.re);
        s.im = fma(c.re, x.im, s.im);
    }
#pragma unroll 1
    for (int k = once(nonzero(c.im)); k > 0; --k) {
        s.re = fma(-c.im, x.im, s.re);
        s.im = fma(c.im, x.re, s.im);
    }
}
__device__ __forceinline__ void res_mac(cx<float> &s, cx<float> c, cx<float> x) { fma_to(s, c, x); }

template <class R, int M>
__global__ void __launch_bounds__(kResThreads) k_rk4_resident(const ResArgs<R> a) {
    extern __shared__ __align__(16) unsigned char res_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5, C = a.C;
    const unsigned rank = C > 1 ? cluster_rank() : 0;
    const int64_t b = blockIdx.x / C;
    const int set = (int)(b / a.cps);
    const int ncoef = 1 + a.nc + a.nS;
    cx<R> *coef = reinterpret_cast<cx<R> *>(res_smem);
    cx<R> *z = reinterpret_cast<cx<R> *>(res_smem + res_align(ncoef * sizeof(cx<R>)));
    uint32_t *prog = reinterpret_cast<uint32_t *>(z + 2 * (size_t)a.P);

    const auto sync = [&] {
        if (C > 1) cluster_sync();
        else __syncthreads();
    };
    const auto load_system = [&](int64_t sample) {
        for (int j = tid; j < a.nS; j += blockDim.x)
            coef[1 + a.nc + j] = ldc(a.s_val + sample * a.s_stride + (int64_t)j * a.n_sets + set);
    };
    for (int i = tid; i <= a.nc; i += blockDim.x) {
        cx<R> c{R(0), R(0)};
        if (i > 0) {
            const ResCoef q = a.coef[i - 1];
            cx<R> l{R(0), R(-1)}, r = l;
            if (q.k >= 0) {
                l = mul_mi(ldc(a.coefL + (int64_t)q.k * a.n_sets + set));
                r = mul_mi(ldc(a.coefR + (int64_t)q.k * a.n_sets + set));
            }
            if (q.lre != 0.0 || q.lim != 0.0) c = l * cx<R>{R(q.lre), R(q.lim)};
            if (q.rre != 0.0 || q.rim != 0.0) c = c + r * cx<R>{R(q.rre), R(q.rim)};
        }
        coef[i] = c;
    }
    load_system(0);
    // a warp's chunks: program into shared memory, y into registers
    int pos[M], len[M], el[M], so[M];
    const uint32_t *rec[M];
    cx<R> y[M], acc[M], dmp[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const int4 s = a.slot[((int)rank * warps + warp) * M + m];
        pos[m] = -1;
        len[m] = 0;
        el[m] = -1;
        so[m] = 0;
        y[m] = acc[m] = dmp[m] = cx<R>{R(0), R(0)};
        rec[m] = prog + s.w * 32 + lane;
        if (s.x < 0) continue;
        pos[m] = s.x * 32 + lane;
        len[m] = s.z;
        el[m] = a.elem[pos[m]];
        so[m] = a.sown[pos[m]];
        for (int t = 0; t < s.z; ++t) prog[(s.w + t) * 32 + lane] = a.prog[(size_t)(s.y + t) * 32 + lane];
        if (el[m] >= 0) {
            y[m] = a.y[(int64_t)el[m] * a.B + b];
            dmp[m] = ldc(a.damp + (int64_t)(el[m] / a.d2) * a.n_sets + set);
        }
    }
    sync();  // every CTA has started and its coefficients are there
    cx<R> own[M];
    const auto own_terms = [&] {
#pragma unroll
        for (int m = 0; m < M; ++m) {
            own[m] = coef[so[m]];
            own[m].re -= dmp[m].re;
            own[m].im -= dmp[m].im;
        }
    };
    own_terms();
#pragma unroll
    for (int m = 0; m < M; ++m)
        if (pos[m] >= 0) store_all(z + pos[m], y[m], C);
    sync();
    int cur = 0;
    for (int64_t step = 1; step <= a.steps; ++step) {
#pragma unroll 1
        for (int stage = 1; stage <= 4; ++stage) {
            if (a.s_stride && stage != 3) {  // sample 2 n, 2 n + 1 (twice), 2 n + 2 of step n
                load_system(2 * (step - 1) + stage / 2);
                __syncthreads();
                own_terms();
            }
            const cx<R> *zi = z + (size_t)cur * a.P;
            cx<R> *zo = z + (size_t)(cur ^ 1) * a.P;
#pragma unroll
            for (int m = 0; m < M; ++m) {
                if (pos[m] < 0) continue;  // the same for the whole warp
                cx<R> k{R(0), R(0)};
                res_mac(k, own[m], zi[pos[m]]);
                for (int t = 0; t < len[m]; t += kResBatch) {
                    cx<R> c[kResBatch], x[kResBatch];
#pragma unroll
                    for (int u = 0; u < kResBatch; ++u) {
                        const uint32_t q = t + u < len[m] ? rec[m][(t + u) * 32] : (uint32_t)pos[m];
                        c[u] = coef[q >> 16];
                        x[u] = zi[q & 0xffff];
                    }
#pragma unroll
                    for (int u = 0; u < kResBatch; ++u)
                        if (t + u < len[m]) res_mac(k, c[u], x[u]);
                }
                cx<R> zv;
                if (stage < 4) {
                    zv = y[m] + (stage == 3 ? a.dt : R(0.5) * a.dt) * k;
                    acc[m] = stage == 1 ? k : acc[m] + R(2) * k;
                } else {
                    zv = y[m] = y[m] + (a.dt / R(6)) * (acc[m] + k);
                }
                store_all(zo + pos[m], zv, C);
            }
            sync();
            cur ^= 1;
        }
        const int64_t at = a.step0 + step;
        if (a.traj && at % a.save == 0) {
#pragma unroll
            for (int m = 0; m < M; ++m)
                if (el[m] >= 0 && el[m] < a.d2) a.traj[(at / a.save * a.d2 + el[m]) * a.B + b] = y[m];
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m)
        if (el[m] >= 0) a.y[(int64_t)el[m] * a.B + b] = y[m];
}

// ------------------------------------------------------------------ the program (host)
// Chunks of 32 elements with their term lists, from the structure of the hierarchy and of its system
// terms. False: too large for any launch.
bool build_plan(const heom_hier *h, ResPlan &p) {
    const int d = h->d, d2 = h->d2;
    const size_t L = (size_t)h->N * d2;
    struct Item { int e, src, c; };  // output element, source element, coefficient (system terms: -1 - j)
    std::map<std::tuple<int, double, double, double, double>, int> index;
    p.coef.clear();
    const auto coef_of = [&](int k, cx<double> l, cx<double> r) {
        const auto key = std::make_tuple(k, l.re, l.im, r.re, r.im);
        const auto it = index.find(key);
        if (it != index.end()) return it->second;
        p.coef.push_back(ResCoef{l.re, l.im, r.re, r.im, k, 0});
        return index[key] = (int)p.coef.size();
    };
    // terms of one kind of entry: operator, exponent (raised: -1), factors
    std::map<std::tuple<int, int, int, int>, std::vector<Item>> kinds;
    const auto items_of = [&](const NbEntry &q) -> const std::vector<Item> & {
        const int k = q.dir > 0 ? -1 : q.k;
        auto &v = kinds[std::make_tuple((int)q.op, k, (int)q.mult_l, (int)q.mult_r)];
        if (!v.empty()) return v;
        const heom_c64 *O = h->ops.data() + (size_t)q.op * d2;
        const cx<double> none{0.0, 0.0};
        const auto add = [&](int e, int src, cx<double> l, cx<double> r) {
            if (k < 0) {  // both sides multiply by -i
                l = l + r;
                r = none;
            }
            if (norm2(l) != 0.0 || norm2(r) != 0.0) v.push_back(Item{e, src, coef_of(k, l, r)});
        };
        for (int r = 0; r < d; ++r)
            for (int c = 0; c < d; ++c)
                for (int l = 0; l < d; ++l) {  // left term O[r][l], right term O[l][c]
                    const heom_c64 ol = O[r * d + l], o2 = O[l * d + c], oc = O[c * d + c];
                    const cx<double> fl{q.mult_l * ol.re, q.mult_l * ol.im}, fr{q.mult_r * o2.re, q.mult_r * o2.im},
                        fc{q.mult_r * oc.re, q.mult_r * oc.im};
                    // left term r and right term c read the element itself: one term
                    add(r * d + c, l * d + c, fl, l == r ? fc : none);
                    if (l != c) add(r * d + c, r * d + l, none, fr);
                }
        if (v.empty()) v.push_back(Item{0, 0, 0});  // a zero operator: one term of coefficient zero
        return v;
    };
    // lists of all elements, one run per element
    std::vector<int32_t> ptr(L + 1, 0), own(L, 0);
    std::vector<const std::vector<Item> *> of_entry;
    of_entry.reserve(h->ent.size());
    for (int64_t n = 0; n < h->N; ++n) {
        for (int e = 0; e < d2; ++e)
            for (int j = h->s_ptr[e]; j < h->s_ptr[e + 1]; ++j) ptr[(size_t)(n * d2 + e) + 1] += h->s_src[j] != e;
        for (int32_t i = h->row_ptr[n]; i < h->row_ptr[n + 1]; ++i) {
            of_entry.push_back(&items_of(h->ent[i]));
            for (const Item &t : *of_entry.back()) ++ptr[(size_t)(n * d2 + t.e) + 1];
        }
        if (p.coef.size() + h->nS > 60000) return false;
    }
    int64_t total = 0;
    for (size_t i = 0; i < L; ++i) total += ptr[i + 1];
    if (total > kResMaxTerms) return false;
    for (size_t i = 0; i < L; ++i) ptr[i + 1] += ptr[i];
    std::vector<std::pair<int32_t, int32_t>> term((size_t)total);  // source element, coefficient
    std::vector<int32_t> fill(ptr.begin(), ptr.end() - 1);
    p.nc = (int)p.coef.size();
    p.nS = h->nS;
    for (int64_t n = 0; n < h->N; ++n) {
        for (int e = 0; e < d2; ++e)
            for (int j = h->s_ptr[e]; j < h->s_ptr[e + 1]; ++j) {
                if (h->s_src[j] == e) own[(size_t)(n * d2 + e)] = 1 + p.nc + j;
                else term[(size_t)fill[(size_t)(n * d2 + e)]++] = {(int32_t)(n * d2 + h->s_src[j]), 1 + p.nc + j};
            }
        for (int32_t i = h->row_ptr[n]; i < h->row_ptr[n + 1]; ++i)
            for (const Item &t : *of_entry[(size_t)i])
                term[(size_t)fill[(size_t)(n * d2 + t.e)]++] = {(int32_t)((int64_t)h->ent[i].nb * d2 + t.src), t.c};
    }
    // order: long lists first, lists whose terms have the same kinds (raised, exponent) together
    std::vector<uint64_t> key(L);
    for (size_t e = 0; e < L; ++e) {
        uint64_t x = 0;
        for (int32_t t = ptr[e]; t < ptr[e + 1]; ++t) {
            const int c = term[(size_t)t].second, kd = c == 0 || c > p.nc ? 0 : p.coef[(size_t)c - 1].k + 2;
            x = (x ^ (uint64_t)kd) * 0x9e3779b97f4a7c15ULL;
            x ^= x >> 29;
        }
        key[e] = x;
    }
    std::vector<int32_t> ord(L), at(L);
    std::iota(ord.begin(), ord.end(), 0);
    std::stable_sort(ord.begin(), ord.end(), [&](int32_t a, int32_t b) {
        const int32_t la = ptr[(size_t)a + 1] - ptr[(size_t)a], lb = ptr[(size_t)b + 1] - ptr[(size_t)b];
        return la != lb ? la > lb : key[(size_t)a] < key[(size_t)b];
    });
    for (size_t i = 0; i < L; ++i) at[(size_t)ord[i]] = (int32_t)i;
    p.chunks = (int)((L + 31) / 32);
    p.elem.assign((size_t)p.chunks * 32, -1);
    p.sown.assign((size_t)p.chunks * 32, 0);
    p.row.assign((size_t)p.chunks + 1, 0);
    p.prog.clear();
    for (size_t c = 0; c < (size_t)p.chunks; ++c) {
        const int32_t first = ord[c * 32];  // the longest of the chunk
        const size_t len = (size_t)(ptr[(size_t)first + 1] - ptr[(size_t)first]), base = p.prog.size();
        p.row[c + 1] = p.row[c] + (int)len;
        p.prog.resize(base + len * 32);
        for (size_t l = 0; l < 32; ++l) {
            const size_t q = c * 32 + l;
            for (size_t t = 0; t < len; ++t) p.prog[base + t * 32 + l] = (uint32_t)q;  // padding: zero times itself
            if (q >= L) continue;
            const size_t e = (size_t)ord[q];
            p.elem[q] = (int32_t)e;
            p.sown[q] = own[e];
            for (int32_t t = ptr[e]; t < ptr[e + 1]; ++t)
                p.prog[base + (size_t)(t - ptr[e]) * 32 + l] =
                    (uint32_t)at[(size_t)term[(size_t)t].first] | (uint32_t)term[(size_t)t].second << 16;
        }
    }
    return true;
}

// Cost of a chunk: FP64 multiply-adds, or FP32 instructions.
template <class R>
int chunk_cost(const ResPlan &p, int c) {
    const int len = p.row[(size_t)c + 1] - p.row[(size_t)c];
    return sizeof(R) == 8 ? 10 + 5 * len / 2 : 20 + 6 * len;  // FP64: multiply-adds; FP32: instructions
}

struct ResGeom {
    int C = 0, warps = 0, M = 0, rows = 0;
    int64_t load = 0;        // cost of the busiest sub-partition
    size_t smem = 0;
    std::vector<int4> slot;  // [C][warps][M]
};
// Chunks over the C CTAs' sub-partitions, longest first onto the least loaded.
template <class R>
bool assign(const ResPlan &p, int C, ResGeom &g) {
    const int per = (p.chunks + C - 1) / C;                       // chunks of a CTA
    g.C = C;
    g.warps = std::min(kResThreads / 32, (per + 3) / 4 * 4);      // whole rounds of the four sub-partitions
    g.M = (per + g.warps - 1) / g.warps;
    if (g.M == 3) g.M = 4;
    if (g.M > kResMaxPerWarp) return false;
    const int bins = C * 4, cap = g.warps / 4 * g.M;
    std::vector<int64_t> load((size_t)bins, 0);
    std::vector<int> cnt((size_t)bins, 0), rows((size_t)C, 0);
    g.slot.assign((size_t)C * g.warps * g.M, int4{-1, 0, 0, 0});
    for (int c = 0; c < p.chunks; ++c) {  // sorted: longest first
        int best = -1;
        for (int q = 0; q < bins; ++q) {  // neighbouring bins belong to different CTAs
            const int bin = (q % C) * 4 + q / C;
            if (cnt[(size_t)bin] < cap && (best < 0 || load[(size_t)bin] < load[(size_t)best])) best = bin;
        }
        if (best < 0) return false;
        const int cta = best / 4, sub = best % 4, i = cnt[(size_t)best]++;
        const int nw = g.warps / 4, warp = (i % nw) * 4 + sub, m = i / nw;
        const int len = p.row[(size_t)c + 1] - p.row[(size_t)c];
        g.slot[(size_t)(cta * g.warps + warp) * g.M + m] = int4{c, p.row[(size_t)c], len, rows[(size_t)cta]};
        rows[(size_t)cta] += len;
        load[(size_t)best] += chunk_cost<R>(p, c);
    }
    g.rows = *std::max_element(rows.begin(), rows.end());
    g.load = *std::max_element(load.begin(), load.end());
    g.smem = res_align((size_t)(1 + p.nc + p.nS) * sizeof(cx<R>)) + 2 * (size_t)p.chunks * 32 * sizeof(cx<R>) +
             (size_t)g.rows * 128;
    return g.smem <= kResSmem;
}

template <class R>
using ResKernel = void (*)(const ResArgs<R>);
template <class R>
ResKernel<R> kernel_of(int M) {
    return M == 1 ? k_rk4_resident<R, 1> : M == 2 ? k_rk4_resident<R, 2> : k_rk4_resident<R, 4>;
}

template <class R>
cudaLaunchConfig_t config_of(const ResGeom &g, int64_t B, cudaStream_t s, cudaLaunchAttribute &at) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(B * g.C), 1, 1);
    cfg.blockDim = dim3((unsigned)g.warps * 32, 1, 1);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)g.C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cfg;
}

// Cluster size: the least time of a stage, in cycles times the number of waves. A sub-partition takes
// about 64 cycles per warp FP64 multiply-add and, for want of warps, about 4 per FP32 instruction; a
// stage ends in a block barrier (about 100 cycles) or a cluster barrier with the stage vector's
// exchange (about 900).
template <class R>
heom_status pick_geom(const ResPlan &p, int64_t B, ResGeom &best, bool &found) {
    found = false;
    double best_t = 0.0;
    for (int C : {1, 2, 3, 4, 6, 8}) {
        if (C > 1 && (p.chunks + C - 1) / C < 2) break;
        ResGeom g;
        if (!assign<R>(p, C, g)) continue;
        const ResKernel<R> k = kernel_of<R>(g.M);
        HEOM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem));
        cudaLaunchAttribute at;
        const cudaLaunchConfig_t cfg = config_of<R>(g, B, nullptr, at);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            continue;
        }
        const double t = (double)((B + n - 1) / n) *
                         ((double)g.load * (sizeof(R) == 8 ? 64.0 : 4.0) + (C == 1 ? 100.0 : 900.0));
        if (!found || t < best_t) {
            best = g;
            best_t = t;
            found = true;
        }
    }
    return HEOM_OK;
}

}  // namespace

bool resident_ok(const heom_hier *h, int64_t B, int prec_bytes) {
    const int64_t L = h->N * h->d2;
    return !h->has_caps && B <= kResMaxB && (L + 31) / 32 * 32 * 2 * prec_bytes <= (int64_t)kResSmem && L <= 65536 - 32;
}

// Runs `steps` steps from step0 on; done = false when the hierarchy does not fit (nothing was changed).
template <class R>
heom_status resident_steps(heom_hier *h, cx<R> *y, int64_t B, double dt, int64_t step0, int64_t steps,
                           int64_t save, cx<R> *traj, const cx<R> *s_val, int64_t s_stride, bool *done,
                           cudaStream_t s) {
    *done = false;
    ResPlan &p = h->res;
    if (p.state == ResPlan::kNone) p.state = build_plan(h, p) ? ResPlan::kBuilt : ResPlan::kTooLarge;
    if (p.state == ResPlan::kTooLarge) return HEOM_OK;
    ResGeom g;
    bool found = false;
    heom_status st = pick_geom<R>(p, B, g, found);
    if (st != HEOM_OK || !found) return st;
    // device copy: program, elements, own terms, coefficients; then the slots of this launch
    const size_t o_elem = res_align(p.prog.size() * 4), o_sown = o_elem + p.elem.size() * 4,
                 o_coef = o_sown + p.sown.size() * 4, o_slot = res_align(o_coef + p.coef.size() * sizeof(ResCoef));
    if ((st = ensure_ws(h->ws_res, o_slot + (size_t)8 * kResThreads / 32 * kResMaxPerWarp * sizeof(int4))) != HEOM_OK)
        return st;
    char *base = (char *)h->ws_res.p;
    if (!p.uploaded) {
        const auto put = [&](size_t off, const void *src, size_t bytes) {
            return bytes ? memcpy_counted(base + off, src, bytes, cudaMemcpyHostToDevice, s) : cudaSuccess;
        };
        HEOM_CUDA(put(0, p.prog.data(), p.prog.size() * 4));
        HEOM_CUDA(put(o_elem, p.elem.data(), p.elem.size() * 4));
        HEOM_CUDA(put(o_sown, p.sown.data(), p.sown.size() * 4));
        HEOM_CUDA(put(o_coef, p.coef.data(), p.coef.size() * sizeof(ResCoef)));
    }
    HEOM_CUDA(memcpy_counted(base + o_slot, g.slot.data(), g.slot.size() * sizeof(int4), cudaMemcpyHostToDevice, s));
    DevView<R> v;
    if constexpr (sizeof(R) == 8) v = h->view64();
    else v = h->view32();
    ResArgs<R> a{};
    a.prog = (const uint32_t *)base;
    a.elem = (const int32_t *)(base + o_elem);
    a.sown = (const int32_t *)(base + o_sown);
    a.coef = (const ResCoef *)(base + o_coef);
    a.slot = (const int4 *)(base + o_slot);
    a.y = y;
    a.traj = traj;
    a.damp = v.damp;
    a.coefL = v.coefL;
    a.coefR = v.coefR;
    a.B = B;
    a.cps = B / h->n_sets;
    a.save = save;
    a.s_stride = s_stride;
    a.dt = (R)dt;
    a.n_sets = h->n_sets;
    a.nS = p.nS;
    a.nc = p.nc;
    a.d2 = h->d2;
    a.P = p.chunks * 32;
    a.C = g.C;
    const ResKernel<R> k = kernel_of<R>(g.M);
    HEOM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem));
    for (int64_t n = 0; n < steps; n += kResSteps) {
        a.step0 = step0 + n;
        a.steps = std::min(kResSteps, steps - n);
        a.s_val = s_stride ? s_val + 2 * n * s_stride : v.s_val;
        Prof pr(HEOM_KC_RK4, s, 4.0 * (double)a.steps * (double)h->N * (double)B,
                2.0 * (double)h->N * h->d2 * (double)B * sizeof(cx<R>));
        cudaLaunchAttribute at;
        const cudaLaunchConfig_t cfg = config_of<R>(g, B, s, at);
        HEOM_CUDA(cudaLaunchKernelEx(&cfg, k, a));
    }
    p.uploaded = true;
    *done = true;
    return HEOM_OK;
}
template heom_status resident_steps<double>(heom_hier *, cx<double> *, int64_t, double, int64_t, int64_t, int64_t,
                                            cx<double> *, const cx<double> *, int64_t, bool *, cudaStream_t);
template heom_status resident_steps<float>(heom_hier *, cx<float> *, int64_t, double, int64_t, int64_t, int64_t,
                                           cx<float> *, const cx<float> *, int64_t, bool *, cudaStream_t);

}  // namespace heom
