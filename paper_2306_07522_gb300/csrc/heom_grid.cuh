// Grid-wide barrier for cooperative launches (all CTAs resident) that also exchanges a few numbers,
// with a bounded wait.
#pragma once

#include "heom_internal.h"

namespace heom {

constexpr int kBarVals = 8;      // numbers a barrier can exchange
constexpr int kBarMaxGrid = 256; // CTAs
// What an inbox slot holds before its sender has arrived: the NaN of 64 one bits. A value that happens
// to be that NaN is sent as the default one.
constexpr unsigned long long kBarEmpty = ~0ull;

// Barrier state in global memory: `err` (a wait ran out), then the inboxes, [receiving CTA][3][vals][G] with
// vals the most numbers a barrier of the launch exchanges and G = gridDim.x.
struct GridBar {
    int err;
    int pad[31];
    unsigned long long slot[1];
};
// a thread's view of it
struct BarState {
    unsigned gen = 0;  // barriers passed
    int n1 = 0, n2 = 0;  // slots used in the last barrier and the one before it
};
inline size_t grid_bar_bytes(int G, int vals) { return 128 + (size_t)3 * vals * G * G * sizeof(unsigned long long); }
// before every launch
inline cudaError_t grid_bar_reset(GridBar *bar, int G, int vals, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(bar, 0, 128, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(bar->slot, 0xff, grid_bar_bytes(G, vals) - 128, s);
    return e;
}

// acquire-release suffices (__threadfence is the sequentially consistent fence)
__device__ __forceinline__ void grid_fence() { asm volatile("fence.acq_rel.gpu;\n" ::: "memory"); }

// Barrier over the grid: a thread returns once every CTA's threads have called it; what they wrote
// before is visible after it. Thread k < nv of each CTA contributes val, and s_out[k] (shared memory) becomes red
// (for which zero is neutral) over all CTAs' values, formed in the same order in every CTA; s_out may be
// read until the next call. nv <= vals, the same in every thread.
//
// No counter: every CTA sends its values to the inbox of every CTA and polls its own inbox, so arrival,
// notification and the exchange of the values take one store and one load. (A counter -- an atomic
// per CTA on one address, a poll of it by all, then a read of the values -- took 3.5 us a barrier on 152
// CTAs and 2.7 us for the values; slots that every CTA polls, without inboxes, took longer than that: all
// polls go to a few lines.) Inboxes are triple-buffered: a CTA empties its slots for the next barrier before
// it arrives at this one. They were last used three barriers earlier and nobody sends to them before
// this CTA has arrived here.
//
// Each wait is bounded by `limit` SM clock cycles (the library's wait limit: by default 4e9,
// about 2 s). A wait that runs out raises the shared error flag; every CTA that waits sees it and leaves
// too, so no CTA waits for one that has gone, and the launch ends on every CTA. Returns
// false in every thread of a CTA that must stop.
template <class Red>
__device__ __forceinline__ bool grid_exchange(GridBar *bar, BarState &st, int vals, long long limit, int nv, double val,
                                              double *s_out, Red red) {
    __shared__ int s_bad;
    __shared__ double s_mine[kBarVals];
    constexpr int U = kBarMaxGrid / 32;
    const int G = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, np = nv > 0 ? nv : 1;
    const size_t box = (size_t)vals * G;  // slots of one buffer
    unsigned long long *mine = bar->slot + (size_t)blockIdx.x * 3 * box, *now = bar->slot + (size_t)(st.gen % 3) * box,
                       *next = mine + (size_t)((st.gen + 1) % 3) * box;
    if (tid == 0) s_bad = 0;
    if (tid < nv) s_mine[tid] = val;
    if (warp < st.n2)
        for (int g = lane; g < G; g += 32) *(volatile unsigned long long *)(next + (size_t)warp * G + g) = kBarEmpty;
    __syncthreads();
    if (warp < np) {  // warp k sends and polls value k
        unsigned long long bits = nv > 0 ? (unsigned long long)__double_as_longlong(s_mine[warp]) : 0ull;
        if (bits == kBarEmpty) bits = 0x7ff8000000000000ull;
        grid_fence();  // what the CTA wrote, and its emptied slots, before its arrival
        for (int g = lane; g < G; g += 32)
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;"
                         ::"l"(now + (size_t)g * 3 * box + (size_t)warp * G + blockIdx.x), "l"(bits) : "memory");
        const unsigned long long *in = mine + (size_t)(st.gen % 3) * box + (size_t)warp * G;
        unsigned long long got[U];
#pragma unroll
        for (int u = 0; u < U; ++u) got[u] = lane + 32 * u < G ? kBarEmpty : 0ull;
        const long long t0 = clock64();
        for (;;) {
            bool all = true;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (got[u] == kBarEmpty)
                    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(got[u]) : "l"(in + lane + 32 * u) : "memory");
#pragma unroll
            for (int u = 0; u < U; ++u) all = all && got[u] != kBarEmpty;
            if (__all_sync(0xffffffffu, all)) break;
            int stop = 0;
            if (lane == 0 && clock64() - t0 > (limit < 20000 ? limit : 20000)) {  // long waits look at the flag
                if (clock64() - t0 > limit) atomicExch(&bar->err, 1);
                stop = *(volatile int *)&bar->err;
            }
            if (__shfl_sync(0xffffffffu, stop, 0)) {
                if (lane == 0) s_bad = 1;
                break;
            }
        }
        grid_fence();
        if (nv > 0) {
            double x = __longlong_as_double((long long)got[0]);  // beyond the grid: zero
#pragma unroll
            for (int u = 1; u < U; ++u)
                if (32 * u < G) x = red(x, __longlong_as_double((long long)got[u]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x = red(x, __shfl_down_sync(0xffffffffu, x, o));
            if (lane == 0) s_out[warp] = x;
        }
    }
    __syncthreads();
    ++st.gen;
    st.n2 = st.n1;
    st.n1 = np;
    return s_bad == 0;
}

struct RedSum {
    __device__ __forceinline__ double operator()(double a, double b) const { return a + b; }
};
struct RedMax {
    __device__ __forceinline__ double operator()(double a, double b) const { return fmax(a, b); }
};

__device__ __forceinline__ bool grid_barrier(GridBar *bar, BarState &st, int vals, long long limit) {
    return grid_exchange(bar, st, vals, limit, 0, 0.0, nullptr, RedSum{});
}

}  // namespace heom
