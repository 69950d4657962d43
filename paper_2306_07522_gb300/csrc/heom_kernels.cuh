// Device building blocks shared by the kernels: the damping table, the block-local
// preconditioner and block reductions into per-column FP64 accumulators.
#pragma once

#include "heom_internal.h"

namespace heom {

// BiCGStab restart rule: when |(rh, r)| < tau ||rh|| ||r|| the shadow residual rh has lost
// its grip on the Krylov space (the Lanczos biorthogonality behind the method has broken
// down in all but name); the iteration restarts with rh = r, p = r. tau = 1e-10. A sparse
// right-hand side such as the trace row of the stationary-state system makes the initial
// rh = b a poor shadow vector, and without the restart the recursion can stagnate.
constexpr double kRestartTau2 = 1e-20;

// Per-column solver state; every field is FP64 (Krylov scalars, dots, residuals).
struct ColState {
    cx<double> rho_old, alpha, omega;      // BiCGStab scalars
    cx<double> acc_rv, acc_ts, acc_tt, acc_rr;  // dot-product accumulators
    double acc_nr;                          // ||r||^2 accumulator
    double bnorm2;                          // ||b||^2
    double rhn;                             // ||rh||^2 of the current shadow residual
    int active;                             // 1 while the column iterates
    int flag;                               // breakdown marker
    int restart;                            // this iteration restarts (rh = r, p = r)
    int pad_;
};

// The parameter set of batch column b: (map ? map[b] : b) / cps, where map gives the original
// column of each column of a compacted working layout (null: the layout is the original).
struct ColSets {
    int64_t cps;
    const int *map;
    __host__ __device__ ColSets(int64_t c, const int *m = nullptr) : cps(c), map(m) {}
    __device__ __forceinline__ int set(int64_t b) const {
        const uint32_t c = map ? (uint32_t)__ldg(map + b) : (uint32_t)b;  // batches stay below 2^21
        return cps == 1 ? (int)c : (int)(c / (uint32_t)cps);
    }
};

template <class R>
__device__ __forceinline__ cx<R> ldc(const cx<R> *p) {
    if constexpr (sizeof(R) == 8) {
        double2 t = __ldg(reinterpret_cast<const double2 *>(p));
        return cx<R>{t.x, t.y};
    } else {
        float2 t = __ldg(reinterpret_cast<const float2 *>(p));
        return cx<R>{t.x, t.y};
    }
}

// Whether parameter set `set` keeps ADO n (heom_set_truncation). Where every set keeps a leading run
// of ADOs -- always with a single kind of bath -- that is a comparison (v.set_end), else a
// look at the ADO's tiers.
struct Kept {
    const int32_t *tier = nullptr;
    int cap = 0;
    int64_t end = INT64_MAX;
    template <class R>
    __device__ __forceinline__ Kept(const DevView<R> &v, int set) {
        if (v.set_end) {
            end = __ldg(v.set_end + set);
        } else if (v.set_cap) {
            tier = v.ado_tier;
            cap = __ldg(v.set_cap + set);
        }
    }
    __device__ __forceinline__ bool operator()(int64_t n) const {
        if (n >= end) return false;
        if (!tier) return true;
        const int t = __ldg(tier + n);
        return (t & 0xffff) <= (cap & 0xffff) && (t >> 16) <= (cap >> 16);
    }
};

// damping sum_k count_k rate_k of ADO n in parameter set `set`
template <class R>
__device__ __forceinline__ cx<R> damping_of(const DevView<R> &v, int64_t n, int set) {
    return ldc(v.damp + n * v.n_sets + set);
}

// Inverse of the ADO-local diagonal: 1 / (L_s[e][e] - damp + shift), with L_s[e][e] the
// coefficient of element e on itself in the system superoperator (-i (H_rr - H_cc) without
// Lindblad terms); the undamped tier-0 ADO is given the smallest positive rate as damping so
// the inverse stays bounded.
template <class R>
__device__ __forceinline__ cx<R> precond_inv(const DevView<R> &v, int64_t n, int e, int set,
                                             const cx<R> &damp, cx<R> shift) {
    cx<R> loc = ldc(v.sdiag + (int64_t)e * v.n_sets + set) - damp + shift;
    if (n == 0) loc.re -= __ldg(v.floor + set);  // the only ADO without an occupied exponent
    const R inv = R(1) / norm2(loc);
    return cx<R>{inv * loc.re, -inv * loc.im};
}

// Complex Givens rotation zeroing b in (a, b): G = [c s; -conj(s) c] with c real, so that
// G (a, b) = (r, 0). Built from two reciprocal square roots: an FP64 division or square root
// is a long instruction sequence on GB300's narrow FP64 pipe. With ia = 1/|a| and
// inr = 1/sqrt(|a|^2 + |b|^2): c = |a| inr, s = (a / |a|) conj(b) inr, r = (a / |a|) nr.
__device__ __forceinline__ void givens_rot(cx<double> a, cx<double> b, double &c, cx<double> &s,
                                           cx<double> &r) {
    const double a2 = norm2(a), b2 = norm2(b);
    if (b2 == 0.0) { c = 1.0; s = cx<double>{0.0, 0.0}; r = a; return; }
    if (a2 == 0.0) {
        const double ib = rsqrt(b2);
        c = 0.0;
        s = ib * conj(b);
        r = cx<double>{b2 * ib, 0.0};
        return;
    }
    const double ia = rsqrt(a2), inr = rsqrt(a2 + b2);
    c = a2 * ia * inr;
    s = (ia * inr) * (a * conj(b));
    r = ((a2 + b2) * inr * ia) * a;
}

}  // namespace heom
