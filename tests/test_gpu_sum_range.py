"""Sums of FP32 products over the whole range of FP32 values: the network's loss through its own entry point, and the
solver's dot products (heom_dots.cuh) through kernels of this file.

FP64 products of FP32 values are exact and do not overflow, so the sums are compared with FP64 ones. A sum of n such
products has a relative error of at most n 2^-53 in FP64 in any order; n stays below 2^11 here: 1e-12.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-30, 1e-25, 1e-17, 1e-8, 1.0, 1e15, 1e20, 1e30])
def test_loss_at_any_scale(scale):
    import torch
    import paper_2306_07522_gb300 as heom
    net = heom.Mlp([3, 8, 7], seed=1)
    net.set_params(np.zeros(net.n_params, np.float32))  # predicts zero: the loss is the mean of t^2
    rng = np.random.default_rng(5)
    t = (scale * rng.uniform(0.5, 2.0, (203, 7))).astype(np.float32)
    x = torch.from_numpy(rng.standard_normal((203, 3)).astype(np.float32)).cuda()
    _, loss = net.gradients(x, torch.from_numpy(t).cuda())
    assert abs(loss / np.mean(t.astype(np.float64) ** 2) - 1.0) < 1e-12


def test_loss_of_infinite_targets_is_infinite():
    import torch
    import paper_2306_07522_gb300 as heom
    net = heom.Mlp([3, 8, 7], seed=1)
    t = torch.ones((64, 7), device="cuda")
    t[5, 3] = float("inf")
    _, loss = net.gradients(torch.zeros((64, 3), device="cuda"), t)
    assert loss == float("inf")


_KERNEL = r"""
#include <cstring>
#include "heom_dots.cuh"
using namespace heom;
// one thread per pair of runs of n values: (re, im, |b|^2), the same in FP64, and whether FP32's range was left
__global__ void k(int m, int n, const cx<float> *a, const cx<float> *b, double *out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    ColDots<float> d;
    ColDots<double> w;
    for (int i = 0; i < n; ++i) {
        d.cross(a[t * n + i], b[t * n + i]);
        d.norm(b[t * n + i]);
        w.cross(cast<double>(a[t * n + i]), cast<double>(b[t * n + i]));
        w.norm(cast<double>(b[t * n + i]));
    }
    double v[3] = {d.c_re(), d.c_im(), d.n()};
    const bool left = !(isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]));
    if (left) wide_dots(v, b + t * n, a + t * n, 1, 0, n, n, n, 1, 1, Kept(DevView<float>{}, 0), false);
    const double o[7] = {v[0], v[1], v[2], w.c_re(), w.c_im(), w.n(), left ? 1.0 : 0.0};
    for (int i = 0; i < 7; ++i) out[t * 7 + i] = o[i];
}
extern "C" int run(int m, int n, const void *a, const void *b, void *out) {
    k<<<(m + 63) / 64, 64>>>(m, n, (const cx<float> *)a, (const cx<float> *)b, (double *)out);
    return (int)cudaDeviceSynchronize();
}
// the sums of `blocks` blocks of one column: runs of ne rows, nrun of them from every step-th on, in ADOs of d2 rows
__global__ void kw(int64_t B, int64_t q_end, int nrun, int ne, int d2, Kept kept, int conj_y, const cx<float> *y,
                   const cx<float> *w, double *out) {
    double v[3];
    wide_dots(v, y, w, B, (int64_t)blockIdx.x * nrun, q_end, (int64_t)gridDim.x * nrun, nrun, ne, d2, kept, conj_y);
    for (int i = 0; i < 3; ++i) out[blockIdx.x * 3 + i] = v[i];
}
extern "C" int rows(int blocks, int64_t B, int64_t q_end, int nrun, int ne, int d2, int64_t end, int conj_y,
                    const void *y, const void *w, void *out) {
    struct { const int32_t *tier; int cap; int64_t end; } k{nullptr, 0, end};
    static_assert(sizeof(k) == sizeof(Kept), "Kept");
    alignas(Kept) char room[sizeof(Kept)];
    memcpy(room, &k, sizeof(k));
    kw<<<blocks, 1>>>(B, q_end, nrun, ne, d2, *(const Kept *)room, conj_y, (const cx<float> *)y, (const cx<float> *)w,
                      (double *)out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def dots(tmp_path_factory):
    import paper_2306_07522_gb300.build as build
    d = tmp_path_factory.mktemp("dots")
    (d / "k.cu").write_text(_KERNEL)
    subprocess.run([os.path.join(build._cuda_home(), "bin", "nvcc"), "-shared", "-Xcompiler", "-fPIC", build.ARCH,
                    "-std=c++17", "-I" + build.CSRC, str(d / "k.cu"), "-o", str(d / "k.so")], check=True)
    return ctypes.CDLL(str(d / "k.so"))


@pytest.mark.parametrize("n", [1, 2, 33, 500])
def test_thread_dot_products_at_any_scale(dots, n):
    import torch
    rng = np.random.default_rng(n)
    scales = [1e-10, 1.0, 1e17, 1e18, 1e19, 1e21, 1e30]
    m = 8 * len(scales)
    s = np.repeat(scales, 8)[:, None]
    z = lambda: (rng.standard_normal((m, n)) + 1j * rng.standard_normal((m, n)))  # noqa: E731
    a, b = (s * z()).astype(np.complex64), (s * z()).astype(np.complex64)
    a[3], b[5] = 0, 0
    b[8:16, n // 2] = 1e25  # one large value among ordinary ones
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.zeros((m, 7), dtype=torch.float64, device="cuda")
    assert dots.run(m, n, ctypes.c_void_p(ta.data_ptr()), ctypes.c_void_p(tb.data_ptr()),
                    ctypes.c_void_p(out.data_ptr())) == 0
    o = out.cpu().numpy()
    assert np.isfinite(o).all()
    size = (np.abs(a.astype(complex)) * np.abs(b.astype(complex))).sum(1)  # of the terms of (re, im)
    assert np.all(np.abs(o[:, 0] - o[:, 3]) <= 1e-12 * size)
    assert np.all(np.abs(o[:, 1] - o[:, 4]) <= 1e-12 * size)
    assert np.all(np.abs(o[:, 2] - o[:, 5]) <= 1e-12 * o[:, 5])
    assert not o[:8, 6].any() and not o[16:24, 6].any() and o[-16:, 6].all() and o[8:16, 6].all()


def test_infinities_and_nan_stay_what_fp64_makes_of_them(dots):
    import torch
    a = np.ones((3, 4), np.complex64)
    b = np.full((3, 4), 2.0, np.complex64)
    b[0, 1], b[1, 2] = np.inf, np.nan
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    out = torch.zeros((3, 7), dtype=torch.float64, device="cuda")
    assert dots.run(3, 4, ctypes.c_void_p(ta.data_ptr()), ctypes.c_void_p(tb.data_ptr()),
                    ctypes.c_void_p(out.data_ptr())) == 0
    o = out.cpu().numpy()
    assert np.array_equal(o[:, :3], o[:, 3:6], equal_nan=True) and o[0, 2] == np.inf and np.isnan(o[1, 2])


@pytest.mark.parametrize("n_ado,d2,ne,nrun,blocks,kept", [(7, 16, 4, 28, 3, 7), (9, 4, 1, 85, 2, 5), (5, 36, 2, 3, 4, 5),
                                                          (1, 16, 16, 256, 1, 1), (3, 4, 4, 1, 5, 0)])
@pytest.mark.parametrize("conj_y", [0, 1])
def test_rows_of_a_block_formed_again(dots, n_ado, d2, ne, nrun, blocks, kept, conj_y):
    import torch
    rng = np.random.default_rng(n_ado)
    B, col, rows = 3, 1, n_ado * d2
    z = lambda: 1e25 * (rng.standard_normal((rows, B)) + 1j * rng.standard_normal((rows, B)))  # noqa: E731
    y, w = z().astype(np.complex64), z().astype(np.complex64)
    ty, tw = torch.from_numpy(y).cuda(), torch.from_numpy(w).cuda()
    out = torch.zeros((blocks, 3), dtype=torch.float64, device="cuda")
    assert dots.rows(blocks, ctypes.c_int64(B), ctypes.c_int64(rows // ne), nrun, ne, d2, ctypes.c_int64(kept), conj_y,
                     ctypes.c_void_p(ty.data_ptr() + 8 * col), ctypes.c_void_p(tw.data_ptr() + 8 * col),
                     ctypes.c_void_p(out.data_ptr())) == 0
    o = out.cpu().numpy()
    block = np.arange(rows) // ne // nrun % blocks  # whose row it is
    use = np.arange(rows) < kept * d2
    for k in range(blocks):
        yk, wk = y[use & (block == k), col].astype(complex), w[use & (block == k), col].astype(complex)
        c = np.vdot(yk, wk) if conj_y else np.vdot(wk, yk)
        size = np.sum(np.abs(yk) * np.abs(wk))
        assert abs(o[k, 0] - c.real) <= 1e-12 * size and abs(o[k, 1] - c.imag) <= 1e-12 * size
        assert abs(o[k, 2] - np.sum(np.abs(yk) ** 2)) <= 1e-12 * np.sum(np.abs(yk) ** 2)
