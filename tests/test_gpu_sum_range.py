"""Sums of FP32 products over the whole range of FP32 values: the network's loss through its own entry point, and the
solver's per-thread dot products (heom_dots.cuh) through a kernel of this file.

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
#include "heom_dots.cuh"
using namespace heom;
// one thread per pair of runs of n values: (re, im, |b|^2, overflowed) and the same in FP64
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
    const DotVals v = d.overflowed() ? DotVals(w) : DotVals(d);
    const double o[7] = {v.re, v.im, v.n, w.c_re(), w.c_im(), w.n(), d.overflowed() ? 1.0 : 0.0};
    for (int i = 0; i < 7; ++i) out[t * 7 + i] = o[i];
}
extern "C" int run(int m, int n, const void *a, const void *b, void *out) {
    k<<<(m + 63) / 64, 64>>>(m, n, (const cx<float> *)a, (const cx<float> *)b, (double *)out);
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
