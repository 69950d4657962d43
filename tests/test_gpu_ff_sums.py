"""Sums of float-float values (Sum3, the Arnoldi dot products' sums over threads) against exact ones.

The inputs are exact in FP64 (two FP32 words), so math.fsum gives the correctly rounded sum. Sum3's three levels keep
about 2^-70 of the terms' size and its value is rounded to FP64 twice more: 2^-52 of the terms' size. Sums of the
same values in float-float are off by up to 2^-47.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

_KERNEL = r"""
#include "heom_ff.cuh"
using namespace heom;
__global__ void k(int m, int n, const float4 *x, double *out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m) return;
    Sum3 s;
    for (int i = 0; i < n; ++i) {
        const float4 v = x[t * n + i];
        s.add(make_float2(v.x, v.y), make_float2(v.z, v.w));
    }
    out[2 * t] = s.x();
    out[2 * t + 1] = s.y();
}
extern "C" int run(int m, int n, const void *x, void *out) {
    k<<<(m + 63) / 64, 64>>>(m, n, (const float4 *)x, (double *)out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("n", [1, 2, 3, 8, 128])
def test_float_float_sums_are_exact_to_fp64(tmp_path, n):
    import torch
    import paper_2306_07522_gb300.build as build
    (tmp_path / "k.cu").write_text(_KERNEL)
    subprocess.run([os.path.join(build._cuda_home(), "bin", "nvcc"), "-shared", "-Xcompiler", "-fPIC", build.ARCH,
                    "-std=c++17", "-I" + build.CSRC, str(tmp_path / "k.cu"), "-o", str(tmp_path / "k.so")], check=True)
    lib = ctypes.CDLL(str(tmp_path / "k.so"))
    rng = np.random.default_rng(n)
    m = 96
    z = rng.standard_normal((m, n, 2)) * 10.0 ** rng.uniform(-6, 2, (m, n, 2))
    z[::3] -= z[::3].mean(1, keepdims=True)  # cancelling sums
    hi = z.astype(np.float32)
    lo = (z - hi).astype(np.float32)
    x = torch.from_numpy(np.concatenate([hi, lo], axis=2)).cuda().contiguous()
    out = torch.zeros((m, 2), dtype=torch.float64, device="cuda")
    assert lib.run(m, n, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr())) == 0
    v = hi.astype(np.float64) + lo.astype(np.float64)
    want = np.array([[math.fsum(v[t, :, c]) for c in (0, 1)] for t in range(m)])
    assert np.all(np.abs(out.cpu().numpy() - want) <= 2.0 ** -52 * np.abs(v).sum(1))
