"""FP32 apply of dense operators by block products against the same hierarchy's FP64 apply.

The FP64 path works term by term, so the two differ in order and arithmetic. An element is a sum
of at most K = 2 d (entries + 1) products; rounding each to FP32 keeps the error below
K x 2^-24 x sum |terms|, and sum |terms| is at most a small multiple of the largest element for
random inputs (taken as 8). The bound is over the whole vector.
"""
import numpy as np
import pytest

import workloads as W
from tests.helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def heom():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_2306_07522_gb300 as heom
    return heom


@pytest.mark.parametrize("batch", [1, 2, 3, 4, 5, 7, 8, 9, 16, 33])
@pytest.mark.parametrize("d", [8, 16, 24, 32])
def test_dense_apply_matches_fp64(heom, d, batch):
    import torch
    prob = W.random_raw_problem(d, [("RI", 1), ("I", 1)], [4], 2, 1, seed=d)
    g = heom.build_hierarchy(prob)
    shape = (g.n_ado, d, d) if batch == 1 else (g.n_ado, d, d, batch)
    rng = np.random.default_rng(batch)
    X = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)
    x = to_dev(X, torch.complex64)
    base = torch.full((x.numel() + 64,), complex(7.0, -7.0), dtype=torch.complex64, device="cuda")
    y = base[: x.numel()].view(shape)
    heom.apply(g, x, y)
    x64 = x.to(torch.complex128)
    ref = heom.apply(g, x64, torch.empty_like(x64))
    assert bool((base[x.numel():] == complex(7.0, -7.0)).all())
    entries = 8  # at most one raised and one lowered neighbour per exponent, of 2 + 4 (+ H)
    tol = 2 * d * entries * 8 * 2.0 ** -24
    assert float((y.to(torch.complex128) - ref).abs().max() / ref.abs().max()) < tol
    # a buffer that is only 8-byte aligned takes the element-wise loads
    b2 = torch.empty(x.numel() + 1, dtype=torch.complex64, device="cuda")
    x2 = b2[1:].view(shape)
    x2.copy_(x)
    assert torch.equal(heom.apply(g, x2, torch.empty_like(x)), y)
