"""Applies and RK4 steps on both sides of the sizes and shapes at which their layout changes: every column of a batch
against the same column alone.

Both sides add the same terms in different orders: an element has at most 2 d (K + 1) products (K exponents), so with
unit roundoff u the difference stays below 2 d (K + 1) u of the sum of the terms' sizes, taken as 8 times the largest
element; an RK4 run of n steps of size h adds n h |M| of that again, below one here.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

U = {"complex128": 2.0 ** -53, "complex64": 2.0 ** -24}


def _check(heom, g, k, batch, dtype):
    import torch
    d = g.d
    gen = torch.Generator(device="cuda").manual_seed(batch)
    x = torch.randn((g.n_ado, d, d, batch), dtype=getattr(torch, dtype), device="cuda", generator=gen)
    tol = 2 * d * (k + 1) * 8 * U[dtype]
    y = heom.apply(g, x, torch.empty_like(x))
    z = x.clone()
    heom.evolve(g, z, 1e-3, 2)
    for b in {0, batch // 2, batch - 1}:
        xb = x[..., b].contiguous()
        yb = heom.apply(g, xb, torch.empty_like(xb))
        assert float((y[..., b] - yb).abs().max() / yb.abs().max()) < tol, b
        heom.evolve(g, xb, 1e-3, 2)
        assert float((z[..., b] - xb).abs().max() / xb.abs().max()) < 2 * tol, b


@pytest.mark.parametrize("dtype", list(U))
@pytest.mark.parametrize("batch", [2, 3, 7, 8, 12, 16, 17, 33])
@pytest.mark.parametrize("d", [3, 5, 8, 16])
def test_dense_operators(d, batch, dtype):
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(W.random_raw_problem(d, [("RI", 2)], [4], 2, 2, seed=d))
    _check(heom, g, 6, batch, dtype)


@pytest.mark.parametrize("dtype", list(U))
@pytest.mark.parametrize("n_fock,batch", [(3, 1), (3, 2), (3, 5), (3, 6), (4, 2), (4, 3), (4, 4), (6, 1), (6, 2), (12, 1)])
def test_sparse_operators(n_fock, batch, dtype):
    """Charge-cavity models of 790 ADOs: blocks of 6, 8, 12 and 24, on both sides of 160,000 elements."""
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(heom.problem_from_model(W.charge_cavity_model(n_fock=n_fock)))
    assert g.n_ado == 790
    if batch == 1:  # two equal columns take another layout
        import torch
        gen = torch.Generator(device="cuda").manual_seed(n_fock)
        x = torch.randn((g.n_ado, g.d, g.d), dtype=getattr(torch, dtype), device="cuda", generator=gen)
        y = heom.apply(g, x, torch.empty_like(x))
        two = torch.stack([x, x], -1).contiguous()
        ref = heom.apply(g, two, torch.empty_like(two))
        assert float((y - ref[..., 1]).abs().max() / y.abs().max()) < 2 * g.d * 16 * 8 * U[dtype]
        return
    _check(heom, g, 15, batch, dtype)


@pytest.mark.parametrize("dtype", list(U))
@pytest.mark.parametrize("n_fock,tier", [(3, 1), (5, 1), (12, 0)])
def test_smallest_blocks_of_one_column(n_fock, tier, dtype):
    """4 and 13 ADOs of 6 x 6, 10 x 10 and 24 x 24: one element per thread in FP32."""
    import torch
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(heom.problem_from_model(W.charge_cavity_model(n_fock=n_fock, tier_b=1 - tier, tier_f=tier)))
    gen = torch.Generator(device="cuda").manual_seed(n_fock)
    x = torch.randn((g.n_ado, g.d, g.d), dtype=getattr(torch, dtype), device="cuda", generator=gen)
    y = heom.apply(g, x, torch.empty_like(x)).to(torch.complex128)
    x64 = torch.stack([x, x], -1).to(torch.complex128).contiguous()
    ref = heom.apply(g, x64, torch.empty_like(x64))[..., 0]
    assert float((y - ref).abs().max() / ref.abs().max()) < 2 * g.d * 16 * 8 * U[dtype]
