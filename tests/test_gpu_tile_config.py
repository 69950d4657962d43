"""heom_set_tile_config and heom_autotune act where another kernel would otherwise take the call: dense FP32 operators
(block products) and RK4 of hierarchies that fit into shared memory.

The kernels add the same terms in different orders, so their FP32 results differ in some last bits
and agree to K 2^-24 of the terms' size, K = 2 d (entries + 1) products per element (taken as 8 times the largest
element, as in the dense apply's own test).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _dense(heom):
    """A chain of 41 ADOs of 8 x 8 with a dense coupling operator (the tiled kernel's term programs hold 4,096 terms:
    an ADO of 24 x 24 with dense operators has more, one of 8 x 8 with two neighbours 2,944)."""
    import torch
    g = heom.build_hierarchy(W.random_raw_problem(8, [("RI", 1)], [], 40, 0, seed=4))
    gen = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((g.n_ado, 8, 8, 64), dtype=torch.complex64, device="cuda", generator=gen)
    return g, x


def _apply(heom, g, x):
    import torch
    return heom.apply(g, x, torch.empty_like(x))


def test_pinned_tiling_runs_for_dense_operators():
    import torch
    import paper_2306_07522_gb300 as heom
    g, x = _dense(heom)
    dense = _apply(heom, g, x)
    heom.set_tile_config(g, 2, 0)
    tiled = _apply(heom, g, x)
    heom.set_tile_config(g, 1, 0)
    assert torch.equal(_apply(heom, g, x), tiled)  # the granularity does not change a bit
    assert not torch.equal(dense, tiled)
    assert float((dense - tiled).abs().max() / tiled.abs().max()) < 2 * 8 * 3 * 8 * 2.0 ** -24


def test_autotuner_times_and_keeps_what_it_reports():
    import torch
    import paper_2306_07522_gb300 as heom
    g, x = _dense(heom)
    dense = _apply(heom, g, x)
    res = heom.autotune(g, 64, heom.FP32)
    kept = _apply(heom, g, x)
    if res["tiled"]:
        heom.set_tile_config(g, res["ctas_per_sm"], res["variant"])
        assert torch.equal(kept, _apply(heom, g, x))
    else:
        assert torch.equal(kept, dense)
    assert all(t > 0 for t in res["candidates_us"])


@pytest.mark.parametrize("prec", ["complex128", "complex64"])
def test_pinned_tiling_runs_for_evolutions(prec):
    import torch
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(heom.problem_from_model(W.spin_boson_model(tier=3)))
    x = torch.zeros((g.n_ado, 2, 2, 32), dtype=getattr(torch, prec), device="cuda")
    x[0, 0, 0] = torch.linspace(0.1, 1.0, 32, device="cuda")
    x[0, 1, 1] = 1 - x[0, 0, 0]
    launches = []
    out = []
    for pin in (False, True):
        if pin:
            heom.set_tile_config(g, 2, 0)
        y = x.clone()
        heom.profile_enable(True)
        heom.evolve(g, y, 1e-3, 7)
        launches.append(heom.profile_read()["rk4"]["launches"])
        heom.profile_enable(False)
        out.append(y)
    assert launches == [1, 28]
    assert float((out[0] - out[1]).abs().max()) < 7 * 64 * (1.2e-16 if prec == "complex128" else 6e-8)
