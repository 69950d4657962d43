"""Stationary states of a few parameter sets of uneven depth, one persistent solve per column up to eight
columns and the batched solver beyond, against each set's own hierarchy.

Both sides drive ||M x|| / ||x|| below 1e-10; the smallest non-zero decay rate of this model is of order 0.1 to 1,
so the states agree to 1e-8. What a set's truncation drops stays exactly zero.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
@pytest.mark.parametrize("sets", [2, 8, 9])
def test_few_truncated_sets_match_their_own_hierarchies(sets, prec):
    import torch
    import paper_2306_07522_gb300 as heom
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    tiers = [2] * ((sets + 1) // 2) + [1] * (sets // 2)
    probs = {t: heom.problem_from_model(W.siam_model(tier=t)) for t in (1, 2)}
    coef = np.concatenate([b["coef"] for b in probs[2]["baths"]])
    rate = np.concatenate([b["rate"] for b in probs[2]["baths"]])
    H = [probs[2]["H"] * (1.0 + 0.02 * s) for s in range(sets)]
    g = heom.build_hierarchy(probs[2])
    heom.set_params(g, np.stack(H), np.stack([coef] * sets), np.stack([rate] * sets))
    heom.set_truncation(g, [0] * sets, tiers)
    x = torch.zeros((g.n_ado, g.d, g.d, sets), dtype=torch.complex128, device="cuda")
    heom.steady(g, x, tol=1e-10, max_iter=4000, prec=getattr(heom, prec))
    for s, t in enumerate(tiers):
        own = heom.build_hierarchy(dict(probs[t], H=H[s]))
        y = torch.zeros((own.n_ado, g.d, g.d), dtype=torch.complex128, device="cuda")
        heom.steady(own, y, tol=1e-10, max_iter=4000, prec=heom.FP64)
        assert float((x[: own.n_ado, ..., s] - y).abs().max() / y.abs().max()) < 1e-8
        assert not bool(x[own.n_ado:, ..., s].abs().any())
