"""Batched stationary states of truncated sets whose ADOs are not a leading run, on both sides of the size at
which the FP32 apply of an iteration changes from one element per thread to one row (320,000 elements), against
each set's own hierarchy.

Both sides drive ||M x|| / ||x|| below 1e-10. The slowest decay of this model comes from the cavity bath (its
coupling 0.01, its cutoff 0.2), so its rate is of order 1e-3 to 1e-2 and the states agree to 1e-10 / 1e-3 = 1e-7.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CAPS = [(2, 2), (1, 2), (2, 1), (1, 1)]


@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
@pytest.mark.parametrize("sets", [9, 26])
def test_sets_truncated_inside_the_order_match_their_own_hierarchies(sets, prec):
    import torch
    import paper_2306_07522_gb300 as heom
    probs = {c: heom.problem_from_model(W.charge_cavity_model(n_fock=2, tier_b=c[0], tier_f=c[1])) for c in CAPS}
    deep = probs[2, 2]
    coef = np.concatenate([b["coef"] for b in deep["baths"]])
    rate = np.concatenate([b["rate"] for b in deep["baths"]])
    caps = [CAPS[s % 4] for s in range(sets)]
    H = [deep["H"] * (1.0 + 0.01 * s) for s in range(sets)]
    g = heom.build_hierarchy(deep)
    assert (g.n_ado * g.d ** 2 * sets < 320e3) == (sets == 9)
    heom.set_params(g, np.stack(H), np.stack([coef] * sets), np.stack([rate] * sets))
    heom.set_truncation(g, [c[0] for c in caps], [c[1] for c in caps])
    x = torch.zeros((g.n_ado, g.d, g.d, sets), dtype=torch.complex128, device="cuda")
    heom.steady(g, x, tol=1e-10, max_iter=4000, prec=getattr(heom, prec))
    kb = sum(len(b["coef"]) for b in deep["baths"] if b["kind"] != "F")
    label = np.stack([heom.ado_label(g, n) for n in range(g.n_ado)])
    tb, tf = label[:, :kb].sum(1), label[:, kb:].sum(1)
    for s in list(range(5)) + [sets - 1]:
        keep = torch.from_numpy((tb <= caps[s][0]) & (tf <= caps[s][1])).to("cuda")
        own = heom.build_hierarchy(dict(probs[caps[s]], H=H[s]))
        assert int(keep.sum()) == own.n_ado
        y = torch.zeros((own.n_ado, g.d, g.d), dtype=torch.complex128, device="cuda")
        heom.steady(own, y, tol=1e-10, max_iter=4000, prec=heom.FP64)
        assert float((x[keep][..., s] - y).abs().max() / y.abs().max()) < 1e-7
        assert not bool(x[~keep][..., s].abs().any())
