"""FP32 apply of operators of which about a third of the entries are non-zero, on both sides of the launch size from which
block products take it, against the same hierarchy's FP64 apply. Bound as for dense operators: K 2^-24 of 8 times the
largest element, K = 2 d (entries + 1) products of an element.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def thinned(d, density, tier=1, seed=3):
    """A random problem whose operators keep `density` of their entries (the same way round the diagonal where they are
    Hermitian)."""
    p = W.random_raw_problem(d, [("RI", 2)], [8], tier, tier, seed=seed)
    rng = np.random.default_rng(seed)
    for b in p["baths"]:
        keep = rng.random((d, d)) < density
        b["op"] = b["op"] * (keep if b["kind"] == "F" else np.triu(keep) | np.triu(keep).T)
    return p


@pytest.mark.parametrize("batch", [1, 4, 5, 16, 33, 64])
@pytest.mark.parametrize("d", [8, 16, 24, 32])
def test_thinned_operators_match_fp64(d, batch):
    import torch
    import paper_2306_07522_gb300 as heom
    p = thinned(d, 0.35)
    assert all(0.25 < np.count_nonzero(b["op"]) / d ** 2 < 0.5 for b in p["baths"])
    g = heom.build_hierarchy(p)
    shape = (g.n_ado, d, d) + ((batch,) if batch > 1 else ())
    gen = torch.Generator(device="cuda").manual_seed(batch)
    x = torch.randn(shape, dtype=torch.complex64, device="cuda", generator=gen)
    y = heom.apply(g, x, torch.empty_like(x))
    x64 = x.to(torch.complex128)
    ref = heom.apply(g, x64, torch.empty_like(x64))
    entries = 2 + 8  # one raised or lowered neighbour per exponent
    assert float((y.to(torch.complex128) - ref).abs().max() / ref.abs().max()) < 2 * d * (entries + 1) * 8 * 2.0 ** -24
