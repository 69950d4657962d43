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


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
@pytest.mark.parametrize("batch", [1, 6, 64])
@pytest.mark.parametrize("d,density", [(8, 0.3), (16, 0.3), (24, 0.6), (32, 0.6)])
def test_infinities_and_nan_spread_over_couplings_only(d, density, batch, bad):
    """One input element is not finite: outputs that do not depend on it are what they are without it, bit for bit."""
    import torch
    import paper_2306_07522_gb300 as heom
    p = thinned(d, density)
    p["H"] = np.triu(np.tril(p["H"], 1), -1)
    g = heom.build_hierarchy(p)
    gen = torch.Generator(device="cuda").manual_seed(batch)
    x = torch.randn((g.n_ado, d, d, batch), dtype=torch.complex64, device="cuda", generator=gen)
    at = (g.n_ado // 2, d // 3, d // 2, batch // 2)

    def out(value, dtype):
        z = x.to(dtype)
        z[at] = value
        if batch == 1:
            z = z[..., 0].contiguous()
        return heom.apply(g, z, torch.empty_like(z))

    free = out(1.0, torch.complex128) == out(2.0, torch.complex128)  # outputs without a term of it
    assert 0 < int((~free).sum()) < free.numel() // 4
    with_bad, without = out(bad, torch.complex64), out(0.0, torch.complex64)
    assert bool(torch.isfinite(torch.view_as_real(with_bad[free])).all())
    assert torch.equal(with_bad[free], without[free])
