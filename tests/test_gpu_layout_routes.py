"""Apply layouts that a size or an operator's shape selects, each against another layout of the same hierarchy.

* FP64, one column, d = 2 and 4, from 38,912 ADOs on (a block per lane): against two equal columns (one or a few
  elements per thread), operators with one and with two non-zeros per row, whole and truncated. Both sides add the same
  terms, at most 2 x 2 x (2 K + 1) per element and K = 10 exponents, in another order: 84 2^-53 of the sum of their
  sizes, taken as 8 times the largest element.
* FP32, one column, real operators with two non-zeros per row (four elements per thread): against the FP64 apply,
  2 x 2 x (entries + 1) products per element, entries below 64: 260 2^-24 likewise.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SX, SZ, I2 = W.SX, W.SZ, W.I2
OPS = {
    (2, 1): SX,
    (2, 2): 0.8 * SX + 0.3 * SZ,
    (4, 1): np.kron(SX, I2),
    (4, 2): np.kron(SX, I2) + 0.4 * np.kron(I2, SX + 0 * SZ),
}


def _boson_problem(d, op, n_exp, tier):
    p = W.random_raw_problem(d, [("RI", n_exp)], [], tier, 0, seed=d)
    p["baths"][0]["op"] = op
    return p


@pytest.mark.parametrize("cut", [None, 6])
@pytest.mark.parametrize("d,width", list(OPS))
def test_block_per_lane_matches_two_columns(d, width, cut):
    import torch
    import paper_2306_07522_gb300 as heom
    op = OPS[d, width]
    assert max((op != 0).sum(0).max(), (op != 0).sum(1).max()) == width
    g = heom.build_hierarchy(_boson_problem(d, op, 10, 8))
    assert g.n_ado == 43758 >= 38912
    gen = torch.Generator(device="cuda").manual_seed(width)
    x = torch.randn((g.n_ado, d, d), dtype=torch.complex128, device="cuda", generator=gen)
    if cut is not None:
        heom.set_truncation(g, [cut], [0])
        kept = 8008  # C(16, 6): the tiers up to 6 come first
        x[kept:] = 0
    y = heom.apply(g, x, torch.full_like(x, complex(9.0, 9.0)))
    two = torch.stack([x, x], -1).contiguous()
    ref = heom.apply(g, two, torch.empty_like(two))
    assert torch.equal(ref[..., 0], ref[..., 1])
    assert float((y - ref[..., 0]).abs().max() / y.abs().max()) < 84 * 8 * 2.0 ** -53
    if cut is not None:
        assert not bool(y[kept:].abs().any()) and bool(y[:kept].abs().any())


@pytest.mark.parametrize("cut", [None, 2])
@pytest.mark.parametrize("d", [4, 8, 24])
def test_four_elements_per_thread_match_fp64(d, cut):
    import torch
    import paper_2306_07522_gb300 as heom
    op = np.kron(SX, np.eye(d // 2)) + 0.4 * np.kron(np.eye(d // 2), SX)
    assert (op != 0).sum(0).max() == 2 and not op.imag.any()
    g = heom.build_hierarchy(_boson_problem(d, op, 4, 4))
    gen = torch.Generator(device="cuda").manual_seed(d)
    x = torch.randn((g.n_ado, d, d), dtype=torch.complex64, device="cuda", generator=gen)
    if cut is not None:
        heom.set_truncation(g, [cut], [0])
        x[15:] = 0  # C(6, 4) ADOs up to tier 2
    y = heom.apply(g, x, torch.empty_like(x))
    x64 = x.to(torch.complex128)
    ref = heom.apply(g, x64, torch.empty_like(x64))
    assert float((y.to(torch.complex128) - ref).abs().max() / ref.abs().max()) < 260 * 8 * 2.0 ** -24
    if cut is not None:
        assert not bool(y[15:].abs().any())


@pytest.mark.parametrize("dtype", ["complex128", "complex64"])
@pytest.mark.parametrize("batch", [1, 2, 19])
@pytest.mark.parametrize("model", ["spin_boson", "siam"])
def test_evolution_route(model, batch, dtype):
    """Hierarchies that fit run all their steps in one launch; a fallback would make four launches a step."""
    import torch
    import paper_2306_07522_gb300 as heom
    m = W.spin_boson_model(tier=8) if model == "spin_boson" else W.siam_model(tier=2)
    g = heom.build_hierarchy(heom.problem_from_model(m))
    x = torch.zeros((g.n_ado, g.d, g.d) + ((batch,) if batch > 1 else ()), dtype=getattr(torch, dtype), device="cuda")
    x[0, 0, 0] = 1
    heom.profile_enable(True)
    heom.evolve(g, x, 1e-3, 6, 2)
    n = heom.profile_read()["rk4"]["launches"]
    heom.profile_enable(False)
    assert n == 1


@pytest.mark.parametrize("dtype", ["complex128", "complex64"])
def test_driven_sets_across_the_sample_chunks(dtype):
    """Three parameter sets under a drive for 1,100 steps in one call (the drive's samples are formed 512 steps at a
    time) and in calls of 90 steps, which never cross a chunk: the same bits."""
    import torch
    import paper_2306_07522_gb300 as heom
    prob = heom.problem_from_model(W.spin_boson_model(tier=3))
    coef = np.concatenate([b["coef"] for b in prob["baths"]])
    rate = np.concatenate([b["rate"] for b in prob["baths"]])
    g = heom.build_hierarchy(prob)
    heom.set_params(g, np.stack([prob["H"] * s for s in (1.0, 0.5, 2.0)]),
                    np.stack([coef, 0.5 * coef, 0.2 * coef]), np.stack([rate, rate, 1.1 * rate]))
    heom.set_drive(g, [W.SZ, W.SX])
    steps, piece = 1100, 90
    t = np.arange(2 * steps + 1)
    f = np.stack([np.sin(0.01 * t), 0.3 + 1e-4 * t])
    x = torch.zeros((g.n_ado, 2, 2, 6), dtype=getattr(torch, dtype), device="cuda")
    x[0, 0, 0] = torch.linspace(0.1, 1.0, 6, device="cuda")
    x[0, 1, 1] = 1 - x[0, 0, 0]
    y = x.clone()
    traj = heom.evolve_td(g, x, 5e-3, steps, f, 100)
    for s in range(0, steps, piece):
        n = min(piece, steps - s)
        heom.evolve_td(g, y, 5e-3, n, f[:, 2 * s:2 * (s + n) + 1])
    assert torch.equal(x, y) and torch.equal(traj[-1], x[0])
    assert float((x[..., 0] - x[..., 2]).abs().max()) > 1e-3  # the sets differ
