"""RK4 from shared memory (heom_evolve on hierarchies that fit) against the launch-per-stage path.

heom_evolve_noalloc always takes one launch per stage, so the two entry points give the two paths on
the same inputs. Both round differently at every multiply-add: over n steps of a stable evolution the
difference stays below n x 64 roundings of the largest element (FP64 1.1e-16, FP32 6e-8).
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


def _random(d, bosons, fermions, tb, tf, seed):
    return W.random_raw_problem(d, bosons, fermions, tb, tf, seed=seed)


CASES = {
    # one chunk of 32 elements with padding lanes; a few chunks; several CTAs per column
    "spin_boson_t1": lambda h: h.problem_from_model(W.spin_boson_model(tier=1)),
    "spin_boson_t4": lambda h: h.problem_from_model(W.spin_boson_model(tier=4)),
    "spin_boson_t8": lambda h: h.problem_from_model(W.spin_boson_model(tier=8)),
    "siam_t1": lambda h: h.problem_from_model(W.siam_model(tier=1)),
    "siam_t2": lambda h: h.problem_from_model(W.siam_model(tier=2)),
    # dense operators, every bosonic kind, odd block sizes
    "dense_d3": lambda h: _random(3, [("RI", 2), ("I", 1)], [4, 2], 2, 2, 5),
    "dense_d5": lambda h: _random(5, [("R", 1), ("I", 1)], [2], 2, 1, 6),
}


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("batch", [1, 2, 5, 19])
@pytest.mark.parametrize("name", list(CASES))
def test_resident_rk4_matches_stages(heom, name, batch, prec):
    import torch
    dt = torch.complex128 if prec == "c128" else torch.complex64
    g = heom.build_hierarchy(CASES[name](heom))
    shape = (g.n_ado, g.d, g.d) if batch == 1 else (g.n_ado, g.d, g.d, batch)
    if 3 * int(np.prod(shape)) * 16 > 16 << 20:
        pytest.skip("beyond the launch-per-stage entry's scratch")
    rng = np.random.default_rng(batch)
    X = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    x, y = to_dev(X, dt), to_dev(X, dt)
    steps, save = 13, 4
    traj = heom.evolve(g, x, 1e-3, steps, save)
    ref_traj = torch.empty_like(traj)
    heom.evolve_noalloc(g, y, 1e-3, steps, save, traj=ref_traj)
    tol = steps * 64 * (1.2e-16 if prec == "c128" else 6e-8)
    assert float((x - y).abs().max() / y.abs().max()) < tol
    assert float((traj - ref_traj).abs().max() / ref_traj.abs().max()) < tol


def test_resident_rk4_parameter_sets_and_long_runs(heom):
    """Columns of several sets, more steps than one launch takes, a snapshot interval that does not
    divide them."""
    import torch
    prob = heom.problem_from_model(W.spin_boson_model(tier=3))
    coef = np.concatenate([b["coef"] for b in prob["baths"]])
    rate = np.concatenate([b["rate"] for b in prob["baths"]])
    g = heom.build_hierarchy(prob)
    heom.set_params(g, np.stack([prob["H"] * s for s in (1.0, 0.5, 2.0)]),
                    np.stack([coef, 0.5 * coef, 0.2 * coef]), np.stack([rate, rate, 1.1 * rate]))
    X = np.zeros((g.n_ado, 2, 2, 6), complex)
    X[0, 0, 0] = np.linspace(0.1, 1.0, 6)
    X[0, 1, 1] = 1 - X[0, 0, 0]
    x, y = to_dev(X, torch.complex128), to_dev(X, torch.complex128)
    steps, save = 2500, 333
    traj = heom.evolve(g, x, 1e-3, steps, save)
    ref = torch.empty_like(traj)
    heom.evolve_noalloc(g, y, 1e-3, steps, save, traj=ref)
    assert float((x - y).abs().max()) < steps * 64 * 1.2e-16
    assert float((traj - ref).abs().max()) < steps * 64 * 1.2e-16
