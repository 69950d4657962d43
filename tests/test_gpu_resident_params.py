"""RK4 from shared memory after a change of parameters: its term program is kept when the system terms keep their
pattern, rebuilt when they do not, and the values are the new ones either way (against the launch-per-stage path)."""
import numpy as np
import pytest

import workloads as W
from tests.helpers import to_dev

pytestmark = pytest.mark.gpu

STEPS = 5


def _evolve_both(heom, g, X):
    """(heom_evolve, heom_evolve_noalloc) results and the bytes the first copied to the device."""
    import torch
    x, y = to_dev(X, torch.complex128), to_dev(X, torch.complex128)
    heom.profile_enable(True)
    heom.evolve(g, x, 1e-3, STEPS)
    h2d, _ = heom.profile_copies()
    assert heom.profile_read()["rk4"]["launches"] == 1  # one launch for all steps
    heom.profile_enable(False)
    heom.evolve_noalloc(g, y, 1e-3, STEPS)
    return x, y, h2d


def test_program_follows_the_pattern_of_the_system_terms():
    import paper_2306_07522_gb300 as heom
    prob = heom.problem_from_model(W.siam_model(tier=2))
    coef = np.concatenate([b["coef"] for b in prob["baths"]])
    rate = np.concatenate([b["rate"] for b in prob["baths"]])
    g = heom.build_hierarchy(prob)
    rng = np.random.default_rng(3)
    X = rng.standard_normal((g.n_ado, 4, 4)) + 1j * rng.standard_normal((g.n_ado, 4, 4))
    _, _, built = _evolve_both(heom, g, X)
    mixing = np.zeros((4, 4))
    mixing[1, 2] = mixing[2, 1] = 0.7
    tol = STEPS * 64 * 1.2e-16  # n x 64 roundings of the largest element
    # the same pattern, new values; another pattern and back: only the launch's table of chunks (8 KB) is copied
    # when the pattern is the one before
    for H, c, kept in ((0.5 * prob["H"], 0.3 * coef, True), (prob["H"] + mixing, coef, False),
                       (prob["H"] + 2 * mixing, coef, True), (prob["H"], coef, False)):
        heom.set_params(g, H[None], c[None], rate[None])
        x, y, h2d = _evolve_both(heom, g, X)
        assert float((x - y).abs().max() / y.abs().max()) < tol
        assert (h2d <= 8192) == kept, (h2d, built)


def test_program_follows_drive_and_dissipation():
    import torch
    import paper_2306_07522_gb300 as heom
    prob = heom.problem_from_model(W.spin_boson_model(tier=3))
    g = heom.build_hierarchy(prob)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((g.n_ado, 2, 2)) + 1j * rng.standard_normal((g.n_ado, 2, 2))
    tol = STEPS * 64 * 1.2e-16
    x, y, _ = _evolve_both(heom, g, X)
    assert float((x - y).abs().max() / y.abs().max()) < tol
    heom.set_lindblad(g, [W.SM], [0.4])
    x, y, _ = _evolve_both(heom, g, X)
    assert float((x - y).abs().max() / y.abs().max()) < tol
    heom.set_drive(g, [W.SZ])
    # a drive of constant amplitude is the same as its operator in H
    x = to_dev(X, torch.complex128)
    heom.evolve_td(g, x, 1e-3, STEPS, np.full((1, 2 * STEPS + 1), 0.8))
    other = heom.build_hierarchy(dict(prob, H=prob["H"] + 0.8 * W.SZ))
    heom.set_lindblad(other, [W.SM], [0.4])
    y = to_dev(X, torch.complex128)
    heom.evolve_noalloc(other, y, 1e-3, STEPS)
    assert float((x - y).abs().max() / y.abs().max()) < tol
