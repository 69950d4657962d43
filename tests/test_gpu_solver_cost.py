"""What the stationary solver does beside its iterations stays small, read from the launch accounting."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _accounted(heom, f):
    """Launches and device time per kernel class of one call, after a first one."""
    f()
    heom.profile_enable(True)
    f()
    out = heom.profile_read()
    heom.profile_enable(False)
    return out


def test_residual_norms_take_no_pass_of_their_own():
    """One column of 29,317 ADOs, four sweeps: scaling, norms and corrections together take less than the FP64
    residuals (each of them reads two or three vectors once; the residual gathers 24 to 56 neighbour blocks per
    ADO)."""
    import torch
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(heom.problem_from_model(W.siam_model(Gamma=1.0, n_poles=6, tier=3)))
    assert g.n_ado == 29317
    x = torch.zeros((g.n_ado, g.d, g.d), dtype=torch.complex128, device="cuda")
    pr = _accounted(heom, lambda: heom.steady(g, x, tol=1e-10, max_iter=20, prec=heom.MIXED, raise_on_error=False))
    assert pr["residual_fp64"]["launches"] >= 2
    assert pr["other"]["ms"] < pr["residual_fp64"]["ms"]
