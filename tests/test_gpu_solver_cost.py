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


@pytest.mark.parametrize("cols", [1, 2, 8])
@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
def test_columns_run_together_where_that_is_faster(prec, cols):
    """35 ADOs of 2 x 2: up to two columns take one launch each and sweep, more run together (eight columns one by
    one took 11 ms in FP64 and 21 ms in mixed precision, together 3.4 and 9.7)."""
    import torch
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(heom.problem_from_model(W.spin_boson_model(tier=4)))
    shape = (g.n_ado, 2, 2) + ((cols,) if cols > 1 else ())
    x = torch.zeros(shape, dtype=torch.complex128, device="cuda")
    pr = _accounted(heom, lambda: heom.steady(g, x, tol=1e-10, max_iter=4000, prec=getattr(heom, prec)))
    sweeps = pr["residual_fp64"]["launches"]  # one more than the solves
    applies = pr["krylov_apply_fp64" if prec == "FP64" else "krylov_apply_fp32"]["launches"]
    assert applies <= cols * sweeps if cols <= 2 else applies > 8 * sweeps
    assert float((x.reshape(g.n_ado, 2, 2, cols)[0, 0, 0] + x.reshape(g.n_ado, 2, 2, cols)[0, 1, 1] - 1).abs().max()) < 1e-9


@pytest.mark.parametrize("tier,cols,prec,one_by_one", [
    (1, 4, "FP64", True), (1, 5, "FP64", False), (1, 5, "MIXED", True), (1, 6, "MIXED", False),
    (2, 8, "MIXED", True), (2, 9, "MIXED", False), (3, 6, "FP64", True), (3, 7, "FP64", False)])
def test_columns_of_long_neighbour_lists(tier, cols, prec, one_by_one):
    """24 entries an ADO: the last number of columns that run one by one and the first that runs together."""
    import torch
    import paper_2306_07522_gb300 as heom
    g = heom.build_hierarchy(heom.problem_from_model(W.siam_model(tier=tier)))
    x = torch.zeros((g.n_ado, 4, 4, cols), dtype=torch.complex128, device="cuda")
    pr = _accounted(heom, lambda: heom.steady(g, x, tol=1e-10, max_iter=4000, prec=getattr(heom, prec)))
    applies = pr["krylov_apply_fp64" if prec == "FP64" else "krylov_apply_fp32"]["launches"]
    assert (applies <= cols * pr["residual_fp64"]["launches"]) == one_by_one
    assert float((torch.diagonal(x[0]).sum(-1) - 1).abs().max()) < 1e-9


@pytest.mark.parametrize("n_omega,one_by_one", [(3, True), (4, False)])
def test_few_frequencies_in_mixed_precision(n_omega, one_by_one):
    """Shifted systems, two columns a frequency: six run one by one, eight together (2,325 ADOs: eight take 8.2 ms one by
    one and 6.3 together)."""
    import numpy as np
    import torch
    import paper_2306_07522_gb300 as heom
    m = W.siam_model(tier=2)
    even, odd = (heom.build_hierarchy(heom.problem_from_model(m, p)) for p in (1, -1))
    x = torch.zeros((even.n_ado, 4, 4), dtype=torch.complex128, device="cuda")
    heom.steady(even, x, tol=1e-10, prec=heom.FP64)
    om = np.linspace(-12.0, 9.0, n_omega)
    out = []
    pr = _accounted(heom, lambda: out.append(heom.spectrum(odd, x, m.fermion_baths[0][0], om, tol=1e-8, max_iter=1500,
                                                           prec=heom.MIXED)[0]))
    applies = pr["krylov_apply_fp32"]["launches"]
    assert (applies <= 2 * n_omega * pr["residual_fp64"]["launches"]) == one_by_one
    ref = heom.spectrum(odd, x, m.fermion_baths[0][0], om, tol=1e-10, max_iter=500, prec=heom.SHIFTED)[0]
    assert float(np.abs(out[-1] - ref).max() / np.abs(ref).max()) < 1e-6
