"""The smallest tolerance a one-column spectrum still reaches: the Arnoldi vectors are normalised in FP64 and kept in
float-float (48 bits), so residual estimates go down to about 1e-14; normalised in float-float they end above it."""
import numpy as np
import pytest

import workloads as W
from oracle import hierarchy as hy
from oracle import liouvillian as lv
from oracle import solvers as so

pytestmark = pytest.mark.gpu


def test_spectrum_of_301_ados_reaches_1e_14():
    import torch
    import paper_2306_07522_gb300 as heom
    m = W.siam_model(tier=2)
    prob = hy.model_to_problem(m)
    X = so.steady_state(lv.build_matrix(prob, hy.problem_hierarchy(prob)), 4)
    om = np.linspace(-15.0, 15.0, 31)
    odd = heom.build_hierarchy(heom.problem_from_model(m, -1))
    _, st, stats = heom.spectrum(odd, torch.from_numpy(X).cuda().contiguous(), m.fermion_baths[0][0], om, tol=1e-14,
                                 max_iter=300, prec=heom.SHIFTED, raise_on_error=False)
    assert st == heom.OK, max(s["residual"] for s in stats)
