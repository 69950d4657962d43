"""Solver workspaces go to the process-wide cache with their hierarchy and come from it for the next one."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [1, 20])
def test_a_second_hierarchy_solves_without_new_device_memory(cols):
    import torch
    import paper_2306_07522_gb300 as heom
    heom.release_workspace_cache()
    prob = heom.problem_from_model(W.siam_model(tier=2))
    taken = []
    for _ in range(2):
        g = heom.build_hierarchy(prob)
        x = torch.zeros((g.n_ado, 4, 4) + ((cols,) if cols > 1 else ()), dtype=torch.complex128, device="cuda")
        before = heom.profile_allocs()["device_allocs"]
        heom.steady(g, x, tol=1e-10, prec=heom.FP64)
        taken.append(heom.profile_allocs()["device_allocs"] - before)
        del g
    assert taken[0] > 0 and taken[1] == 0


def test_a_second_hierarchy_solves_on_a_full_device():
    """What the first hierarchy's solve held is enough for the same solve of a second one."""
    import torch
    import paper_2306_07522_gb300 as heom
    heom.release_workspace_cache()
    torch.cuda.empty_cache()
    prob = heom.problem_from_model(W.siam_model(tier=3))

    def solve(x):
        g = heom.build_hierarchy(prob)
        hold = torch.empty(max(torch.cuda.mem_get_info()[0] - (64 << 20), 1), dtype=torch.uint8, device="cuda") if x.any() else None
        st, _ = heom.steady(g, x, tol=1e-6, max_iter=4, prec=heom.MIXED, raise_on_error=False)
        del hold
        return st

    x = torch.zeros((2325, 4, 4, 256), dtype=torch.complex128, device="cuda")  # 152 MB: the right-hand side too
    try:
        assert solve(x) in (heom.OK, heom.ENOCONV)
        assert bool(x.any())
        assert solve(x) in (heom.OK, heom.ENOCONV)  # 64 MB free beside the cache
    finally:
        torch.cuda.empty_cache()
        heom.release_workspace_cache()


def test_a_change_of_parameters_keeps_the_damping_tables():
    """64 sets of 2,325 ADOs: the tables of the damping sums take 3.6 MB, everything else that a change of parameters
    uploads less than 1 MB."""
    import numpy as np
    import paper_2306_07522_gb300 as heom
    sets = 64
    prob = heom.problem_from_model(W.siam_model(tier=3))
    g = heom.build_hierarchy(prob)
    args = [np.stack([a] * sets) for a in (prob["H"], np.concatenate([b["coef"] for b in prob["baths"]]),
                                           np.concatenate([b["rate"] for b in prob["baths"]]))]
    heom.set_params(g, *args)
    before = heom.profile_allocs()["device_bytes"]
    heom.set_params(g, *args)
    assert heom.profile_allocs()["device_bytes"] - before < 1 << 20
