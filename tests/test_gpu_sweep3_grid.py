"""BURA_SWEEP_GRID in 3-D: a plan that asks for the grid sweeps runs no staged one (the profile names the sweeps), and the two
agree.  Constant coefficients: both within tol of the oracle's exact value, so within 2 tol of one another; variable ones: the
same from the rigorous bound that the solver certifies (err_bound <= tol each).  The sweeps do the same operations per point
and group their dot products differently, so the iterations agree to one a refinement step.
"""
import numpy as np
import pytest

from oracle import exact, tables
from paper_1612_04846_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def lib():
    from paper_1612_04846_gb300 import build_lib, bura
    build_lib.build(verbose=False)
    return bura


@pytest.mark.parametrize("var", [False, True])
@pytest.mark.parametrize("shape,k", [((63, 63, 31), 4), ((127, 63, 47), 9)])
def test_grid_sweeps_are_the_grid_sweeps(lib, shape, k, var):
    nps, tol = tuple(reversed(shape)), 1e-6
    faces = W.block_lognormal_faces(nps, 8, 1e-2, 1.0, 5) if var else None
    fh = W.rhs_uniform(nps, 95)
    f = torch.from_numpy(fh).cuda()
    got = {}
    for sweeps in (lib.BURA_SWEEP_AUTO, lib.BURA_SWEEP_GRID):
        o = lib.bura_default_options()
        o.sweeps = sweeps
        plan = lib.bura_setup(shape, 0.5, k, faces=faces, options=o)
        try:
            u = torch.zeros_like(f)
            assert lib.bura_solve(plan, f, u, tol) == lib.BURA_OK
            torch.cuda.synchronize()
            st = lib.bura_get_stats(plan)
            lib.bura_set_profiling(plan, True)
            assert lib.bura_solve(plan, f, torch.zeros_like(f), tol) == lib.BURA_OK
            names = {e["name"] for e in lib.bura_get_profile(plan)}
            lib.bura_set_profiling(plan, False)
            got[sweeps] = (u.cpu().numpy(), st, names)
        finally:
            lib.bura_destroy(plan)
    (ua, sa, na), (ug, sg, ng) = got[lib.BURA_SWEEP_AUTO], got[lib.BURA_SWEEP_GRID]
    staged, grid = {"prolong_cheb_f32", "cheb_pre2_f32"}, {"prolong_add_f32", "residual_f32", "p_update_f32"}
    assert staged <= na and not grid & na
    assert grid <= ng and not staged & ng
    assert sa["outer"] == sg["outer"] and abs(sa["iters"] - sg["iters"]) <= sa["outer"]
    assert 0 <= sa["err_bound"] <= tol and 0 <= sg["err_bound"] <= tol
    assert np.linalg.norm(ua - ug) <= 2 * tol * np.linalg.norm(fh)
    if not var:
        e = tables.entry(0.5, k)
        ur = exact.bura_value(nps, fh, e["c"], e["d"])
        assert max(np.linalg.norm(ua - ur), np.linalg.norm(ug - ur)) <= tol * np.linalg.norm(ur)
