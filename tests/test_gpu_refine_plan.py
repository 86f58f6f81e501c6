"""The refinement plan of the one-launch solve against the graph of kernels (an explicit ring depth keeps it) at inner
reductions other than the default: the same refinement steps, also where the plan is longer than the counts found by
multiplication.
"""
import numpy as np
import pytest

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


@pytest.mark.parametrize("inner_rtol,tol,max_outer", [(0.5, 1e-3, 40), (0.1, 1e-6, 20), (1e-2, 1e-8, 12), (1e-7, 1e-6, 12)])
def test_same_refinement_steps(lib, inner_rtol, tol, max_outer):
    shape, k = (127, 63), 6
    f = torch.from_numpy(W.rhs_uniform(tuple(reversed(shape)), 92)).cuda()
    got = []
    for stages in (0, 2):
        o = lib.bura_default_options()
        o.inner_rtol, o.max_outer, o.tma_stages = inner_rtol, max_outer, stages
        plan = lib.bura_setup(shape, 0.5, k, options=o)
        try:
            u = torch.zeros_like(f)
            assert lib.bura_solve(plan, f, u, tol) == lib.BURA_OK
            torch.cuda.synchronize()
            st = lib.bura_get_stats(plan)
            got.append((st["outer"], st["iters"], st["launches"] == 2))
        finally:
            lib.bura_destroy(plan)
    assert got[0][2] and not got[1][2]
    assert got[0][0] == got[1][0] and abs(got[0][1] - got[1][1]) <= got[0][0], got  # (iterations: within one a step)
