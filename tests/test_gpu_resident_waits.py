"""Failure detection of the one-launch solve with variable coefficients, whose only waits are those for the other CTAs of a
cluster: every wait outlasts a budget of one SM clock, so the solve reports BURA_ETIMEOUT (each phase is still waited for
under the default budget), and the plan then solves as before.
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


@pytest.mark.parametrize("shape,k", [((31, 31), 4), ((95, 63), 6)])
def test_exchange_wait_budget(lib, shape, k):
    nps = tuple(reversed(shape))
    f = torch.from_numpy(W.rhs_uniform(nps, 93)).cuda()
    u = torch.zeros_like(f)
    plan = lib.bura_setup(shape, 0.5, k, faces=W.block_lognormal_faces(nps, 4, 1e-2, 1.0, 6))
    try:
        assert lib.bura_solve(plan, f, u, 1e-6) == lib.BURA_OK
        torch.cuda.synchronize()
        assert lib.bura_get_stats(plan)["launches"] == 2
        first = u.cpu().numpy()
        lib.bura_set_tma_wait_cycles(plan, 1)
        with pytest.raises(lib.BuraError) as ei:
            lib.bura_solve(plan, f, u, 1e-6)
        assert ei.value.code == lib.BURA_ETIMEOUT
        torch.cuda.synchronize()
        lib.bura_set_tma_wait_cycles(plan, 0)
        assert lib.bura_solve(plan, f, u, 1e-6) == lib.BURA_OK
        torch.cuda.synchronize()
        assert np.array_equal(u.cpu().numpy(), first)
    finally:
        lib.bura_destroy(plan)
