"""The TMA-staged 2-D sweeps with variable coefficients at the edges of their range: ragged tiles on both axes, thin grids
with the finest level alone above the coarse solver, one to four chunks of systems; against the rigorous bound that every
system's true residual gives (assembled matrix, FP64).
"""
import numpy as np
import pytest

from oracle import operators
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


@pytest.mark.parametrize("shape,k", [((255, 255), 3), ((319, 207), 7), ((1023, 31), 9), ((31, 511), 5), ((383, 447), 12)])
def test_staged_variable(lib, shape, k):
    nps, tol = tuple(reversed(shape)), 1e-6
    faces = W.block_lognormal_faces(nps, 8, 1e-2, 1.0, 5)
    f = W.rhs_uniform(nps, 74)
    plan = lib.bura_setup(shape, 0.5, k, faces=faces)
    try:
        V = torch.zeros((k + 1, f.size), dtype=torch.float64, device="cuda")
        assert lib.bura_solve_systems(plan, torch.from_numpy(f).cuda(), V, tol) == lib.BURA_OK
        torch.cuda.synchronize()
        c, d, _ = lib.bura_get_rational(plan, k)
        lam_lo = lib.bura_get_stats(plan)["lambda_lo"]
    finally:
        lib.bura_destroy(plan)
    A, _ = operators.scaled_matrix(nps, faces)
    V = V.cpu().numpy()
    bound = sum(c[j] * np.linalg.norm(f - (A @ V[j] - d[j] * V[j])) / (lam_lo - d[j]) for j in range(k + 1))
    assert bound <= 1.001 * tol * np.linalg.norm(f)  # the solver's own stopping rule, its residuals in another order


def test_staged_wait_budget(lib):
    """A wait budget far below a copy's latency: BURA_ETIMEOUT, and the plan solves again with the default budget."""
    shape, k = (511, 255), 6
    nps = tuple(reversed(shape))
    f = torch.from_numpy(W.rhs_uniform(nps, 75)).cuda()
    u = torch.zeros_like(f)
    plan = lib.bura_setup(shape, 0.5, k, faces=W.block_lognormal_faces(nps, 8, 1e-2, 1.0, 6))
    try:
        lib.bura_set_tma_wait_cycles(plan, 200)
        with pytest.raises(lib.BuraError) as ei:
            lib.bura_solve(plan, f, u, 1e-6)
        assert ei.value.code == lib.BURA_ETIMEOUT
        torch.cuda.synchronize()
        lib.bura_set_tma_wait_cycles(plan, 0)
        assert lib.bura_solve(plan, f, u, 1e-6) == lib.BURA_OK
    finally:
        lib.bura_destroy(plan)
