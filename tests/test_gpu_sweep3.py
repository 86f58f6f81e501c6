"""The TMA-staged 3-D sweeps at the edges of their range: the smallest staged level, ragged tiles on every axis, items of
8 to 128 planes, levels below the staged ones, one to four chunks of systems, smoothing of degree 2 and 3 (which keeps
a direction between the pre-smoothing steps).  Constant coefficients against the oracle's exact BURA value; variable ones
by the rigorous bound that every system's true residual gives (assembled matrix, FP64).
"""
import numpy as np
import pytest

from oracle import exact, operators, tables
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


def _options(lib, degree):
    o = lib.bura_default_options()
    o.smoother_degree = degree
    return o


SHAPES = [((63, 31, 31), 3, 2), ((79, 63, 111), 7, 3), ((127, 31, 63), 9, 2), ((95, 47, 31), 12, 2)]


@pytest.mark.parametrize("shape,k,degree", SHAPES)
def test_staged_constant(lib, shape, k, degree):
    nps, tol = tuple(reversed(shape)), 1e-6
    f = W.rhs_uniform(nps, 71)
    e = tables.entry(0.5, k)
    plan = lib.bura_setup(shape, 0.5, k, options=_options(lib, degree))
    try:
        u = torch.zeros(f.size, dtype=torch.float64, device="cuda")
        assert lib.bura_solve(plan, torch.from_numpy(f).cuda(), u, tol) == lib.BURA_OK
        torch.cuda.synchronize()
    finally:
        lib.bura_destroy(plan)
    ur = exact.bura_value(nps, f, e["c"], e["d"])
    assert np.linalg.norm(u.cpu().numpy() - ur) <= tol * np.linalg.norm(ur)


@pytest.mark.parametrize("shape,k,degree", SHAPES)
def test_staged_variable(lib, shape, k, degree):
    nps, tol = tuple(reversed(shape)), 1e-6
    faces = W.block_lognormal_faces(nps, 8, 1e-2, 1.0, 5)
    f = W.rhs_uniform(nps, 72)
    plan = lib.bura_setup(shape, 0.5, k, faces=faces, options=_options(lib, degree))
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
    shape, k = (63, 63, 63), 5
    f = torch.from_numpy(W.rhs_uniform(shape, 73)).cuda()
    u = torch.zeros_like(f)
    plan = lib.bura_setup(shape, 0.5, k)
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
