"""The FP64 sweeps of 2-D constant-coefficient levels at the edges of their range: ragged and thin grids, even axes next to
odd ones, system counts whose thread rows do not divide a block; against the oracle's exact BURA value, and against the
general sweeps.
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


def _solve(lib, shape, k, f, tol, sweeps):
    o = lib.bura_default_options()
    o.precision = lib.BURA_PREC_FP64
    o.sweeps = sweeps
    plan = lib.bura_setup(shape, 0.5, k, options=o)
    try:
        u = torch.zeros(f.size, dtype=torch.float64, device="cuda")
        assert lib.bura_solve(plan, torch.from_numpy(f).cuda(), u, tol) == lib.BURA_OK
        torch.cuda.synchronize()
    finally:
        lib.bura_destroy(plan)
    return u.cpu().numpy()


@pytest.mark.parametrize("shape,k", [((127, 127), 3), ((255, 63), 5), ((31, 511), 7), ((383, 47), 8), ((191, 223), 9),
                                     ((95, 63), 11), ((127, 255), 12), ((63, 511), 10)])
def test_lean_sweeps(lib, shape, k):
    nps, tol = tuple(reversed(shape)), 1e-10
    f = W.rhs_uniform(nps, 81)
    e = tables.entry(0.5, k)
    u = _solve(lib, shape, k, f, tol, lib.BURA_SWEEP_AUTO)
    ur = exact.bura_value(nps, f, e["c"], e["d"])
    assert np.linalg.norm(u - ur) <= tol * np.linalg.norm(ur)  # what the stopping rule promises
    g = _solve(lib, shape, k, f, tol, lib.BURA_SWEEP_GRID)
    assert np.linalg.norm(u - g) <= 2 * tol * np.linalg.norm(ur)
