"""The block reduction of the FP32 dot products at the shapes where it can go wrong: blocks of fewer rows than a step adds,
smaller than a warp, with a partial last warp, of one step more or less; one to four chunks of systems; threads that fold
their products and threads that do not.  Against the oracle's exact BURA value within the solve's own tolerance.
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


@pytest.mark.parametrize("k", [3, 7, 9, 12])
@pytest.mark.parametrize("points,per_sm", [(4, 0), (9, 0), (20, 1), (33, 0), (64, 1), (100, 0), (256, 0)])
def test_block_shapes(lib, k, points, per_sm):
    shape, tol = (127, 95), 1e-6
    nps = tuple(reversed(shape))
    f = W.rhs_uniform(nps, 94)
    e = tables.entry(0.5, k)
    o = lib.bura_default_options()
    o.sweeps = lib.BURA_SWEEP_GRID  # (the grid sweeps: a block is points x chunks)
    o.block_points, o.blocks_per_sm = points, per_sm
    plan = lib.bura_setup(shape, 0.5, k, options=o)
    try:
        u = torch.zeros(f.size, dtype=torch.float64, device="cuda")
        assert lib.bura_solve(plan, torch.from_numpy(f).cuda(), u, tol) == lib.BURA_OK
        torch.cuda.synchronize()
    finally:
        lib.bura_destroy(plan)
    ur = exact.bura_value(nps, f, e["c"], e["d"])
    assert np.linalg.norm(u.cpu().numpy() - ur) <= tol * np.linalg.norm(ur)


@pytest.mark.parametrize("points", [1, 3])
@pytest.mark.parametrize("precision", [0, 1])
def test_the_smallest_blocks(lib, points, precision):
    """Blocks of fewer threads than systems, in which no thread would hold some system's total: they take a thread each."""
    shape, k, tol = (31, 15), 7, 1e-6
    nps = tuple(reversed(shape))
    f = W.rhs_uniform(nps, 97)
    e = tables.entry(0.5, k)
    o = lib.bura_default_options()
    o.precision, o.sweeps, o.block_points = precision, lib.BURA_SWEEP_GRID, points
    plan = lib.bura_setup(shape, 0.5, k, options=o)
    try:
        u = torch.zeros(f.size, dtype=torch.float64, device="cuda")
        assert lib.bura_solve(plan, torch.from_numpy(f).cuda(), u, tol) == lib.BURA_OK
        torch.cuda.synchronize()
    finally:
        lib.bura_destroy(plan)
    ur = exact.bura_value(nps, f, e["c"], e["d"])
    assert np.linalg.norm(u.cpu().numpy() - ur) <= tol * np.linalg.norm(ur)
