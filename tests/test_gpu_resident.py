"""The one-launch solve of small 2-D plans (vectors resident in shared memory, a cluster per system).

Shapes at the edges of its layout: one point, an even exact level, slabs thinner than the halo, a last slab with
more rows than the others, two CTAs per SM and one, inner iterates in shared memory and in global memory, clusters
of 16 and of 8, more systems than resident clusters.  Against the oracle's exact BURA value within the solve's own
tolerance, and against the graph of kernels (an explicit ring depth keeps it): the same counts of refinement steps,
iterations within one (the dot products are grouped differently).
"""
import numpy as np
import pytest

from oracle import direct, exact, operators, tables
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


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _solve(lib, shape, k, f, tol, **kw):
    o = lib.bura_default_options()
    for name, v in kw.items():
        setattr(o, name, v)
    plan = lib.bura_setup(shape, 0.5, k, options=o)
    try:
        u = torch.full_like(f, 3.0)
        rc = lib.bura_solve(plan, f, u, tol)
        torch.cuda.synchronize()
        return rc, u.cpu().numpy(), lib.bura_get_stats(plan)
    finally:
        lib.bura_destroy(plan)


@pytest.mark.parametrize("shape,k,tol", [((1, 1), 3, 1e-8), ((62, 50), 4, 1e-9), ((63, 63), 10, 1e-6), ((127, 31), 5, 1e-6),
                                         ((111, 95), 7, 1e-9), ((127, 447), 6, 1e-6), ((255, 255), 12, 1e-6),
                                         ((255, 255), 3, 1e-6), ((383, 255), 8, 1e-6), ((351, 255), 5, 1e-6)])
def test_one_launch_solve(lib, shape, k, tol):
    fh = W.rhs_uniform(tuple(reversed(shape)), 61)
    f = torch.from_numpy(fh).cuda()
    e = tables.entry(0.5, k)
    rc, u, st = _solve(lib, shape, k, f, tol)
    assert rc == lib.BURA_OK and st["launches"] == 2, st  # the solve and its output stage
    assert _rel(u, exact.bura_value(tuple(reversed(shape)), fh, e["c"], e["d"])) <= tol
    rc, _, sg = _solve(lib, shape, k, f, tol, tma_stages=2)
    assert rc == lib.BURA_OK and sg["launches"] > 2
    assert st["outer"] == sg["outer"] and abs(st["iters"] - sg["iters"]) <= 1
    assert 0 <= st["err_bound"] <= tol


def test_one_launch_outcomes(lib):
    """A zero right-hand side, the iteration caps, a right-hand side that is not finite; then the plan's next solve."""
    shape, k = (127, 127), 5
    n = 127 * 127
    f = torch.from_numpy(W.rhs_uniform((127, 127), 62)).cuda()
    o = lib.bura_default_options()
    plan = lib.bura_setup(shape, 0.5, k, options=o)
    try:
        u = torch.ones_like(f)
        assert lib.bura_solve(plan, torch.zeros_like(f), u, 1e-6) == lib.BURA_OK
        assert float(u.abs().max()) == 0.0
        bad = f.clone()
        bad[n // 2] = float("nan")
        with pytest.raises(lib.BuraError) as ei:
            lib.bura_solve(plan, bad, u, 1e-6)
        assert ei.value.code == lib.BURA_ENOTSPD
        assert lib.bura_solve(plan, f, u, 1e-6) == lib.BURA_OK
        V = torch.empty((k + 1, n), dtype=torch.float64, device="cuda")
        assert lib.bura_solve_systems(plan, f, V, 1e-6) == lib.BURA_OK
        c = torch.tensor(lib.bura_get_rational(plan, k)[0], device="cuda")
        assert _rel((c[:, None] * V).sum(0).cpu().numpy(), u.cpu().numpy()) <= 1e-14
    finally:
        lib.bura_destroy(plan)
    rc, _, st = _solve(lib, shape, k, f, 1e-6, max_iters=1, max_outer=3)
    assert rc == lib.BURA_ENOCONV and st["outer"] == 3 and st["iters"] == 3


@pytest.mark.parametrize("shape,k,tol", [((11, 9), 4, 1e-9), ((31, 31), 10, 1e-6), ((63, 23), 5, 1e-8), ((127, 31), 5, 1e-6),
                                         ((79, 79), 9, 1e-6), ((191, 191), 6, 1e-6)])
def test_one_launch_solve_variable(lib, shape, k, tol):
    """Variable coefficients: the tail of the hierarchy in CTA 0, its dense level, slabs of one row to all of them."""
    nps = tuple(reversed(shape))
    faces = W.block_lognormal_faces(nps, 4, 1e-2, 1.0, 6)
    fh = W.rhs_uniform(nps, 63)
    plan = lib.bura_setup(shape, 0.5, k, faces=faces)
    try:
        f = torch.from_numpy(fh).cuda()
        u = torch.zeros_like(f)
        assert lib.bura_solve(plan, f, u, tol) == lib.BURA_OK
        torch.cuda.synchronize()
        assert lib.bura_get_stats(plan)["launches"] == 2
    finally:
        lib.bura_destroy(plan)
    A, _ = operators.scaled_matrix(nps, faces)
    e = tables.entry(0.5, k)
    ur = direct.bura_sparse(A, fh, e["c"], e["d"])
    assert _rel(u.cpu().numpy(), ur) <= tol


@pytest.mark.parametrize("shape,k,var,kind", [((255, 255), 6, True, "CTA"), ((255, 127), 9, True, "CTA"),
                                              ((511, 255), 10, False, "FDIAG"), ((1023, 511), 7, False, "FDIAG")])
def test_resident_cycle(lib, shape, k, var, kind):
    """The lower V-cycle as one launch inside a larger plan against the coarse kernel it replaces: the same operations in
    the same order per point, so the same iterations and (to the rounding of the FP32 cycle) the same result."""
    nps, tol = tuple(reversed(shape)), 1e-6
    faces = W.block_lognormal_faces(nps, 8, 1e-2, 1.0, 7) if var else None
    f = torch.from_numpy(W.rhs_uniform(nps, 64)).cuda()
    got = []
    for coarse in (lib.BURA_COARSE_AUTO, getattr(lib, "BURA_COARSE_" + kind)):
        o = lib.bura_default_options()
        o.coarse_kernel = coarse
        o.tma_stages = 2  # (the graph of kernels)
        plan = lib.bura_setup(shape, 0.5, k, faces=faces, options=o)
        try:
            u = torch.zeros_like(f)
            assert lib.bura_solve(plan, f, u, tol) == lib.BURA_OK
            torch.cuda.synchronize()
            st = lib.bura_get_stats(plan)
            got.append((u.cpu().numpy(), st["iters"], st["outer"], st["launches"]))
        finally:
            lib.bura_destroy(plan)
    assert got[0][1:3] == got[1][1:3] and got[0][3] < got[1][3]
    assert _rel(got[0][0], got[1][0]) <= 1e-8
