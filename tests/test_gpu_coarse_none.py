"""2-D variable coefficients without a coarse kernel (BURA_COARSE_NONE): such a plan has a level small enough for the dense
inverses but no kernel that uses them, so its set-up and bura_retarget have none to fill.  Against the rigorous bound that
every system's true residual gives (assembled matrix, FP64), before and after a retarget.
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


@pytest.mark.parametrize("shape,k,precision", [((31, 31), 5, 1), ((63, 47), 7, 1), ((31, 15), 4, 0)])
def test_variable_without_a_coarse_kernel(lib, shape, k, precision):
    nps, tol = tuple(reversed(shape)), 1e-6
    faces = W.block_lognormal_faces(nps, 4, 1e-2, 1.0, 6)
    f = W.rhs_uniform(nps, 91)
    A, _ = operators.scaled_matrix(nps, faces)
    o = lib.bura_default_options()
    o.precision = precision
    o.coarse_kernel = lib.BURA_COARSE_NONE
    plan = lib.bura_setup(shape, 0.5, k, faces=faces, options=o)
    try:
        for alpha in (0.5, 0.25):
            if alpha != 0.5:
                lib.bura_retarget(plan, alpha)
            V = torch.zeros((k + 1, f.size), dtype=torch.float64, device="cuda")
            assert lib.bura_solve_systems(plan, torch.from_numpy(f).cuda(), V, tol) == lib.BURA_OK
            torch.cuda.synchronize()
            c, d, _ = lib.bura_get_rational(plan, k)
            lam_lo = lib.bura_get_stats(plan)["lambda_lo"]
            v = V.cpu().numpy()
            bound = sum(c[j] * np.linalg.norm(f - (A @ v[j] - d[j] * v[j])) / (lam_lo - d[j]) for j in range(k + 1))
            assert bound <= 1.001 * tol * np.linalg.norm(f)  # the solver's own stopping rule, its residuals in another order
    finally:
        lib.bura_destroy(plan)
