"""The sparse sweeps at the edges of their range: rows of exactly 1, 7, 8, 9, 16 and 17 entries (a batch of eight and its
remainders), row counts around a CTA's, one to four chunks of systems; against dense inverses of every shifted system.
"""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def lib():
    from paper_1612_04846_gb300 import build_lib, bura
    build_lib.build(verbose=False)
    return bura


def _blocks(n, seed):
    """Diagonal blocks of the sizes above (the last one cut to n rows), each full and diagonally dominant."""
    rng = np.random.default_rng(seed)
    out, left, i = [], n, 0
    while left:
        m = min((1, 7, 8, 9, 16, 17)[i % 6], left)
        B = -rng.uniform(0.1, 1.0, (m, m))
        B = (B + B.T) / 2
        np.fill_diagonal(B, 0.0)
        np.fill_diagonal(B, -B.sum(axis=1) + rng.uniform(0.5, 1.0, m))
        out.append(B)
        left, i = left - m, i + 1
    return sp.block_diag(out).tocsr()


@pytest.mark.parametrize("n,k,prec", [(1, 3, "MIXED"), (63, 3, "FP64"), (64, 4, "MIXED"), (129, 5, "MIXED"), (128, 9, "FP64"),
                                      (1023, 9, "MIXED"), (700, 12, "MIXED")])
def test_rows(lib, n, k, prec):
    A = _blocks(n, n)
    f = np.random.default_rng(1).uniform(-1.0, 1.0, n)
    tol = 1e-9
    lmin = float(np.linalg.eigvalsh(A.toarray())[0])
    o = lib.bura_default_options()
    o.precision = getattr(lib, "BURA_PREC_" + prec)
    plan = lib.bura_setup_csr(A.indptr, A.indices, A.data, 0.5, k, lambda_min=0.999 * lmin, options=o)
    try:
        V = torch.zeros((k + 1, n), dtype=torch.float64, device="cuda")
        assert lib.bura_solve_systems(plan, torch.from_numpy(f).cuda(), V, tol) == lib.BURA_OK
        torch.cuda.synchronize()
        c, d, _ = lib.bura_get_rational(plan, k)
        lam = lib.bura_get_stats(plan)["Lambda"]
        lo = lib.bura_get_stats(plan)["lambda_lo"]
    finally:
        lib.bura_destroy(plan)
    As, V = A.toarray() / lam, V.cpu().numpy()
    err = sum(c[j] * np.linalg.norm(V[j] - np.linalg.solve(As - d[j] * np.eye(n), f)) for j in range(k + 1))
    assert err <= 1.001 * tol * np.linalg.norm(f)  # what the stopping rule promises, by ||(A - d I)^-1|| <= 1 / (lo - d)
    assert lo > 0
