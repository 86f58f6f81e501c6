"""Profiling a small 2-D plan profiles the solve that the plan runs: one launch and its output stage, with the same result."""
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


@pytest.mark.parametrize("shape,k,var", [((63, 63), 5, False), ((255, 127), 8, False), ((63, 47), 5, True)])
def test_profile_of_a_one_launch_solve(lib, shape, k, var):
    nps = tuple(reversed(shape))
    f = torch.from_numpy(W.rhs_uniform(nps, 96)).cuda()
    faces = W.block_lognormal_faces(nps, 4, 1e-2, 1.0, 6) if var else None
    plan = lib.bura_setup(shape, 0.5, k, faces=faces)
    try:
        u, v = torch.zeros_like(f), torch.zeros_like(f)
        assert lib.bura_solve(plan, f, u, 1e-6) == lib.BURA_OK
        torch.cuda.synchronize()
        s1 = lib.bura_get_stats(plan)
        lib.bura_set_profiling(plan, True)
        assert lib.bura_solve(plan, f, v, 1e-6) == lib.BURA_OK
        assert lib.bura_solve_async(plan, f, v, 1e-6) == lib.BURA_OK
        V = torch.zeros((k + 1, f.numel()), dtype=torch.float64, device="cuda")
        assert lib.bura_solve_systems(plan, f, V, 1e-6) == lib.BURA_OK
        torch.cuda.synchronize()
        s2 = lib.bura_get_stats(plan)
        prof = {e["name"]: e for e in lib.bura_get_profile(plan)}
        lib.bura_set_profiling(plan, False)
        assert set(prof) == {"resident_solve_f32", "resident_output"}
        assert all(e["launches"] == 3 and e["ms"] > 0 and e["bytes"] > 0 for e in prof.values())
        assert s1["launches"] == s2["launches"] == 2 and s1["iters"] == s2["iters"] and s1["outer"] == s2["outer"]
        assert np.array_equal(u.cpu().numpy(), v.cpu().numpy())
        w = torch.zeros_like(f)
        assert lib.bura_solve(plan, f, w, 1e-6) == lib.BURA_OK
        torch.cuda.synchronize()
        assert np.array_equal(u.cpu().numpy(), w.cpu().numpy())
    finally:
        lib.bura_destroy(plan)
