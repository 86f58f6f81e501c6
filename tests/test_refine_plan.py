"""The step count of the refinement plan (csrc/refine_plan.h, the code that the one-launch solver runs on the device,
compiled here for the host): the closed form for every accepted inner_rtol, in constant time.
"""
import ctypes
import math
import os
import shutil
import subprocess
import time

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_04846_gb300", "csrc")


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("plan")
    src = d / "plan.cpp"
    src.write_text('#include "refine_plan.h"\n'
                   'extern "C" double steps(double t, double r) { return bura::plan_steps(t, r, pow(r, 1e-9), log(r)); }\n')
    so = d / "plan.so"
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + CSRC, str(src), "-o", str(so)], check=True)
    fn = ctypes.CDLL(str(so)).steps
    fn.argtypes = [ctypes.c_double, ctypes.c_double]
    fn.restype = ctypes.c_double
    return fn


def _exact(t, r):
    return min(max(1, math.ceil(math.log(t) / math.log(r) - 1e-9)), 2 ** 31 - 1)


@pytest.mark.parametrize("r", [1e-300, 1e-12, 1e-5, 1e-3, 0.1, 0.5, 0.9, 0.999, 1 - 1e-6])
def test_count_is_the_closed_form(steps, r):
    for i in range(1, 1200):
        t = 10.0 ** (-i / 4.0)  # 0.56 to 1e-299, never within the margin of a power of these inner_rtol by accident
        x = math.log(t) / math.log(r)
        if abs(x - round(x)) < 1e-8 * max(1.0, abs(x)) + 2e-9:
            continue  # at the margin itself either rounding is right
        assert steps(t, r) == _exact(t, r), (t, r)


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 9, 12])
def test_an_exact_power_needs_no_further_step(steps, n):
    assert steps(1e-5 ** n, 1e-5) == n
    assert steps(0.5 ** n, 0.5) == n
    assert steps(0.5 ** n * (1 - 1e-6), 0.5) == n + 1


@pytest.mark.parametrize("r", [1 - 1e-9, 1 - 1e-12, math.nextafter(1.0, 0.0)])
@pytest.mark.parametrize("t", [0.9, 1e-8, 1e-300, 5e-324, 0.0])
def test_constant_time_next_to_one(steps, r, t):
    """inner_rtol next to 1 and a threshold that underflows: the count is large (capped at 2^31 - 1) but not counted out."""
    t0 = time.perf_counter()
    n = steps(t, r)
    assert time.perf_counter() - t0 < 0.01
    assert 8 < n <= 2 ** 31 - 1 and n == math.floor(n)
    if t > 0:
        assert abs(n - _exact(t, r)) <= 1e-6 * n + 1
    assert steps(0.0, 0.75) == 2 ** 31 - 1
