"""The three-word FP32 sums of the inner solves' dot products (csrc/sum3.h, the code that the kernels run, compiled here for
the host) against exact rational arithmetic: no larger an error than FP64 sums in the same order, in the kernels' orders.
"""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1612_04846_gb300", "csrc")

SOURCE = r"""
#include "sum3.h"
using namespace bura;
static void out(const Sum3& t, float* w) { w[0] = t.s; w[1] = t.c; w[2] = t.e; }
extern "C" {
// `chains` threads add x[t], x[t + chains], ... in order; their sums are added in a chain, or in a tree of halves
void total(const float* x, long long n, int chains, int tree, float* w) {
    Sum3* t = new Sum3[chains]();
    for (long long i = 0; i < n; ++i) t[i % chains].add(x[i]);
    if (tree) {
        for (int h = chains / 2; h; h /= 2)
            for (int i = 0; i < h; ++i) t[i].add(t[i + h]);
    } else {
        for (int i = 1; i < chains; ++i) t[0].add(t[i]);
    }
    out(t[0], w);
    delete[] t;
}
// the same in FP64
double total64(const float* x, long long n, int chains) {
    double* t = new double[chains]();
    for (long long i = 0; i < n; ++i) t[i % chains] += (double)x[i];
    for (int i = 1; i < chains; ++i) t[0] += t[i];
    const double r = t[0];
    delete[] t;
    return r;
}
// what keeping two words only would give
void total2(const float* x, long long n, int chains, float* w) {
    Sum3 r{};
    float* s = new float[chains]();
    float* c = new float[chains]();
    for (long long i = 0; i < n; ++i) c[i % chains] += two_sum_err(s[i % chains], x[i], s[i % chains]);
    for (int i = 0; i < chains; ++i) { r.c += two_sum_err(r.s, s[i], r.s); r.c += c[i]; }
    out(r, w);
    delete[] s;
    delete[] c;
}
float quotient(const float* a, const float* b) { return sum3_div(Sum3{a[0], a[1], a[2]}, Sum3{b[0], b[1], b[2]}); }
int le(const float* a, const float* b) { return sum3_le(Sum3{a[0], a[1], a[2]}, Sum3{b[0], b[1], b[2]}); }
void of(double x, float* w) { out(sum3_of(x), w); }
void merge(const float* a, const float* b, float* w) { Sum3 t{a[0], a[1], a[2]}; t.add(Sum3{b[0], b[1], b[2]}); out(t, w); }
// the sum of a warp's 32 values by limbs
void warp(const float* a, float* w) {
    unsigned top = 0u;
    for (int i = 0; i < 32; ++i) { const unsigned m = limb_top(Sum3{a[3 * i], a[3 * i + 1], a[3 * i + 2]}); top = m > top ? m : top; }
    Limbs t{};
    for (int i = 0; i < 32; ++i) {
        const Limbs l = to_limbs(Sum3{a[3 * i], a[3 * i + 1], a[3 * i + 2]}, top);
        t.top = l.top;
        for (int j = 0; j < 3; ++j) t.w[j] += l.w[j];
    }
    out(from_limbs(t), w);
}
void normal(const float* a, float* w) { out(Sum3{a[0], a[1], a[2]}.normal(), w); }
}
"""


@pytest.fixture(scope="module")
def c(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("sum3")
    (d / "s.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I" + CSRC, str(d / "s.cpp"), "-o",
                    str(d / "s.so")], check=True)
    lib = ctypes.CDLL(str(d / "s.so"))
    F, L, I = ctypes.POINTER(ctypes.c_float), ctypes.c_longlong, ctypes.c_int
    lib.total.argtypes = [F, L, I, I, F]
    lib.total64.argtypes, lib.total64.restype = [F, L, I], ctypes.c_double
    lib.total2.argtypes = [F, L, I, F]
    lib.quotient.argtypes, lib.quotient.restype = [F, F], ctypes.c_float
    lib.le.argtypes, lib.le.restype = [F, F], ctypes.c_int
    lib.of.argtypes = [ctypes.c_double, F]
    lib.normal.argtypes = [F, F]
    lib.merge.argtypes = [F, F, F]
    lib.warp.argtypes = [F, F]
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_float))


def _value(w):
    return sum(Fraction(float(v)) for v in w)


def _total(c, x, chains, tree):
    w = np.zeros(3, np.float32)
    c.total(_p(x), x.size, chains, tree, _p(w))
    return w


def _vectors():
    rng = np.random.default_rng(5)
    n = 60000
    pos = (rng.standard_normal(n) ** 2).astype(np.float32)          # r . r
    yield "squares", pos
    mix = rng.standard_normal(n).astype(np.float32)
    yield "signs", mix                                               # cancellation to about sqrt(n)
    wide = (mix * np.exp2(rng.uniform(-60, 20, n))).astype(np.float32)
    yield "range", wide
    y = np.concatenate([wide[:n // 2], -wide[:n // 2]])
    y[-1] += np.float32(1e-7)
    yield "cancel", rng.permutation(y).astype(np.float32)            # the large part cancels
    yield "tiny", (pos * np.float32(1e-25)).astype(np.float32)


# chains: one thread's folds; a block's; the finishing step's 64 groups of 19 block sums; a cluster's lanes
@pytest.mark.parametrize("chains,tree", [(1, 0), (64, 0), (512, 1), (1216, 0), (4096, 1)])
@pytest.mark.parametrize("name,x", list(_vectors()), ids=lambda v: v if isinstance(v, str) else "")
def test_error_is_below_that_of_fp64(c, name, x, chains, tree):
    exact = sum(Fraction(float(v)) for v in x)
    mag = sum(abs(Fraction(float(v))) for v in x)
    n = -(-x.size // chains) + (chains.bit_length() if tree else chains)  # additions on the longest chain
    err = abs(_value(_total(c, x, chains, tree)) - exact)
    assert err <= mag * n ** 3 / Fraction(2) ** 72
    err64 = abs(Fraction(c.total64(_p(x), x.size, chains)) - exact)
    assert err <= max(err64, mag / Fraction(2) ** 60)


def test_two_words_are_not_enough(c):
    """The check notices the precision it is about: with the second word's rounding dropped the error is above FP64's."""
    x = dict(_vectors())["squares"]
    exact = sum(Fraction(float(v)) for v in x)
    w = np.zeros(3, np.float32)
    c.total2(_p(x), x.size, 1, _p(w))
    assert abs(_value(w) - exact) > max(abs(Fraction(c.total64(_p(x), x.size, 1)) - exact),
                                        sum(Fraction(float(v)) for v in x) / Fraction(2) ** 60)


def test_order_of_the_operands_does_not_matter(c):
    """a + b and b + a have the same bits (every lane of a butterfly of shuffles holds the same total)."""
    rng = np.random.default_rng(6)
    v, w, z = (np.zeros(3, np.float32) for _ in range(3))
    for _ in range(2000):
        a, b = (np.array([rng.standard_normal(), rng.standard_normal() * 2.0 ** -22, rng.standard_normal() * 2.0 ** -44]) for _ in range(2))
        a, b = a.astype(np.float32), (b * 2.0 ** rng.integers(-30, 30)).astype(np.float32)
        c.merge(_p(a), _p(b), _p(v))
        c.merge(_p(b), _p(a), _p(w))
        assert np.array_equal(v.view(np.uint32), w.view(np.uint32))
        exact = _value(a) + _value(b)
        # only the three additions of last words round, by 2^-24 of what they add: those words and the two errors of c's
        sw, cw, ew = (abs(Fraction(float(a[j]))) + abs(Fraction(float(b[j]))) for j in range(3))
        u = Fraction(1, 2 ** 24)
        assert abs(_value(v) - exact) <= 4 * u * (ew + 3 * u * cw + 2 * u * u * sw)
        c.normal(_p(v), _p(z))
        assert _value(z) == _value(v) and abs(z[1]) <= 0.51 * np.spacing(abs(z[0]))


def _round32(q):
    """The FP32 value nearest to the rational q (ties to even)."""
    f = np.float32(float(q))
    best = min((f, np.nextafter(f, np.float32(np.inf)), np.nextafter(f, np.float32(-np.inf))),
               key=lambda v: (abs(Fraction(float(v)) - q), int(v.view(np.uint32)) & 1))
    return best


def test_quotients_are_rounded_once(c):
    """Random sums, and quotients placed within 2^-50 of the middle between two FP32 values on either side."""
    rng = np.random.default_rng(7)
    for i in range(4000):
        b = np.array([rng.uniform(0.5, 2), rng.uniform(-1, 1) * 2.0 ** -25, rng.uniform(-1, 1) * 2.0 ** -50], np.float32)
        b *= np.float32(2.0 ** rng.integers(-40, 20))
        if i % 2:
            a = np.array([rng.uniform(0.5, 2), rng.uniform(-1, 1) * 2.0 ** -20, rng.uniform(-1, 1) * 2.0 ** -45], np.float32)
            a *= np.float32(2.0 ** rng.integers(-40, 20))
        else:
            q = Fraction(int(rng.integers(2 ** 23, 2 ** 24)) * 2 + 1, 2 ** 24)  # a middle
            t = (q * (1 + Fraction(int(rng.integers(-3, 4)), 2 ** 51))) * _value(b)
            a = np.zeros(3, np.float32)
            for j in range(3):
                a[j] = np.float32(float(t))
                t -= Fraction(float(a[j]))
        got = np.float32(c.quotient(_p(a), _p(b)))
        q = _value(a) / _value(b)
        off = q * Fraction(2) ** -66  # (a middle itself, which 70 bits do not decide, may go either way)
        assert got in (_round32(q - off), _round32(q + off)), (i, a, b)


def test_threshold_words(c):
    """An FP64 threshold is held exactly, and the comparison with it is exact to the last bit."""
    rng = np.random.default_rng(8)
    w, v = np.zeros(3, np.float32), np.zeros(3, np.float32)
    for _ in range(500):
        t = float(2.0 ** rng.uniform(-60, 10))
        c.of(t, _p(w))
        assert _value(w) == Fraction(t)
        for d, want in ((0.0, 1), (np.nextafter(t, 1e9) - t, 0), (np.nextafter(t, 0) - t, 1)):
            c.of(t + d, _p(v))
            assert c.le(_p(v), _p(w)) == want
    c.of(1e-60, _p(w))
    assert _value(w) <= Fraction(1e-60)  # below the FP32 range: never rounded up
    nan = np.array([np.nan, 0, 0], np.float32)
    assert c.le(_p(nan), _p(w)) == 0


def test_warp_sums_by_limbs(c):
    """32 lanes' sums as integers: within the stated 2^-65 of the largest value (32 lanes round by half a unit of the last
    limb, 2^-43 2^-21 of a scale of at most the largest value, and the result's last word by 2^-24 of its)."""
    rng = np.random.default_rng(9)
    w = np.zeros(3, np.float32)
    for i in range(3000):
        a = rng.standard_normal((32, 3))
        a[:, 1] *= 2.0 ** -20
        a[:, 2] *= 2.0 ** -42
        if i % 3 == 0:
            a[:, 0] = np.abs(a[:, 0]) * np.exp2(rng.uniform(-40, 0, 32))
        elif i % 3 == 1:
            a[:, 0] = 0.0 if i % 2 else np.repeat(a[:16, 0], 2) * np.tile([1, -1], 16)  # words of one size; cancellation
        a = (a * 2.0 ** rng.integers(-50, 60)).astype(np.float32)
        c.warp(_p(a), _p(w))
        exact = sum(Fraction(float(v)) for v in a.ravel())
        top = Fraction(float(np.abs(a).max()))
        assert abs(_value(w) - exact) <= top * 32 / Fraction(2) ** 64 + abs(exact) / Fraction(2) ** 69
    for bad in (np.inf, np.nan):
        a = rng.standard_normal((32, 3)).astype(np.float32)
        a[7, 0] = bad
        c.warp(_p(a), _p(w))
        assert np.isnan(w[0])
    z = np.zeros((32, 3), np.float32)
    c.warp(_p(z), _p(w))
    assert _value(w) == 0
