"""The generated M2M / L2L blocks (csrc/translate_gen.cuh), compiled on the host in float64, against the definitions:
M2M must give the parent's moments of a child's particles, L2L must re-expand a local polynomial about the
child's centre (s/4 away along each axis), for all eight child offsets and p = 1..6; the harmonic completion must
return a harmonic expansion unchanged.  The generator must reproduce the committed header."""
import ctypes
import itertools
import os
import shutil
import subprocess
import sys
from math import factorial

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1712_10116_gb300", "csrc")

HARNESS = r"""
#define __device__
#define __forceinline__ inline
#include "translate_gen.cuh"
template <int P> static void coef(double s, double (&c)[P + 1]) { c[0] = 1; for (int d = 1; d <= P; ++d) c[d] = c[d - 1] * 0.25 * s / d; }
template <int P> static void run(int what, const double *s, const double *in, double *out)
{
    constexpr int NC = XlGen<P>::NC;
    double v[NC], x[P + 1], y[P + 1], z[P + 1], h[XlGen<P>::NH];
    coef<P>(s[0], x); coef<P>(s[1], y); coef<P>(s[2], z);
    for (int k = 0; k < NC; ++k) v[k] = in[k];
    if (what == 0) { XlGen<P>::moments_in(v); XlGen<P>::shift_moments(v, x, y, z); XlGen<P>::moments_out(v); }
    if (what == 1) { XlGen<P>::shift_locals(v, x, y, z); XlGen<P>::locals_out(v); }
    if (what == 2) { for (double &q : h) q = 0; XlGen<P>::locals_harmonic(v, h); }
    if (what == 3) XlGen<P>::moments_scale(v);
    for (int k = 0; k < NC; ++k) out[k] = v[k];
}
extern "C" void xl(int p, int what, const double *s, const double *in, double *out)
{
    switch (p) {
    case 1: run<1>(what, s, in, out); break;
    case 2: run<2>(what, s, in, out); break;
    case 3: run<3>(what, s, in, out); break;
    case 4: run<4>(what, s, in, out); break;
    case 5: run<5>(what, s, in, out); break;
    case 6: run<6>(what, s, in, out); break;
    }
}
"""


def _mi(p):
    return [(a, b, o - a - b) for o in range(p + 1) for a in range(o, -1, -1) for b in range(o - a, -1, -1)]


@pytest.fixture(scope="module")
def xl(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("xl")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "h.cpp"), "-o", str(d / "h.so")],
                   check=True)
    f = ctypes.CDLL(str(d / "h.so")).xl
    p = ctypes.POINTER(ctypes.c_double)
    f.argtypes = [ctypes.c_int, ctypes.c_int, p, p, p]

    def call(order, what, s, v):
        s, v, out = np.array(s, float), np.ascontiguousarray(v, float), np.zeros(len(v))
        f(order, what, *(a.ctypes.data_as(p) for a in (s, v, out)))
        return out
    return call


@pytest.mark.parametrize("p", range(1, 7))
def test_shifts_are_exact_translations(xl, p):
    g = np.random.default_rng(p)
    mi = _mi(p)
    x, m = g.uniform(-0.5, 0.5, (3, 20)), g.uniform(0.5, 1.5, 20)   # in units of the child's side
    for s in itertools.product((-1.0, 1.0), repeat=3):
        z = 0.25 * np.array(s)[:, None]
        child = np.array([(m * x[0] ** a * x[1] ** b * x[2] ** c).sum() for a, b, c in mi])
        X = 0.5 * x + z                                             # in units of the parent's side
        want = np.array([(m * X[0] ** a * X[1] ** b * X[2] ** c).sum() for a, b, c in mi])
        assert np.abs(xl(p, 0, s, child) - want).max() < 1e-14 * 20
        # phi(X) = sum_n L^n X^n / n! (parent's units); about the child: coefficients times 2^-(|n| + 1)
        L = g.uniform(-1, 1, len(mi))
        got = xl(p, 1, s, L)
        y = g.uniform(-0.5, 0.5, 3)
        ev = lambda c, r: sum(q * r[0] ** a * r[1] ** b * r[2] ** d / (factorial(a) * factorial(b) * factorial(d))  # noqa: E731
                              for q, (a, b, d) in zip(c, mi))
        assert abs(2.0 * ev(got, y) - ev(L, 0.5 * y + z[:, 0])) < 1e-13


@pytest.mark.parametrize("p", range(1, 7))
def test_completion_and_scaling(xl, p):
    g = np.random.default_rng(p)
    mi = _mi(p)
    idx = {v: k for k, v in enumerate(mi)}
    v = g.uniform(-1, 1, len(mi))
    for k, (a, b, c) in enumerate(mi):
        if c >= 2:
            v[k] = -v[idx[(a + 2, b, c - 2)]] - v[idx[(a, b + 2, c - 2)]]
    assert np.array_equal(xl(p, 2, (1, 1, 1), v), v)
    want = np.array([q if k < 4 else q * (1.0 / (factorial(a) * factorial(b) * factorial(c)))
                     for k, (q, (a, b, c)) in enumerate(zip(v, mi))])
    assert np.abs(xl(p, 3, (1, 1, 1), v) - want).max() < 1e-15


def test_generator_reproduces_committed_header():
    out = subprocess.run([sys.executable, os.path.join(CSRC, "gen_translate.py")], capture_output=True, check=True).stdout
    assert out == open(os.path.join(CSRC, "translate_gen.cuh"), "rb").read()
