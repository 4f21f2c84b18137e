"""The FP64 step coefficients of the cached evaluation (csrc/step_coef.cuh),
compiled for the host, against 60-digit values: optical depths on both sides of
the series' limit, thin layers, the exponential's cut-off, inverted populations.

Tolerances, with u = 2^-53: the series are Horner sums whose last steps dominate
(4 u relative); om is a table entry plus a small term (4 u relative below ln 2, e =
1 - om to 4 u, where both are of the order of 1; a product of two rounded factors
above); w = om r adds three roundings (8 u), a = 1 - w keeps w's absolute error and
bq = (w - e) r divides it by x.
"""
import ctypes
import shutil
import subprocess

import pytest

HARNESS = r"""
#include "step_coef.cuh"
extern "C" void coef(int n, const double* x, double* out) {
  jfnk::ExpEntry tab[jfnk::kExpTab];
  for (int j = 0; j < jfnk::kExpTab; ++j) tab[j] = jfnk::exp_entry(j);
  for (int i = 0; i < n; ++i) {
    double* o = out + 5 * i;
    jfnk::step_coef(x[i], 1.0 / x[i], tab, o[0], o[1], o[2], o[3], o[4]);
  }
}
"""


@pytest.fixture(scope="module")
def coef(tmp_path_factory):
    import os
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    d = tmp_path_factory.mktemp("coef")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I", os.path.join(root, "paper_2406_17234_gb300", "csrc"), "-o", str(d / "h.so"),
                    str(d / "h.cpp")], check=True)
    f = ctypes.CDLL(str(d / "h.so")).coef

    def call(xs):
        a, o = (ctypes.c_double * len(xs))(*xs), (ctypes.c_double * (5 * len(xs)))()
        f(len(xs), a, o)
        return [o[5 * i:5 * i + 5] for i in range(len(xs))]
    return call


def _span(lo, hi, n):
    return [lo * (hi / lo) ** (i / (n - 1)) for i in range(n)]


@pytest.mark.parametrize("xs", [
    _span(1e-12, 9.99e-6, 201), _span(1e-5, 9.99e-4, 2001), _span(1e-3, 0.6931, 4001), _span(0.6932, 699.9, 2001),
    [-x for x in _span(1e-12, 9.99e-4, 401)], [-x for x in _span(1e-3, 30.0, 401)],
], ids=["tiny", "below the series' limit", "thin", "thick", "inverted, thin", "inverted"])
def test_step_coefficients_against_multiprecision(coef, xs):
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 60
    u = 2.0 ** -53
    for x, (e, w, a, bq, om) in zip(xs, coef(xs)):
        X = mp.mpf(x)
        E = mp.exp(-X)
        OM = -mp.expm1(-X)
        W = OM / X
        A, BQ = 1 - W, (W - E) / X
        assert abs(e - E) <= 4 * u * max(E, 1) if x < 0.6931 else abs(e - E) <= 8 * u * E
        assert abs(om - OM) <= (4 * u * abs(OM) if x < 0.6931 else 2 * u)
        assert abs(w - W) <= 8 * u * abs(W)
        if abs(x) < 1e-3:
            assert abs(a - A) <= 4 * u * abs(A) and abs(bq - BQ) <= 4 * u * abs(BQ)
        else:
            assert abs(a - A) <= 8 * u * max(1, abs(W)) and abs(bq - BQ) <= 8 * u * (abs(W) + E) / abs(x)


def test_step_coefficients_past_the_cutoff(coef):
    xs = [700.5, 1e4, 1e100]
    for x, (e, w, a, bq, om) in zip(xs, coef(xs)):
        assert e == 0.0 and om == 1.0 and a == 1.0 - w
        assert abs(w * x - 1.0) < 1e-15 and abs(bq * x * x - 1.0) < 1e-15
