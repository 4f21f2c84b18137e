"""The oracle's piecewise-linear coefficients at negative optical depths
(inverted populations), against 40-digit values: 4e-16/x^2 from the direct forms'
cancellation, as at positive ones."""
import numpy as np
import pytest

from oracle import formal as OF


def test_coefficients_of_inverted_steps():
    mp = pytest.importorskip("mpmath").mp
    from mpmath import exp, mpf
    mp.dps = 40
    for xv in (-1e-9, -1e-3, -0.099, -0.101, -1.0, -5.0, -20.0):
        X = mpf(xv)
        w = (1 - exp(-X)) / X
        e, a, b, bq = OF.pl_coefficients(np.array([xv]))
        for got, ref in ((e, exp(-X)), (a, 1 - w), (b, w - exp(-X)), (bq, (w - exp(-X)) / X)):
            assert got[0] == pytest.approx(float(ref), rel=1e-13)
