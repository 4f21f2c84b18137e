"""The cached FP64 evaluation where its arithmetic is near a limit: source
functions below the FP32 range.

References are plain 80- or 128-bit sums of the same short characteristics
(App. A.1) over the column's own tables, so that only the evaluation's own
rounding counts.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")
L = np.longdouble


def _context():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return B.Context(0)


def _mean_intensity(chi, S, z, n_mu, I_bottom, absolute=False):
    """J of one frequency in extended precision (absolute: over the sizes of its terms)."""
    x, w = np.polynomial.legendre.leggauss(n_mu)
    mu, wmu = (L(1) + x) / 2, w / L(2)
    dz = np.abs(np.diff(z.astype(L)))
    J = np.zeros(len(z), dtype=L)
    for m, h in zip(mu, wmu):
        t = dz * (chi[1:] + chi[:-1]) / (2 * m)
        e, om = np.exp(-t), -np.expm1(-t)
        series = sum((-t) ** k * (k + 1) / L(np.prod(np.arange(1, k + 3, dtype=float))) for k in range(18))
        bq = np.where(np.abs(t) < 0.5, series, (om / t - e) / t)
        a, b = om - bq * t, bq * t
        if absolute:
            a, b, S = np.abs(a), np.abs(b), np.abs(S)
        for order in (range(1, len(z)), range(len(z) - 2, -1, -1)):
            up = order[0] != 1
            I = I_bottom if up else L(0)
            J[-1 if up else 0] += h / 2 * I
            for k in order:
                u, l = (k + 1, k) if up else (k - 1, k - 1)
                I = I * e[l] + a[l] * S[k] + b[l] * S[u]
                J[k] += h / 2 * I
    return J


@pytest.mark.parametrize("n_mu", [1, 5])
def test_thin_layers_far_below_the_fp32_range(n_mu):
    """A cold layer of optical depth 1e-8: J, 1e-8 of S, is the sum of the
    intensities, not S plus the sum of I - S, also where both are below the FP32
    range. Every term is positive: about 5 roundings per layer and angle, 1e-13
    with a margin of ten."""
    ctx = _context()
    nz = 20
    atom = W.two_level_atom(n_nu=5)
    T = np.full(nz, 300.0)   # h nu/k T = 96: S = 2e-42
    T[-1] = 100.0            # nothing comes in from below
    z = np.linspace(1e8, 0.0, nz)
    one = np.ones(nz)
    col = W.Column(z=z, T=T, ne=1e10 * one, ntot=1e8 * one, rho=1e-8 / z[0] * (1.0 + 0.5 * np.sin(np.arange(nz))),
                   kappa=1.0)
    atm = B.Atmosphere(ctx, B.Atom(ctx, atom), col, n_mu=n_mu)
    N = atm.n_nu * nz
    chi, eta = (atm.table(i, N).reshape(atm.n_nu, nz).astype(L) for i in (6, 7))
    _, J, _ = B.residual(atm, np.zeros((nz, 2)), want_J=True)
    for q in range(atm.n_nu):
        S = eta[q] / chi[q]
        ref = _mean_intensity(chi[q], S, z, n_mu, L(atm.planck()[q, -1]))
        np.testing.assert_array_less(ref[:-1], 1e-7 * S[:-1])
        np.testing.assert_allclose(J[q], ref.astype(np.float64), rtol=1e-13)
