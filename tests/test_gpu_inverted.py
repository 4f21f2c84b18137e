"""Columns with inverted populations (negative opacity over a few layers): J of
every FP64 formal-solution kernel against extended-precision sums of the same short
characteristics, and the mixed mode's sweeps against one another.

The scale of an element is the same sum over the absolute values of its terms.
Tolerance: 1e-11 of it (coefficients to 4e-13 at optical depths of 1e-3; tens of
layers count). A series used outside its range is off by 2e-4 at an optical depth of
-1.
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from test_gpu_cached_limits import _mean_intensity

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")
L = np.longdouble


def _inverted(nz, n_mu, moving=False, depth=0.5):
    """(atmosphere, populations, J, scale): a two-level column whose layers 5 to 9
    are inverted, line-centre optical depths of about 1 per layer, -depth in the
    inverted ones."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = B.Context(0)
    atom = W.two_level_atom(n_nu=9)
    one = np.ones(nz)
    z = np.linspace(1e6, 0.0, nz)
    T = 5000.0 + 300.0 * np.sin(0.3 * np.arange(nz))
    col = W.Column(z=z, T=T, ne=1e10 * one, ntot=1e8 * one, rho=1e-3 / (z[0] - z[1]) * one, kappa=1.0,
                   vlos=1e-9 * one if moving else None)
    atm = B.Atmosphere(ctx, B.Atom(ctx, atom), col, n_mu=n_mu)
    nq = atm.n_nu
    chi_c, eta_c = (atm.table(i, nq * nz).reshape(nq, nz).astype(L) for i in (6, 7))
    V, G = (atm.table(i, nq * nz).reshape(nq, nz).astype(L) for i in (3, 4))
    # line-centre optical depth of a layer: V n |dz|
    lo = 1.0 / (float(V.max()) * (z[0] - z[1])) * one
    up = 0.1 * lo
    up[5:10], lo[5:10] = (1.0 + 2.0 * depth) * lo[5:10], 0.5 * lo[5:10]   # g = 1/2
    n = np.stack([lo, up], axis=1)
    nu = np.array(atm.atom.frequencies()).astype(L)
    c2 = 2 * L(6.62607015e-27) * nu ** 3 / L(2.99792458e10) ** 2
    J, scale = np.zeros((2, nq, nz))
    for q in range(nq):
        s = L(1.0) * G[q] * up
        chi = chi_c[q] + V[q] * (lo - s)
        S = (eta_c[q] + c2[q] * V[q] * s) / chi
        assert (chi < 0).any() or q != nq // 2
        Ib = L(atm.planck()[q, -1])
        J[q] = _mean_intensity(chi, S, z, n_mu, Ib)
        scale[q] = _mean_intensity(chi, S, z, n_mu, Ib, absolute=True)
    return atm, n, J, scale


def _device(atm, n):
    import torch
    n_d = torch.from_numpy(n.copy()).cuda()
    F_d = torch.zeros_like(n_d)
    J_d = torch.zeros((atm.n_nu, atm.n_depth), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    B.check(atm.ctx.lib.jfnk_residual_static(atm.ctx.h, atm.h, n_d.data_ptr(), None, F_d.data_ptr(), J_d.data_ptr(),
                                             None), "jfnk_residual_static")
    torch.cuda.synchronize()
    return J_d.cpu().numpy()


# n_mu = 8 at 1,000 depths: too deep for a block's rays, the separate per-ray kernels
@pytest.mark.parametrize("path,nz,n_mu", [("cached", 24, 2), ("moving", 24, 3), ("moving", 1000, 8), ("static", 24, 2),
                                          ("static", 1000, 8)])
def test_inverted_layers(path, nz, n_mu):
    atm, n, ref, scale = _inverted(nz, n_mu, path == "moving")
    J = _device(atm, n) if path == "static" else B.residual(atm, n, want_J=True)[1]
    assert np.all(np.abs(J - ref) <= 1e-11 * scale)


@pytest.mark.parametrize("n_mu", [1, 5])
def test_mixed_sweeps_agree_on_inverted_layers(n_mu):
    """The same bits from the warp, thread and fused sweeps after one Newton step."""
    out = []
    for variant in (B.JFNK_FORMAL_SWEEP_WARP, B.JFNK_FORMAL_SWEEP_THREAD, B.JFNK_FORMAL_SWEEP_THREAD_FUSED):
        atm, n, _, _ = _inverted(24, n_mu, depth=0.1)
        o = B.default_options(precision=B.JFNK_MIXED, formal_variant=variant, maxiter=1, max_ticks=20)
        o.init = B.JFNK_INIT_USER
        J = atm.planck()
        st = B.jfnk_stats()
        atm.ctx.lib.jfnk_solve(atm.ctx.h, atm.h, C.byref(o), n.ctypes.data, J.ctypes.data, C.byref(st),
                               B.JFNK_MEM_HOST, None)
        assert st.formal_kernel == variant and st.jvp_calls > 0
        out.append((n, J, st.F_calls, st.F_norm))
    for other in out[1:]:
        assert out[0][2:] == other[2:]
        np.testing.assert_array_equal(out[0][0], other[0])
        np.testing.assert_array_equal(out[0][1], other[1])
