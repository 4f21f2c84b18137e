"""The cached FP64 evaluation (one kernel per tile of frequencies) at the edges
of its tiling, against the CPU oracle: depths around its chunks of 16 layers
and its 64-depth tiles of level sums, a last tile that is not full, one to
eight angles, more transitions at a frequency than a packed list holds, and
the deepest column.

Tolerance: F and J_F v per element against the gross rates of their depth, 1e-10
as in the parity tests (the tables agree to 1e-9 in the line wings, whose share
of a rate is below 0.1); J 1e-9 relative; blocks against their depth's largest
entry, 1e-9.
"""
import numpy as np
import pytest

import workloads as W
from oracle import model as OM
from oracle.precond import block_jacobi as ora_P
from oracle.residual import jvp_complex, residual as ora_residual
from oracle.rh92 import rh92_update as ora_rh92

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")

CASES = [
    ("two-level", lambda: W.config1(n_depth=2, n_nu=5), 1),
    ("two-level", lambda: W.config1(n_depth=17, n_nu=41), 8),
    ("ca", lambda: W.config2(nu_scale=0.21, n_depth=16), 3),
    ("ca", lambda: W.config2(nu_scale=0.7, n_depth=65), 5),
    ("ca", lambda: W.config2(nu_scale=0.05, n_depth=1024), 5),
    ("h", lambda: W.config3(nu_scale=0.3, n_depth=34), 6),
    ("dense", lambda: W.dense_overlap_workload(n_depth=33), 2),
]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_cached_evaluation_matches_oracle_at_tile_edges(i):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _, make, nmu = CASES[i]
    wl = make()
    ctx = B.Context(0)
    atom = B.Atom(ctx, wl.atom)
    atm = B.Atmosphere(ctx, atom, wl.columns[0], n_mu=nmu)
    m = OM.build_model(wl.atom, wl.columns[0], nmu)
    rng = np.random.default_rng(100 + i)
    n = W.perturbed_populations(m.nstar, rng, 0.02)
    Jd = m.B * np.exp(rng.normal(0.0, 0.05, m.B.shape))
    v = n * rng.normal(0.0, 1.0, n.shape)
    ref = ora_residual(m, n, Jd, want_lambda=True)
    gross, dgross = np.zeros_like(n), np.zeros_like(n)
    for t, tr in enumerate(m.trans):
        up = m.Cmat[:, tr.lo, tr.up] + ref.R_up[t]
        dn = m.Cmat[:, tr.up, tr.lo] + ref.R_dn[t]
        for l in (tr.lo, tr.up):
            gross[:, l] += n[:, tr.lo] * up + n[:, tr.up] * dn
            dgross[:, l] += np.abs(v[:, tr.lo]) * up + np.abs(v[:, tr.up]) * dn
    k = np.arange(m.nz)
    gross[k, ref.istar] = n.sum(axis=1)
    dgross += gross
    F, J, I = B.residual(atm, n, Jd, want_J=True, want_emergent=True)
    assert np.all(np.abs(F - ref.F) <= 1e-10 * gross)
    np.testing.assert_allclose(J, ref.J, rtol=1e-9)
    np.testing.assert_allclose(I, ref.I_emergent, rtol=1e-9)
    Jv = B.jvp(atm, n, v, Jd)
    assert np.all(np.abs(Jv - jvp_complex(m, n, Jd, v, ref.istar)) <= 1e-10 * dgross)
    for variant in (1, 3):
        P, _ = B.block_jacobi_variant(atm, n, variant, Jd)
        rP = ora_P(m, n, ref, variant)
        assert np.all(np.abs(P - rP) <= 1e-9 * np.abs(rP).max(axis=(1, 2), keepdims=True))
    new, _ = B.rh92_update(atm, n, Jd)
    rn = ora_rh92(m, n, ref)
    assert np.all(np.abs(new - rn) <= 1e-7 * np.abs(rn).max(axis=1, keepdims=True))


MOVING = [
    # (depths, line points, angles): chunk edges, ragged tiles; the last is too
    # deep for a block's rays and takes the separate kernels
    (2, 5, 1), (9, 7, 3), (17, 21, 8), (34, 9, 5), (1000, 5, 8),
]


@pytest.mark.parametrize("nz,nq,nmu", MOVING)
def test_moving_evaluation_matches_oracle_at_tile_edges(nz, nq, nmu):
    from dataclasses import replace
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = W.tiny_workload(n_depth=nz, n_nu_line=nq, n_nu_cont=3)
    col = replace(wl.columns[0], vlos=np.linspace(3e5, -1e5, nz))
    ctx = B.Context(0)
    atom = B.Atom(ctx, wl.atom)
    atm = B.Atmosphere(ctx, atom, col, n_mu=nmu)
    m = OM.build_model(wl.atom, col, nmu)
    rng = np.random.default_rng(nz)
    n = W.perturbed_populations(m.nstar, rng, 0.02)
    Jd = m.B * np.exp(rng.normal(0.0, 0.05, m.B.shape))
    v = n * rng.normal(0.0, 1.0, n.shape)
    ref = ora_residual(m, n, Jd, want_lambda=True)
    gross, dgross = np.zeros_like(n), np.zeros_like(n)
    for t, tr in enumerate(m.trans):
        up = m.Cmat[:, tr.lo, tr.up] + ref.R_up[t]
        dn = m.Cmat[:, tr.up, tr.lo] + ref.R_dn[t]
        for l in (tr.lo, tr.up):
            gross[:, l] += n[:, tr.lo] * up + n[:, tr.up] * dn
            dgross[:, l] += np.abs(v[:, tr.lo]) * up + np.abs(v[:, tr.up]) * dn
    gross[np.arange(nz), ref.istar] = n.sum(axis=1)
    dgross += gross
    F, J, I = B.residual(atm, n, Jd, want_J=True, want_emergent=True)
    assert np.all(np.abs(F - ref.F) <= 1e-10 * gross)
    np.testing.assert_allclose(J, ref.J, rtol=1e-9)
    np.testing.assert_allclose(I, ref.I_emergent, rtol=1e-9)
    Jv = B.jvp(atm, n, v, Jd)
    assert np.all(np.abs(Jv - jvp_complex(m, n, Jd, v, ref.istar)) <= 1e-10 * dgross)
    P, rP = B.block_jacobi(atm, n, Jd), ora_P(m, n, ref)
    assert np.all(np.abs(P - rP) <= 1e-9 * np.abs(rP).max(axis=(1, 2), keepdims=True))


@pytest.mark.parametrize("precision", [B.JFNK_FP64, B.JFNK_MIXED])
def test_explicit_calls_take_device_arrays_off_the_double_boundary(precision):
    """Arrays that start between two doubles are copied, not read by a kernel:
    the same results to the bit as from aligned ones."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = W.config1(n_depth=21, n_nu=17)
    ctx = B.Context(0)
    atm = B.Atmosphere(ctx, B.Atom(ctx, wl.atom), wl.columns[0], n_mu=3)
    N, QZ, QM = atm.n_depth * atm.n_levels, atm.n_nu * atm.n_depth, atm.n_nu * atm.n_mu

    def device(x, off):
        raw = torch.empty(8 * x.size + 8, dtype=torch.uint8, device="cuda")
        raw[off:off + 8 * x.size] = torch.from_numpy(x.ravel().view(np.uint8).copy()).cuda()
        return raw

    def host(raw, off, n):
        return raw[off:off + 8 * n].cpu().numpy().view(np.float64)

    n, J = atm.lte(), atm.planck()
    got = []
    for off in (0, 4):
        a = [device(x, off) for x in (n, J, 0.1 * n)]
        out = [device(np.zeros(k), off) for k in (N, QZ, QM, N)]
        p, q = [t.data_ptr() + off for t in a], [t.data_ptr() + off for t in out]
        torch.cuda.synchronize()
        B.check(ctx.lib.jfnk_residual(ctx.h, atm.h, precision, p[0], p[1], q[0], q[1], q[2], B.JFNK_MEM_DEVICE, None),
                "jfnk_residual")
        B.check(ctx.lib.jfnk_jvp(ctx.h, atm.h, precision, p[0], p[1], p[2], q[3], B.JFNK_MEM_DEVICE, None), "jfnk_jvp")
        torch.cuda.synchronize()
        got.append([host(t, off, k) for t, k in zip(out, (N, QZ, QM, N))])
    for x, y in zip(*got):
        assert np.abs(x).max() > 0.0
        np.testing.assert_array_equal(x, y)
