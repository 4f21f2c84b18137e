"""FP64 solves on the paths that keep no coefficients: the server's fused kernel
and, for slots too deep for it, the per-ray kernels; and a batch whose coefficient
planes would exceed their limit. Each is compared with the same columns solved
alone, by the cached evaluation.

Tolerance: the two evaluations round differently (3e-13 of an element after a
solve, measured on the 82-depth Ca II-like column; the stopping rule is the same),
so populations agree to 1e-9 relative and take the same steps. A difference
quotient divides the rounding of F (1e-13 of its gross rates) by its step: products
agree to about 1e-5, populations to 1e-4.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return B.Context(0)


OPTIONS = {
    "rh92 start": dict(rh92_warmup=10, rh92_switch=0.1),
    "newton": dict(),
    "central differences": dict(jvp=B.JFNK_JVP_CENTRAL),
    "local preconditioner": dict(precond=3, rh92_warmup=3, rh92_switch=0.1),
    "rh92 only": dict(solver=B.JFNK_SOLVER_RH92, maxiter=30),
}


def _columns(ctx):
    out = []
    for wl, mu in ((W.config1(n_depth=41, n_nu=31), 3), (W.config2(nu_scale=0.15, n_depth=45), 5),
                   (W.config2(seed=2, nu_scale=0.11, n_depth=57), 4)):
        atom = B.Atom(ctx, wl.atom)
        out.append(B.Atmosphere(ctx, atom, wl.columns[0], n_mu=mu))
    return out


# 1,024-depth slots: no block holds the rays, the per-ray kernels; 60: the fused one.
# 40 slots of 1,024 depths: the RH92 update by a thread per depth, else by a warp
@pytest.mark.parametrize("max_depth,slots,kernel", [(60, 3, B.JFNK_FORMAL_FUSED), (1024, 40, B.JFNK_FORMAL_PER_RAY)])
def test_fp64_server(ctx, max_depth, slots, kernel):
    atms = _columns(ctx)
    jobs = [(a, B.default_options(**kw)) for kw in OPTIONS.values() for a in atms]
    sv = B.Server(ctx, max_slots=slots, max_depth=max_depth, max_freq=max(a.n_nu for a in atms), max_levels=6,
                  max_trans=16, max_mu=5, mem_bytes=2 << 30, opts=B.default_options())
    for i, (a, o) in enumerate(jobs):
        sv.submit(a, i, o)
    res = {}
    for _ in range(3000):
        sv.step()
        res.update({r["id"]: r for r in sv.poll()})
        if len(res) == len(jobs):
            break
    sv.close()
    for i, (a, o) in enumerate(jobs):
        n, _, st = B.solve(a, o, raise_on_fail=False)
        assert st["formal_kernel"] == B.JFNK_FORMAL_CACHED and res[i]["stats"]["formal_kernel"] == kernel
        assert res[i]["status"] == st["status"]
        assert res[i]["stats"]["F_calls"] == st["F_calls"] or o.jvp
        np.testing.assert_allclose(res[i]["n"], n, rtol=1e-4 if o.jvp else 1e-9)


def test_fp64_batch_above_the_plane_limit(ctx):
    """160 columns (one atmosphere, used by all) of 300 depths, about 2,000
    frequencies and 8 angles: 190 MB of planes each. The fused kernel, tuned on
    the batch, one RH92 iteration and the first Newton step. (The Ca II-like atom:
    a change of one rounding in T moves its populations by 4e-12 here, those of the
    H I-like atom by 1e-9.)"""
    wl = W.config2(n_depth=300, nu_scale=2.0)
    atm = B.Atmosphere(ctx, B.Atom(ctx, wl.atom), wl.columns[0], n_mu=8)
    kw = dict(rh92_warmup=1, maxiter=1, krylov_max=8, max_restarts=0)
    n, _, st = B.solve(atm, B.default_options(**kw), raise_on_fail=False)
    assert st["formal_kernel"] == B.JFNK_FORMAL_CACHED
    plan = B.BatchPlan(ctx, [atm] * 160, krylov_max=8)
    ns, sts = plan.run(B.default_options(**kw), raise_on_fail=False)
    plan.close()
    for x, s in zip(ns, sts):
        assert s["formal_kernel"] == B.JFNK_FORMAL_FUSED
        assert (s["status"], s["F_calls"], s["jvp_calls"]) == (st["status"], st["F_calls"], st["jvp_calls"])
        np.testing.assert_array_equal(x, ns[0])
    np.testing.assert_allclose(ns[0], n, rtol=1e-9)
