"""The packed tangent sweep with every angle count, alone and below the launch's
largest one, odd and even frequency counts: a batch of columns of one to eight
angles, forced to the thread sweep, gives each column the bits it gets alone from
the warp sweep (the same rounded operations in the same order).
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")


@pytest.mark.parametrize("counts", [(1,), (2, 1), (3, 5), (6,), (7,), (4, 6), (1, 2, 3, 4, 5, 6, 7, 8)])
def test_thread_sweep_of_any_angle_counts(counts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = B.Context(0)
    kw = dict(precision=B.JFNK_MIXED, rh92_warmup=1, maxiter=1, max_ticks=40)
    atms = []
    for i, mu in enumerate(counts):
        wl = W.config2(seed=i, nu_scale=0.07 + 0.011 * i, n_depth=19 + i) if i % 2 else W.config1(n_depth=23 + i, n_nu=41)
        atms.append(B.Atmosphere(ctx, B.Atom(ctx, wl.atom), wl.columns[0], n_mu=mu))
    ns, sts = B.batch_solve(ctx, atms, B.default_options(formal_variant=B.JFNK_FORMAL_SWEEP_THREAD, **kw),
                            raise_on_fail=False)
    for a, n, st in zip(atms, ns, sts):
        alone, _, sa = B.solve(a, B.default_options(formal_variant=B.JFNK_FORMAL_SWEEP_WARP, **kw), raise_on_fail=False)
        assert sa["formal_kernel"] == B.JFNK_FORMAL_SWEEP_WARP and sa["jvp_calls"] > 0
        assert (st["F_calls"], st["jvp_calls"], st["F_norm"]) == (sa["F_calls"], sa["jvp_calls"], sa["F_norm"])
        np.testing.assert_array_equal(n, alone)
