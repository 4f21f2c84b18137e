"""The mixed mode's small-launch sweep (warp per frequency pair, opacity formed
in the block) against the thread sweep with its separate opacity kernels, at the
edges of its chunks of 16 depths, with odd and even depth counts (a middle depth
is reached by both hemispheres at once), ragged frequency counts, one to eight
angles and more overlapping transitions than a packed list holds.

Both evaluate the same explicitly rounded operations in the same order, so the
populations and mean intensities after an RH92 iteration, a base evaluation and
a few products must agree bit for bit.
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")

CASES = [
    ("two-level", lambda: W.config1(n_depth=2, n_nu=5), 1),
    ("two-level", lambda: W.config1(n_depth=3, n_nu=7), 8),
    ("ca", lambda: W.config2(nu_scale=0.11, n_depth=16), 3),
    ("ca", lambda: W.config2(nu_scale=0.13, n_depth=17), 5),
    ("h", lambda: W.config3(nu_scale=0.1, n_depth=65), 4),
    ("ca", lambda: W.config2(nu_scale=0.06, n_depth=700), 5),
    ("dense", lambda: W.dense_overlap_workload(n_depth=34), 2),
    ("h", lambda: W.config3(nu_scale=0.07, n_depth=33), 6),
]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_small_sweep_gives_the_bits_of_the_thread_sweep(i):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    _, make, nmu = CASES[i]
    wl = make()
    ctx = B.Context(0)
    atom = B.Atom(ctx, wl.atom)
    out = []
    for variant in (B.JFNK_FORMAL_SWEEP_WARP, B.JFNK_FORMAL_SWEEP_THREAD):
        atm = B.Atmosphere(ctx, atom, wl.columns[0], n_mu=nmu)
        o = B.default_options(precision=B.JFNK_MIXED, formal_variant=variant, rh92_warmup=1, maxiter=1, max_ticks=40)
        n = np.zeros((atm.n_depth, atm.n_levels))
        J = atm.planck()
        st = B.jfnk_stats()
        ctx.lib.jfnk_solve(ctx.h, atm.h, C.byref(o), n.ctypes.data, J.ctypes.data, C.byref(st), B.JFNK_MEM_HOST, None)
        assert st.formal_kernel == variant and st.F_calls > 3
        out.append((n, J, st.F_calls, st.F_norm))
    assert out[0][2:] == out[1][2:]
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
