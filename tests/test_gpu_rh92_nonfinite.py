"""An RH92 update whose solved populations are not finite at one depth (an
infinite total density there, from finite starting populations) stops the solve
with JFNK_E_NAN and leaves the populations it started from. Both solvers of the
update are reached: a warp per depth (FP64, small launches) and a thread per
depth (mixed, large ones).
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")


@pytest.mark.parametrize("precision,columns,nz", [(B.JFNK_FP64, 1, 33), (B.JFNK_MIXED, 1, 33), (B.JFNK_MIXED, 12, 400)])
def test_non_finite_update_is_not_committed(precision, columns, nz):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = B.Context(0)
    wl = W.config1(n_depth=nz, n_nu=9)
    col = wl.columns[0]
    atom = B.Atom(ctx, wl.atom)
    n0 = B.Atmosphere(ctx, atom, col, n_mu=2).lte()
    col.ntot = col.ntot.copy()
    col.ntot[nz // 2] = np.inf
    atms = [B.Atmosphere(ctx, atom, col, n_mu=2) for _ in range(columns)]
    o = B.default_options(precision=precision, solver=B.JFNK_SOLVER_RH92, maxiter=1)
    o.init = B.JFNK_INIT_USER
    n = [n0.copy() for _ in atms]
    st = (B.jfnk_stats * columns)()
    hs = (C.c_void_p * columns)(*[a.h for a in atms])
    ps = (C.c_void_p * columns)(*[x.ctypes.data for x in n])
    rc = ctx.lib.jfnk_batch_solve(ctx.h, columns, hs, C.byref(o), ps, None, st, B.JFNK_MEM_HOST, None)
    assert rc == B.JFNK_E_NAN
    for x, s in zip(n, st):
        assert s.status == B.JFNK_E_NAN
        np.testing.assert_array_equal(x, n0)
