"""Device arrays of the explicit calls that end before the call's last element
are refused on the host, and nothing is written, whichever argument it is.

The short arrays start 64 bytes before the end of their allocation; the test
reads that end, and that the allocation is one the library judges, from the
driver first.
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")

RANGE_START, RANGE_SIZE, PLAIN = 11, 12, 10   # CU_POINTER_ATTRIBUTE_*


def _attribute(which, ptr, kind):
    v = kind(0)
    rc = C.CDLL("libcuda.so.1").cuPointerGetAttribute(C.byref(v), which, C.c_uint64(ptr))
    return v.value if rc == 0 else None


# (call, index of the short argument)
CASES = [("residual", i) for i in range(5)] + [("jvp", i) for i in range(4)] + \
        [("block_jacobi", i) for i in range(3)] + [("rh92_update", i) for i in range(4)]


@pytest.mark.parametrize("call,short", CASES)
def test_array_past_its_allocation_is_refused(call, short):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = W.config1(n_depth=21, n_nu=17)
    ctx = B.Context(0)
    atm = B.Atmosphere(ctx, B.Atom(ctx, wl.atom), wl.columns[0], n_mu=3)
    N, QZ, QM, NP = atm.n_depth * 2, atm.n_nu * atm.n_depth, atm.n_nu * atm.n_mu, atm.n_depth * 4
    n, J = (torch.from_numpy(x.ravel().copy()).cuda() for x in (atm.lte(), atm.planck()))
    raw = torch.zeros(32 << 20, dtype=torch.uint8, device="cuda")
    lo, size = _attribute(RANGE_START, raw.data_ptr(), C.c_uint64), _attribute(RANGE_SIZE, raw.data_ptr(), C.c_size_t)
    if not lo or not size or _attribute(PLAIN, raw.data_ptr(), C.c_int) != 1:
        pytest.skip("not a plain cudaMalloc allocation")
    end = lo + size - 64   # room for eight doubles
    zeros = {k: torch.zeros(k, dtype=torch.float64, device="cuda") for k in (N, QZ, QM, NP)}
    need = {"residual": [n, J, zeros[N], zeros[QZ], zeros[QM]], "jvp": [n, J, n, zeros[N]],
            "block_jacobi": [n, J, zeros[NP]], "rh92_update": [n, J, zeros[N], zeros[QZ]]}[call]
    args = [t.data_ptr() for t in need]
    fn = getattr(ctx.lib, "jfnk_" + call)
    torch.cuda.synchronize()
    B.check(fn(ctx.h, atm.h, B.JFNK_FP64, *args, B.JFNK_MEM_DEVICE, None), call)   # as they should be
    torch.cuda.synchronize()
    for t in zeros.values():
        t.zero_()
    args[short] = end
    torch.cuda.synchronize()
    assert fn(ctx.h, atm.h, B.JFNK_FP64, *args, B.JFNK_MEM_DEVICE, None) == B.JFNK_E_INVALID
    assert b"shorter" in ctx.lib.jfnk_last_error()
    torch.cuda.synchronize()
    assert int(raw.count_nonzero()) == 0
    assert all(int(t.count_nonzero()) == 0 for t in zeros.values())
    # and the context serves the next call
    args[short] = need[short].data_ptr()
    B.check(fn(ctx.h, atm.h, B.JFNK_FP64, *args, B.JFNK_MEM_DEVICE, None), call)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(np.isfinite(need[-1].cpu().numpy()), True)
