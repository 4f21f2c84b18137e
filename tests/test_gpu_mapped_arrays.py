"""Explicit calls on device memory that the caller mapped itself (the driver's
virtual memory management): inputs mapped for reading only, and inputs and
results mapped for both, give the bits of ordinary arrays.
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")

READ, READWRITE = 1, 3


class Location(C.Structure):
    _fields_ = [("type", C.c_int), ("id", C.c_int)]


class AllocationProp(C.Structure):
    _fields_ = [("type", C.c_int), ("handles", C.c_int), ("location", Location), ("win32", C.c_void_p),
                ("flags", C.c_ubyte * 8)]


class AccessDesc(C.Structure):
    _fields_ = [("location", Location), ("flags", C.c_int)]


class Mapped:
    """``bytes`` of device memory behind an address range of its own."""

    def __init__(self, nbytes):
        self.cu = C.CDLL("libcuda.so.1")
        prop = AllocationProp(type=1, location=Location(1, 0))
        gran, self.ptr, self.handle = C.c_size_t(), C.c_uint64(), C.c_uint64()
        self._do("cuMemGetAllocationGranularity", C.byref(gran), C.byref(prop), 0)
        self.size = (nbytes + gran.value - 1) // gran.value * gran.value
        self._do("cuMemCreate", C.byref(self.handle), C.c_size_t(self.size), C.byref(prop), C.c_ulonglong(0))
        self._do("cuMemAddressReserve", C.byref(self.ptr), C.c_size_t(self.size), C.c_size_t(0), C.c_uint64(0),
                 C.c_ulonglong(0))
        self._do("cuMemMap", self.ptr, C.c_size_t(self.size), C.c_size_t(0), self.handle, C.c_ulonglong(0))
        self.access(READWRITE)

    def _do(self, name, *args):
        rc = getattr(self.cu, name)(*args)
        if rc != 0:
            pytest.skip(f"{name}: {rc}")

    def access(self, flags):
        d = AccessDesc(Location(1, 0), flags)
        self._do("cuMemSetAccess", self.ptr, C.c_size_t(self.size), C.byref(d), C.c_size_t(1))

    def put(self, x):
        self._do("cuMemcpyHtoD_v2", self.ptr, C.c_void_p(x.ctypes.data), C.c_size_t(x.nbytes))

    def get(self, n):
        out = np.zeros(n)
        self._do("cuMemcpyDtoH_v2", C.c_void_p(out.ctypes.data), self.ptr, C.c_size_t(out.nbytes))
        return out

    def free(self):
        self.cu.cuMemUnmap(self.ptr, C.c_size_t(self.size))
        self.cu.cuMemRelease(self.handle)
        self.cu.cuMemAddressFree(self.ptr, C.c_size_t(self.size))


@pytest.mark.parametrize("precision", [B.JFNK_FP64, B.JFNK_MIXED])
def test_arrays_the_caller_mapped(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.zeros(1, device="cuda")
    wl = W.config1(n_depth=21, n_nu=17)
    ctx = B.Context(0)
    atm = B.Atmosphere(ctx, B.Atom(ctx, wl.atom), wl.columns[0], n_mu=3)
    n, J = atm.lte(), atm.planck()
    F0, J0, _ = B.residual(atm, n, J, precision=precision, want_J=True)
    for inputs in (READWRITE, READ):
        mem = [Mapped(x.nbytes) for x in (n, J, n, J)]
        mem[0].put(n)
        mem[1].put(J)
        for m in mem[:2]:
            m.access(inputs)
        B.check(ctx.lib.jfnk_residual(ctx.h, atm.h, precision, *[m.ptr.value for m in mem], None, B.JFNK_MEM_DEVICE,
                                      None), "jfnk_residual")
        torch.cuda.synchronize()
        np.testing.assert_array_equal(mem[2].get(n.size).reshape(n.shape), F0)
        np.testing.assert_array_equal(mem[3].get(J.size).reshape(J.shape), J0)
        for m in mem:
            m.free()
