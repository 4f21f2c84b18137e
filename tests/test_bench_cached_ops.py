"""The bench's FP64 roofline counts the operations of the kernel that ran: the
cached evaluations have no exponential in a product, so their peak is above the
fused kernel's, and a fraction against the latter would exceed one."""
import importlib.util
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cached_kernels_have_their_own_counts():
    spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    assert b.kernel_ops(1, 2) is b.ALG_OPS and b.kernel_ops(4, 0) is b.ALG_OPS
    assert b.kernel_ops(6, 7) is b.CACHED_OPS and b.kernel_ops(4, 7) is b.CACHED_MOVING_OPS
    peaks = {"fp64_fma_per_s": 5.3e11, "fp64_exp_per_s": 3.3e10}
    for ops, fmas in ((b.CACHED_OPS, 3), (b.CACHED_MOVING_OPS, 5)):
        assert abs(b.peak_rate("jvp", True, peaks, ops) / (5.3e11 / fmas) - 1) < 1e-12
        assert b.peak_rate("jvp", True, peaks, ops) > b.peak_rate("jvp", True, peaks)
        assert b.peak_rate("value", True, peaks, ops) >= b.peak_rate("value", True, peaks)
