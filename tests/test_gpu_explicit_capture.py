"""A captured explicit call replays with its own options, whatever calls come
between: preconditioner blocks of the first solution, captured, replayed after the
third solution's were built. The same bits as the call made directly.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2406_17234_gb300.binding")


@pytest.mark.parametrize("precision", [B.JFNK_FP64, B.JFNK_MIXED])
def test_captured_blocks_keep_their_variant(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = W.config2(nu_scale=0.1, n_depth=33)
    ctx = B.Context(0)
    atm = B.Atmosphere(ctx, B.Atom(ctx, wl.atom), wl.columns[0], n_mu=3)
    n = torch.from_numpy(atm.lte()).cuda()
    P = torch.zeros((atm.n_depth, atm.n_levels, atm.n_levels), dtype=torch.float64, device="cuda")

    def call():
        B.check(ctx.lib.jfnk_block_jacobi(ctx.h, atm.h, precision, n.data_ptr(), None, P.data_ptr(), B.JFNK_MEM_DEVICE,
                                          torch.cuda.current_stream().cuda_stream), "jfnk_block_jacobi")

    call()   # buffers
    torch.cuda.synchronize()
    first = P.cpu().numpy()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        call()
    third, _ = B.block_jacobi_variant(atm, atm.lte(), 3, precision=precision)
    assert np.abs(third - first).max() > 0.0
    P.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(P.cpu().numpy(), first)
