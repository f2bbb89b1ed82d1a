"""FP64-accurate products queued one behind the other on one stream and one workspace, each reading what
the one before wrote: their kernels are placed before the previous one ends and wait for it on the
device.  The same calls with a synchronisation after each are the reference, bit for bit."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _chain(n, ops, dtype, wait):
    h = hsmm()
    g = torch.Generator(device="cuda").manual_seed(n)
    A, B = (torch.randn(n, n, device="cuda", dtype=dtype, generator=g).t() / n ** 0.5 for _ in range(2))
    C, D = h.colmajor(n, n, dtype), h.colmajor(n, n, dtype)
    R = h.R_64F if dtype == torch.float64 else h.C_64F
    ws = torch.empty(h.workspace_size(h.hsmm.make_config(R, R, R, h.COMPUTE_64F_OZAKI), "N", "N", n, n, n),
                     dtype=torch.uint8, device="cuda")
    for ta, tb in ops:
        for x, y, z in ((A, B, C), (C, A, D), (D, C, B)):
            h.gemm(x, y, z, ta, tb, compute=h.COMPUTE_64F_OZAKI, workspace=ws)
            if wait:
                torch.cuda.synchronize()
        A.mul_(0.5)
        if wait:
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    return [t.clone() for t in (A, B, C, D)]


# few tiles (anti-diagonals cut, planes zeroed), several, one; rows in blocks of 64 columns and not
@pytest.mark.parametrize("n", [40, 320, 1001])
@pytest.mark.parametrize("dtype", [torch.float64, torch.complex128])
def test_queued_products_wait_for_each_other(n, dtype):
    ops = [("T", "N"), ("N", "N"), ("N", "T")]
    want = _chain(n, ops, dtype, True)
    for _ in range(3):
        for w, o in zip(want, _chain(n, ops, dtype, False)):
            assert torch.equal(w, o)
