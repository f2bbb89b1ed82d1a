"""gemm_host, FP64-accurate form, at sizes whose panels are chosen by the estimated time (one to four
row and column panels, ragged last panels): the same bits as gemm on device copies."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _host(rows, cols, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(cols, rows, dtype=dtype, generator=g).pin_memory().t()


@pytest.mark.parametrize("m,n,k,ta,tb,beta,dtype", [
    (1500, 1500, 1500, "N", "N", 0.0, torch.float64), (2300, 2050, 2048, "N", "T", 0.5, torch.float64),
    (3000, 600, 3000, "T", "N", 0.0, torch.float64), (700, 3100, 2900, "N", "N", -1.0, torch.float64),
    (4500, 4100, 1000, "T", "T", 0.0, torch.float64), (1300, 1100, 1000, "N", "C", 0.5, torch.complex128)])
def test_same_bits_as_device(m, n, k, ta, tb, beta, dtype):
    h = hsmm()
    A = _host(*((m, k) if ta == "N" else (k, m)), dtype, 1)
    B = _host(*((k, n) if tb == "N" else (n, k)), dtype, 2)
    C = _host(m, n, dtype, 3)
    dA, dB, dC = (X.t().cuda().t() for X in (A, B, C))
    h.gemm_host(A, B, C, ta, tb, beta=beta, compute=h.COMPUTE_64F_OZAKI)
    h.gemm(dA, dB, dC, ta, tb, beta=beta, compute=h.COMPUTE_64F_OZAKI)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.equal(C, dC.cpu())
