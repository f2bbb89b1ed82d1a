"""FP64-accurate products whose slices are kept in blocks of 64 columns (k rounded up to 8 is not a
multiple of 64): the same bits as with zeros appended to the contraction up to whole blocks, which
keeps the slices row by row.  Both orders of each operand, one and several tiles and panels."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _operand(rows, k, kp, op_first, dtype, seed):
    """op(X) as rows x k and the same with zeros to kp columns, stored transposed if op_first."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(rows, k, dtype=dtype, device="cuda", generator=g)
    y = torch.zeros(rows, kp, dtype=dtype, device="cuda")
    y[:, :k] = x
    # column-major storage of op(X) (rows x k) or of its transpose
    return [t.t().contiguous().t() if not op_first else t.contiguous().t() for t in (x, y)]


@pytest.mark.parametrize("kernel", ["pair", "single"])
@pytest.mark.parametrize("ta,tb", [("N", "N"), ("T", "N"), ("N", "T"), ("T", "T")])
@pytest.mark.parametrize("m,n", [(100, 60), (300, 517)])
def test_same_bits_as_whole_blocks(m, n, ta, tb, kernel, monkeypatch):
    monkeypatch.setenv("HSMM_OZAKI_KERNEL", kernel)
    h = hsmm()
    for dtype, unit in ((torch.float64, 64), (torch.complex128, 32)):
        for k in (1, 9, 56, 57, 63, 65, 120, 129, 200, 516):
            kp = (k + unit - 1) // unit * unit
            A, Ap = _operand(m, k, kp, ta == "T", dtype, k)
            B, Bp = _operand(n, k, kp, tb == "N", dtype, k + 1000)      # rows of op(B)^T
            C, Cp = h.colmajor(m, n, dtype), h.colmajor(m, n, dtype)
            h.gemm(A, B, C, ta, tb, compute=h.COMPUTE_64F_OZAKI)
            h.gemm(Ap, Bp, Cp, ta, tb, compute=h.COMPUTE_64F_OZAKI)
            torch.cuda.synchronize()
            assert h.sync_status() == 0
            assert torch.equal(C, Cp), (dtype, k)


@pytest.mark.parametrize("dtype", [torch.float64, torch.complex128])
def test_panels_of_blocks(dtype):
    """gemm_host: row panels are rows in the middle of the blocks."""
    h = hsmm()
    m, n, k = (4200, 700, 1003) if dtype == torch.float64 else (4200, 300, 501)
    A = torch.randn(k, m, dtype=dtype).pin_memory().t()
    B = torch.randn(n, k, dtype=dtype).pin_memory().t()
    C = torch.empty(n, m, dtype=dtype).pin_memory().t()
    D = h.colmajor(m, n, dtype)
    h.gemm_host(A, B, C, compute=h.COMPUTE_64F_OZAKI)
    h.gemm(A.t().cuda().t(), B.t().cuda().t(), D, compute=h.COMPUTE_64F_OZAKI)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.equal(C, D.cpu())
