"""Lines along memory that are scanned and sliced by two kernels (digits other than seven of seven bits,
real lines over 8192 entries, complex lines that do not fit three CTAs an SM), bit-exact: one to eight
warps a line, clusters of one to eight CTAs, ragged ends, unaligned loads and stores, row panels."""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import dev_colmajor, hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("by_rows", [True, False])
@pytest.mark.parametrize("bits,s", [(6, 9), (7, 10), (2, 16), (7, 7)])
@pytest.mark.parametrize("lines,length", [(1, 1), (9, 33), (300, 127), (3, 1025), (2700, 132), (5, 8193), (2, 16390)])
@pytest.mark.parametrize("pad,q_off", [(0, 0), (1, 0), (0, 1)])
def test_digits_and_lengths(ora, by_rows, bits, s, lines, length, pad, q_off):
    h = hsmm()
    rows, cols = (lines, length) if by_rows else (length, lines)
    M = W.scaled_f64((rows, cols), lines + length + bits)
    if lines > 1:
        M[(1, slice(None)) if by_rows else (slice(None), 1)] = 0.0
    ldq = (length + 7) // 8 * 8
    buf = torch.full((s * lines * ldq + q_off,), -1.0, dtype=torch.bfloat16, device="cuda")
    expo, q = h.ozaki_split(dev_colmajor(M, ld=(rows + 1) // 2 * 2 + pad), by_rows, bits, s,
                            q=buf[q_off:].view(s, lines, ldq))
    e_ref, q_ref = ora.ozaki_split(M, by_rows, bits, s)
    assert np.array_equal(expo.cpu().numpy(), e_ref)
    got = q.float().cpu().numpy()
    assert (got[:, :, length:] == 0).all() and not np.signbit(got[got == 0]).any()
    assert np.array_equal(got[:, :, :length], q_ref if by_rows else np.transpose(q_ref, (0, 2, 1)))


@pytest.mark.parametrize("ta,tb", [("T", "N"), ("C", "N"), ("T", "T"), ("N", "C")])
@pytest.mark.parametrize("m,n,k", [(3, 4, 4336), (3, 4, 4337), (160, 150, 5003), (2, 3, 9000)])
@pytest.mark.parametrize("bits,s", [(7, 7), (5, 8)])
def test_complex_lines(m, n, k, ta, tb, bits, s):
    """op(A) op(B) equals the product of the real matrices it stands for, by the same method."""
    h = hsmm()
    kw = {"compute": h.COMPUTE_64F_OZAKI, "slices": s, "bits": bits}
    g = torch.Generator(device="cuda").manual_seed(m + k)

    def rand(rows, cols):
        return torch.randn(cols, rows, 2, dtype=torch.float64, device="cuda", generator=g).view(cols, rows * 2).view(
            torch.complex128).t()

    A = rand(*((m, k) if ta == "N" else (k, m)))
    B = rand(*((k, n) if tb == "N" else (n, k)))
    C = torch.zeros((n, m), dtype=torch.complex128, device="cuda").t()
    h.gemm(A, B, C, ta, tb, **kw)
    op = {"N": lambda x: x, "T": lambda x: x.t(), "C": lambda x: x.t().conj()}
    a, b = op[ta](A).resolve_conj(), op[tb](B).resolve_conj()
    Ar = torch.cat([a.real, a.imag], 1).t().contiguous().t()
    Br = torch.cat([torch.cat([b.real, b.imag], 1), torch.cat([-b.imag, b.real], 1)], 0).t().contiguous().t()
    R = torch.zeros((2 * n, m), dtype=torch.float64, device="cuda").t()
    h.gemm(Ar, Br, R, **kw)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.equal(C.real, R[:, :n]) and torch.equal(C.imag, R[:, n:])


@pytest.mark.parametrize("m,n,k,bits,s,dtype", [(1500, 1300, 1001, 6, 8, torch.float64),
                                                (600, 600, 9001, 7, 7, torch.float64),
                                                (700, 600, 4500, 7, 7, torch.complex128)])
def test_row_panels(m, n, k, bits, s, dtype):
    h = hsmm()
    g = torch.Generator().manual_seed(k)
    A, B = (torch.randn(r, k, dtype=dtype, generator=g).pin_memory().t() for r in (m, n))      # k x m, k x n
    C = torch.zeros(n, m, dtype=dtype).pin_memory().t()
    D = C.t().cuda().t()
    kw = {"compute": h.COMPUTE_64F_OZAKI, "slices": s, "bits": bits}
    h.gemm_host(A, B, C, "T", "N", **kw)
    h.gemm(A.t().cuda().t(), B.t().cuda().t(), D, "T", "N", **kw)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.equal(C, D.cpu())
