"""Splitting kernels at the edges of their schedules, bit-exact: lines held by one to eight warps
and longer ones, clusters of one to eight CTAs, ragged tiles; complex operands against the real
split of the real form they stand for."""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import dev_colmajor, hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("by_rows", [True, False])
@pytest.mark.parametrize("lines,length", [(1, 1), (9, 1024), (9, 1032), (5, 2049), (3, 4097), (3, 8192), (2, 8200),
                                          (2, 20001), (31, 65), (129, 130), (2600, 40), (70, 1100)])
@pytest.mark.parametrize("pad", [0, 1])
def test_split_lines(ora, by_rows, lines, length, pad):
    """pad = 1: an odd leading dimension, no 16-byte loads."""
    h = hsmm()
    rows, cols = (lines, length) if by_rows else (length, lines)
    M = W.scaled_f64((rows, cols), lines + length)
    if lines > 1:
        M[(1, slice(None)) if by_rows else (slice(None), 1)] = 0.0
    ld = (rows + 1) // 2 * 2 + pad
    expo, q = h.ozaki_split(dev_colmajor(M, ld=ld), by_rows, 7, 7)
    e_ref, q_ref = ora.ozaki_split(M, by_rows, 7, 7)
    assert np.array_equal(expo.cpu().numpy(), e_ref)
    got = q.float().cpu().numpy()
    assert (got[:, :, length:] == 0).all()
    assert np.array_equal(got[:, :, :length], q_ref if by_rows else np.transpose(q_ref, (0, 2, 1)))


@pytest.mark.parametrize("ta", ["N", "T", "C"])
@pytest.mark.parametrize("tb", ["N", "T", "C"])
@pytest.mark.parametrize("m,n,k", [(5, 7, 1), (33, 40, 66), (64, 34, 67), (37, 33, 132), (3, 2, 13001), (40, 3, 2053)])
def test_complex_operands_equal_their_real_form(ora, ta, tb, m, n, k):
    h = hsmm()
    # seven slices of seven bits take contractions up to 19018 (2^31 / (7 127^2)); longer ones fewer bits
    kw = {"compute": h.COMPUTE_64F_OZAKI} if 2 * k < 19018 else {"compute": h.COMPUTE_64F_OZAKI, "slices": 9, "bits": 5}
    A = W.scaled_c128((m, k) if ta == "N" else (k, m), 3 + m)
    B = W.scaled_c128((k, n) if tb == "N" else (n, k), 4 + n)
    C = torch.zeros((n, m), dtype=torch.complex128, device="cuda").t()
    h.gemm(dev_colmajor(A), dev_colmajor(B), C, ta, tb, **kw)
    op = {"N": lambda x: x, "T": lambda x: x.T, "C": lambda x: x.conj().T}
    a, b = op[ta](A), op[tb](B)
    Ar = np.asfortranarray(np.hstack([a.real, a.imag]))
    Br = np.asfortranarray(np.vstack([np.hstack([b.real, b.imag]), np.hstack([-b.imag, b.real])]))
    R = torch.zeros((2 * n, m), dtype=torch.float64, device="cuda").t()
    h.gemm(dev_colmajor(Ar), dev_colmajor(Br), R, **kw)
    assert torch.equal(C.real, R[:, :n]) and torch.equal(C.imag, R[:, n:])
