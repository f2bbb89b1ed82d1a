"""Digits of every width and count, lines across memory, bit-exact against the oracle's splitting: ends of
the scan's batches and of tiles, zeros without a sign, one value at a time where slices are unaligned."""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import dev_colmajor, hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("bits,s", [(2, 3), (4, 16), (6, 8), (7, 7), (7, 9), (7, 16)])
@pytest.mark.parametrize("lines,length", [(1, 1), (33, 65), (130, 383), (2, 3100), (4000, 25)])
@pytest.mark.parametrize("q_off", [0, 1])
def test_lines_across_memory(ora, bits, s, lines, length, q_off):
    h = hsmm()
    M = W.scaled_f64((lines, length), lines + length + s)
    M[0, 0] = 2.0 ** -1070 if length > 1 else 1.0
    ldq = (length + 7) // 8 * 8
    buf = torch.full((s * lines * ldq + q_off,), -1.0, dtype=torch.bfloat16, device="cuda")
    expo, q = h.ozaki_split(dev_colmajor(M), True, bits, s, q=buf[q_off:].view(s, lines, ldq))
    e_ref, q_ref = ora.ozaki_split(M, True, bits, s)
    assert np.array_equal(expo.cpu().numpy(), e_ref)
    got = q.float().cpu().numpy()
    assert (got[:, :, length:] == 0).all() and not np.signbit(got[got == 0]).any()
    assert np.array_equal(got[:, :, :length], q_ref)
