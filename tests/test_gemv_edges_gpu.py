"""Matrix-vector products at the edges of their kernels: rows that end inside a vector with aligned
columns (the last column ends the buffer), unaligned columns, few rows or few columns (a CTA's
threads on several column groups, several warps per column), empty column splits."""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

U32 = 2.0 ** -24


def exact_end(A, ld, dtype):
    """Column-major device copy whose storage ends with the last element of the last column; the
    padding rows of the other columns hold NaN (FP32) or 77."""
    m, n = A.shape
    buf = np.full((n - 1) * ld + m, np.nan if dtype == np.float32 else 77, dtype=dtype)
    for j in range(n):
        buf[j * ld:j * ld + m] = A[:, j]
    d = torch.from_numpy(buf).cuda()
    return d, torch.as_strided(d, (m, n), (1, ld))


SHAPES = [(5, 3), (127, 130), (129, 64), (1023, 66), (1025, 700), (2100, 531), (37, 16385), (16390, 9), (4099, 500),
          (300, 2500)]


@pytest.mark.parametrize("trans", ["N", "T"])
@pytest.mark.parametrize("pad", [16, 1])
@pytest.mark.parametrize("m,n", SHAPES)
def test_i8(ora, m, n, pad, trans):
    h = hsmm()
    A = W.integers((m, n), 1 + m, -128, 127, np.int8)
    x = W.integers((n if trans == "N" else m,), 2 + n, -128, 127, np.int8)
    keep, dA = exact_end(A, (m + pad - 1) // pad * pad, np.int8)
    y = torch.full((m if trans == "N" else n,), 5, dtype=torch.int32, device="cuda")
    h.gemv(dA, torch.from_numpy(x).cuda(), y, trans, alpha=2, beta=-3)
    want = ora.gemv_i8(A, x, trans, 2, -3, np.full(y.numel(), 5, np.int32))
    assert np.array_equal(y.cpu().numpy().astype(np.int64), want)


@pytest.mark.parametrize("trans", ["N", "T"])
@pytest.mark.parametrize("pad,incx", [(4, 1), (1, 1), (1, 3)])
@pytest.mark.parametrize("m,n", SHAPES)
def test_f32(ora, m, n, pad, incx, trans):
    h = hsmm()
    A = W.uniform_f32((m, n), 3 + m)
    lenx = n if trans == "N" else m
    x = W.uniform_f32((lenx * incx,), 4 + n)
    keep, dA = exact_end(A, (m + pad - 1) // pad * pad, np.float32)
    y = torch.zeros(m if trans == "N" else n, device="cuda")
    h.gemv(dA, torch.from_numpy(x).cuda(), y, trans, incx=incx)
    A64, x64 = A.astype(np.float64), x.astype(np.float64)
    want = ora.gemv(A64, x64, trans, 1.0, 0.0, None, incx, 1)
    mag = ora.gemv(np.abs(A64), np.abs(x64), trans, 1.0, 0.0, None, incx, 1)
    g = (lenx + 2) * U32 / (1 - (lenx + 2) * U32)
    assert (np.abs(y.double().cpu().numpy() - want) <= g * mag + 1e-38).all()
