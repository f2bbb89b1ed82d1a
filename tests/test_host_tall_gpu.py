"""Tall and narrow FP64-accurate products, where few row panels cost least: gemm_host takes what the
split takes in four panels (more than 65535 lines along the contraction, more than 2097120 across),
with the bits of gemm on device copies, and gemm itself takes more than 65535 lines either way."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _dev(rows, cols, seed, dtype=torch.float64):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(cols, rows, dtype=dtype, device="cuda", generator=g).t()


@pytest.mark.parametrize("m,n,k,ta,dtype", [(70000, 8, 16, "T", torch.float64), (131073, 40, 9, "T", torch.float64),
                                            (262140, 8, 8, "T", torch.float64), (66000, 5, 12, "C", torch.complex128),
                                            (2097121, 8, 8, "N", torch.float64)])
def test_tall_from_host(m, n, k, ta, dtype):
    h = hsmm()
    dA, dB = _dev(*((m, k) if ta == "N" else (k, m)), 1, dtype), _dev(k, n, 2, dtype)
    A, B, C = (x.t().cpu().pin_memory().t() for x in (dA, dB, _dev(m, n, 3, dtype)))
    want = _dev(m, n, 3, dtype)
    rows = dA if ta == "N" else (dA.t().conj() if ta == "C" else dA.t())      # op(A), by rows of up to 2^20
    for i in range(0, m, 1 << 20):
        part = rows[i:i + (1 << 20)].t().contiguous().t()
        c = want[i:i + (1 << 20)].t().contiguous().t()
        h.gemm(part, dB, c, beta=0.5, compute=h.COMPUTE_64F_OZAKI)
        want[i:i + (1 << 20)] = c
    h.gemm_host(A, B, C, ta, "N", beta=0.5, compute=h.COMPUTE_64F_OZAKI)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.equal(C, want.cpu())


@pytest.mark.parametrize("m,n,ta,tb", [(70000, 9, "T", "N"), (9, 70001, "N", "N"), (66001, 3, "T", "T")])
def test_long_sides_on_device(m, n, ta, tb):
    h = hsmm()
    k = 24
    A, B = _dev(m, k, 1), _dev(k, n, 2)
    want, got = _dev(m, n, 3), _dev(m, n, 3)
    def stored(x, op):                      # column-major, as op(x) reads it
        return x if op == "N" else x.contiguous().t()

    h.gemm(A, stored(B, "T"), want, "N", "T", compute=h.COMPUTE_64F_OZAKI)      # lines across the contraction
    h.gemm(stored(A, ta), stored(B, tb), got, ta, tb, compute=h.COMPUTE_64F_OZAKI)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.equal(want, got)


def test_more_lines_are_refused():
    h = hsmm()
    A, B, C = _dev(2097121, 1, 1), _dev(1, 1, 2), _dev(2097121, 1, 3)
    with pytest.raises(h.HsmmError) as e:
        h.gemm(A, B, C, compute=h.COMPUTE_64F_OZAKI)
    assert e.value.status == h.hsmm.NOT_SUPPORTED
