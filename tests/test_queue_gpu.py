"""Calls queued one behind the other on one stream, each reading what the one before wrote and
overwriting what it read: native FP64 products, the two-array n^2 kernel, grouped products.  Their
kernels are placed before the previous one ends and wait for it on the device.  The same calls with
a synchronisation after each are the reference, bit for bit."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _rand(rows, cols, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(cols, rows, device="cuda", dtype=dtype, generator=g).t() / cols ** 0.5


def _native(h, n, dtype, sync):
    A, B, C = (_rand(n, n, dtype, s) for s in (1, 2, 3))
    for _ in range(4):
        for x, y, z in ((A, B, C), (C, A, B), (B, C, A)):
            h.gemm(x, y, z)
            sync()
    return A, B, C


def _nbody(h, n, dtype, sync):
    g = torch.Generator(device="cuda").manual_seed(n)
    x, z = torch.rand(2, n, 4, device="cuda", generator=g)
    out = torch.zeros_like(x)
    for _ in range(4):
        h.nbody(x, z, 1e-2, out)
        sync()
        h.nbody(out, x, 1e-2, z)
        sync()
    return x, z, out


def _grouped(h, n, dtype, sync):
    A, B = (_rand(n, n, dtype, s) for s in (1, 2))
    C, D = (torch.zeros(n, n, device="cuda", dtype=dtype).t() for _ in range(2))
    half = n // 2 // 8 * 8
    first = h.GroupedPlan([(A, B[:, :half], C[:, :half], "N", "N"), (A, B[:, half:], C[:, half:], "N", "N")],
                          h.R_16BF, h.R_16BF)
    second = h.GroupedPlan([(B, C, D, "N", "N")], h.R_16BF, h.R_16BF)
    third = h.GroupedPlan([(D, A, C, "N", "N")], h.R_16BF, h.R_16BF)
    for _ in range(4):
        for plan in (first, second, third):
            plan.launch()
            sync()
    return C, D


@pytest.mark.parametrize("chain,n,dtype", [
    (_native, 60, torch.float64), (_native, 300, torch.float64), (_native, 70, torch.complex128),
    (_nbody, 1000, torch.float32), (_nbody, 3001, torch.float32), (_grouped, 64, torch.bfloat16),
    (_grouped, 520, torch.bfloat16)])
def test_queued_calls_wait_for_each_other(chain, n, dtype):
    h = hsmm()
    want = [t.clone() for t in chain(h, n, dtype, torch.cuda.synchronize)]
    for _ in range(3):
        got = chain(h, n, dtype, lambda: None)
        torch.cuda.synchronize()
        assert h.sync_status() == 0
        for w, o in zip(want, got):
            assert torch.equal(w, o)
