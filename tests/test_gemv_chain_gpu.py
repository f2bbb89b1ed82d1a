"""Matrix-vector products queued one behind the other, each reading what the one before wrote and
overwriting what it read: their kernels are placed before the previous one ends and wait for it on
the device.  The same calls with a synchronisation after each are the reference, bit for bit."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _matrix(dtype, m, n, ld, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if dtype == torch.int8:
        a = torch.randint(-3, 4, (n, ld), device="cuda", dtype=dtype, generator=g)
    else:
        a = torch.randn(n, ld, device="cuda", dtype=dtype, generator=g) / (m + n) ** 0.5
    return a.t()[:m]


def _chain(A, steps, wait):
    h = hsmm()
    m, n = A.shape
    i8 = A.dtype == torch.int8
    acc = torch.int32 if i8 else torch.float32
    x = torch.ones(n, device="cuda", dtype=A.dtype)
    y = torch.zeros(m, device="cuda", dtype=acc)
    xm = torch.empty(m, device="cuda", dtype=A.dtype)
    z = torch.zeros(n, device="cuda", dtype=acc)
    code = h.R_8I if i8 else h.R_32F
    ws = torch.empty(max(16, h.hsmm.gemv_workspace_size(code, "N", m, n)), dtype=torch.uint8, device="cuda")
    sync = torch.cuda.synchronize if wait else lambda: None
    for _ in range(steps):
        h.gemv(A, x, y, "N", beta=1, workspace=ws)
        sync()
        xm.copy_(y % 5 if i8 else y)
        sync()
        h.gemv(A, xm, z, "T", beta=1, workspace=ws)
        sync()
        if i8:
            x.copy_(z % 7)
        else:
            h.gemv(A, z, y, "N", workspace=ws)
            sync()
            h.gemv(A, y, x, "T", workspace=ws)
        sync()
    return [t.clone() for t in (x, y, z)]


# whole vectors, ragged rows, unaligned columns; the widest form of op = N (no wait of its own)
@pytest.mark.parametrize("dtype,m,n,ld", [
    (torch.float32, 1000, 1000, 1000), (torch.float32, 37, 5000, 40), (torch.float32, 501, 300, 501),
    (torch.float32, 8192, 4096, 8192), (torch.int8, 2100, 5300, 2112), (torch.int8, 777, 900, 777),
    (torch.int8, 16384, 2048, 16384)])
def test_queued_calls_wait_for_each_other(dtype, m, n, ld):
    A = _matrix(dtype, m, n, ld, m + n)
    want = _chain(A, 3, True)
    for _ in range(5):
        got = _chain(A, 3, False)
        torch.cuda.synchronize()
        for w, o in zip(want, got):
            assert torch.equal(w, o)
