"""Products on CTA pairs with tiles narrower than 256 columns (224 or 192 where that saves part of a
last round): sizes that take each width, ragged last tiles, every majorness of A, FP32 and BF16 C,
beta.  The entries are small integers, so FP32 sums are exact and every value has one right answer."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def _ints(rows, cols, dtype, first, seed):
    """rows x cols, stored column-major (first: transposed)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    pad = lambda v: (v + 7) // 8 * 8
    if first:
        return torch.randint(-3, 4, (rows, pad(cols)), device="cuda", generator=g).to(dtype)[:, :cols].t()   # cols x rows
    return torch.randint(-3, 4, (cols, pad(rows)), device="cuda", generator=g).to(dtype)[:, :rows].t()


@pytest.mark.parametrize("ta", ["N", "T"])
@pytest.mark.parametrize("m,n,k", [(2048, 4096, 72), (1801, 4090, 200), (4392, 1384, 136), (4400, 1350, 64)])
@pytest.mark.parametrize("ab,out", [(torch.bfloat16, torch.float32), (torch.bfloat16, torch.bfloat16),
                                    (torch.float32, torch.float32)])
def test_widths(m, n, k, ta, ab, out, monkeypatch):
    monkeypatch.setenv("HSMM_GEMM_KERNEL", "pair")
    h = hsmm()
    A = _ints(m, k, ab, ta == "T", 1)            # op(A) = m x k
    B = _ints(k, n, ab, False, 2)
    exact = (A.t() if ta == "T" else A).double() @ B.double()
    compute = h.COMPUTE_DEFAULT if ab == torch.bfloat16 else h.COMPUTE_32F_FAST_TF32
    for beta in (0.0, 0.5):
        ldc = m + 8 - m % 8
        buf = torch.full((n, ldc), 4.0, dtype=out, device="cuda")
        C = buf.t()[:m]
        h.gemm(A, B, C, ta, "N", alpha=2.0, beta=beta, compute=compute)
        torch.cuda.synchronize()
        assert h.sync_status() == 0
        assert torch.equal(C, (2 * exact + beta * 4).float().to(out))
        assert (buf.t()[m:] == 4).all()
