"""C of a grouped launch stored in blocks of 128 rows, or of 32 where most of it lies on whole 32-byte
sectors: columns that begin or end inside a sector (odd multiples of 16 bytes in the leading dimension
or the base, ragged rows), short and long k (the edges are fetched ahead up to six k-blocks), tile
widths that end inside a block.  The entries are small integers, so FP32 sums are exact and every
value has one right answer."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

SHAPES = [(m, n, k) for k in (64, 384, 448, 1000) for m, n in
          [(1, 40), (8, 33), (127, 96), (128, 160), (129, 300), (255, 64), (256, 256), (257, 31), (300, 224), (700, 513)]]


def _ints(rows, cols, ld, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-3, 4, (cols, ld), device="cuda", generator=g).to(dtype).t()[:rows]


@pytest.mark.parametrize("ab,out", [("bf16", torch.float32), ("bf16", torch.bfloat16), ("tf32", torch.float32)])
@pytest.mark.parametrize("offset,extra,whole", [(0, 0, False), (1, 0, False), (0, 1, False), (1, 1, False),
                                                (0, 0, True)])
def test_blocks_of_c(ab, out, offset, extra, whole):
    h = hsmm()
    dt = torch.bfloat16 if ab == "bf16" else torch.float32
    unit = 16 // (4 if out == torch.float32 else 2)       # elements of 16 bytes
    bufs, probs = [], []
    for q, (m, n, k) in enumerate(SHAPES):
        if whole and q % 4:
            m = (m + 15) // 16 * 16                       # three in four on whole sectors
        A = _ints(m, k, (m + 7) // 8 * 8, dt, 2 * q)
        B = _ints(k, n, (k + 7) // 8 * 8, dt, 2 * q + 1)
        ldc = ((m + 2 * unit - 1) // (2 * unit) * 2 + extra) * unit
        buf = torch.full((offset * unit + n * ldc,), float("nan"), dtype=out, device="cuda")
        bufs.append(buf)
        probs.append((A, B, buf[offset * unit:].view(n, ldc).t()[:m], "N", "N"))
    plan = h.GroupedPlan(probs, h.R_16BF if ab == "bf16" else h.R_32F, h.R_32F if out == torch.float32 else h.R_16BF,
                         h.COMPUTE_DEFAULT if ab == "bf16" else h.COMPUTE_32F_FAST_TF32)
    for _ in range(2):
        plan.launch(alpha=2.0)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    for buf, (A, B, C, _, _) in zip(bufs, probs):
        want = (2 * (A.double() @ B.double())).to(torch.float32).to(out)
        assert torch.equal(C, want), C.shape
        C.fill_(float("nan"))                             # nothing else of the buffer was written
        assert torch.isnan(buf.float()).all(), C.shape
    plan.close()
