"""Exact anti-diagonal sums where the slice-product kernel deals parts of tiles to the CTA pairs:
fewer tiles than pairs, one tile more than a whole wave, whole anti-diagonals and pieces of them
(summed with integer atomics into planes that hold garbage before the call)."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("m,n,k,s,bits", [
    (256, 256, 3000, 7, 7),        # one tile: single slice pairs
    (130, 90, 1500, 7, 7),         # one ragged tile
    (513, 600, 1100, 7, 7),        # 9 tiles, pieces
    (1000, 1200, 200, 7, 7),       # 20 tiles, whole anti-diagonals
    (1792, 2816, 700, 7, 7),       # 77 tiles: one more than a wave on 76 pairs
    (300, 300, 2000, 1, 7), (300, 300, 2000, 2, 7), (513, 300, 1000, 8, 6), (300, 513, 700, 16, 5)])
def test_slice_products_exact(m, n, k, s, bits):
    h = hsmm()
    ldq = (k + 7) // 8 * 8
    top = (1 << bits) - 1
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n + k + s)

    def slices(lines):
        q = torch.randint(-top, top + 1, (s, lines, ldq), device="cuda", generator=g).to(torch.bfloat16)
        q[:, :, k:] = 0
        return q

    qa, qb = slices(m), slices(n)
    sd = torch.full((s, n, m), -123456789, dtype=torch.int32, device="cuda")
    for _ in range(2):             # the second call finds the first one's sums
        h.hsmm.ozaki_slice_products(qa, qb, k, bits, sd=sd)
    assert h.sync_status() == 0
    for d in range(2, s + 2):
        want = torch.zeros((n, m), dtype=torch.float64, device="cuda")
        for t in range(max(1, d - s), min(s, d - 1) + 1):
            want += qb[d - t - 1].double() @ qa[t - 1].double().t()     # |sums| < 2^31: exact
        assert torch.equal(sd[d - 2].double(), want), f"d = {d}"
