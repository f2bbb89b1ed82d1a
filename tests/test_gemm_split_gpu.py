"""Products on narrow tiles with the contraction split over a cluster (gemm_split_tc.cu) against
the oracle: edges of the 128-row tiles, of the 16-column tile widths, of the k-blocks and of the
split, aligned and unaligned C, beta, every operand form and type.

Bound: FP32 accumulation of k exact products in any order, |C - C*| <= 2 gamma_k(2^-24) (|A||B|)
(TF32 inputs are rounded to TF32 values first, so their products are exact too), plus one BF16
rounding for BF16 results.
"""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import dev_bf16_colmajor, dev_colmajor, hsmm, padded, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.fixture(autouse=True)
def split_kernel(monkeypatch):
    monkeypatch.setenv("HSMM_GEMM_KERNEL", "split")


def tf32_values(shape, seed):
    """FP32 values with ten fraction bits: exact in TF32."""
    x = W.uniform_f32(shape, seed)
    return np.asfortranarray((x.view(np.uint32) & np.uint32(0xFFFFE000)).view(np.float32))


def run(ora, m, n, k, ta, tb, kind, alpha=1.0, beta=0.0, aligned=True):
    h = hsmm()
    sa, sb = ((m, k) if ta == "N" else (k, m)), ((k, n) if tb == "N" else (n, k))
    if kind == "tf32":
        A, B = tf32_values(sa, 11 + m), tf32_values(sb, 12 + n)
        A64, B64 = A.astype(np.float64), B.astype(np.float64)
        dA, dB = dev_colmajor(A, ld=padded(sa[0], 4)), dev_colmajor(B, ld=padded(sb[0], 4))
        out, compute = torch.float32, h.COMPUTE_32F_FAST_TF32
    else:
        Ab, Bb = W.uniform_bf16(sa, 13 + m), W.uniform_bf16(sb, 14 + n)
        A64, B64 = W.bf16_bits_to_f64(Ab), W.bf16_bits_to_f64(Bb)
        dA, dB = dev_bf16_colmajor(Ab, ld=padded(sa[0])), dev_bf16_colmajor(Bb, ld=padded(sb[0]))
        out, compute = (torch.bfloat16 if kind == "bf16" else torch.float32), h.COMPUTE_DEFAULT
    ldc = padded(m) + 8 if aligned else m + 3 + (m % 2)
    base = torch.full((n, ldc), float("nan"), dtype=out, device="cuda")
    C = base[:, :m].t()
    C0 = None
    if beta != 0.0:
        C0 = W.bf16_bits_to_f64(W.bf16_bits_from_f32(W.uniform_f32((m, n), 15)))
        C.copy_(torch.from_numpy(C0).to("cuda"))
    h.gemm(dA, dB, C, ta, tb, alpha=alpha, beta=beta, compute=compute)
    torch.cuda.synchronize()
    assert h.sync_status() == 0
    assert torch.isnan(base[:, m:].float()).all(), "rows beyond m were written"
    got = C.double().cpu().numpy()
    want = ora.gemm(A64, B64, ta, tb, alpha, beta, C0)
    mag = ora.gemm(np.abs(A64), np.abs(B64), ta, tb, abs(alpha))
    if C0 is not None:
        mag = mag + abs(beta) * np.abs(C0)
    gam = (k + 2) * 2.0 ** -24
    bound = 2 * gam * mag + 1e-30 + (2.0 ** -8 * np.abs(want) if out == torch.bfloat16 else 0.0)
    err = np.abs(got - want)
    assert (err <= bound).all(), float((err / bound).max())


@pytest.mark.parametrize("kind", ["f32", "bf16", "tf32"])
@pytest.mark.parametrize("ta,tb", [("N", "N"), ("T", "N"), ("N", "T"), ("T", "T")])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 15, 63), (128, 16, 64), (129, 17, 65), (300, 33, 520),
                                   (260, 130, 1000), (640, 257, 72), (64, 64, 128)])
def test_edges(ora, m, n, k, ta, tb, kind):
    run(ora, m, n, k, ta, tb, kind)


@pytest.mark.parametrize("kind", ["f32", "bf16", "tf32"])
@pytest.mark.parametrize("m,n,k", [(130, 16, 4100), (256, 72, 2048), (40, 9, 6000)])
def test_long_contraction_split_over_a_cluster(ora, m, n, k, kind):
    run(ora, m, n, k, "T", "N", kind)
    run(ora, m, n, k, "N", "T", kind)


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("kind", ["f32", "bf16", "tf32"])
@pytest.mark.parametrize("m,n,k", [(133, 20, 1500), (300, 100, 200)])
def test_alpha_beta_and_unaligned_c(ora, m, n, k, kind, aligned):
    run(ora, m, n, k, "T", "N", kind, alpha=-0.75, beta=1.25, aligned=aligned)
    run(ora, m, n, k, "T", "N", kind, aligned=aligned)


def test_sums_are_deterministic(ora):
    h = hsmm()
    A = dev_bf16_colmajor(W.uniform_bf16((4096, 512), 21))
    B = dev_bf16_colmajor(W.uniform_bf16((4096, 24), 22))
    C1, C2 = h.colmajor(512, 24, torch.float32), h.colmajor(512, 24, torch.float32)
    h.gemm(A, B, C1, "T", "N")
    h.gemm(A, B, C2, "T", "N")
    assert torch.equal(C1, C2)


def test_size_rule(monkeypatch):
    """Without the variable the size decides: either route gives the exact integer product."""
    monkeypatch.delenv("HSMM_GEMM_KERNEL")
    h = hsmm()
    for m, n, k in ((6144, 16, 512), (520, 1280, 256), (2048, 2304, 128), (16, 3000, 96)):
        A = torch.randint(-4, 5, (k, m), device="cuda").bfloat16().t()
        B = torch.randint(-4, 5, (n, k), device="cuda").bfloat16().t()
        C = h.colmajor(m, n, torch.float32)
        h.gemm(A, B, C)
        assert torch.equal(C.double(), A.double() @ B.double())
