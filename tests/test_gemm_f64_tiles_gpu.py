"""Native FP64 products, real and complex, at sizes that take each tile edge (64, 32, 16, 8) and at
their ragged edges: |C - C*| <= gamma_k(2^-53) times the sums of magnitudes (complex: two
products a part, gamma_2k)."""
import numpy as np
import pytest
import torch

import workloads as W
from _gpu import dev_colmajor, hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

U = 2.0 ** -53


@pytest.mark.parametrize("ta,tb", [("N", "N"), ("T", "N"), ("N", "T"), ("T", "T")])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (7, 9, 17), (64, 65, 33), (100, 300, 40), (257, 129, 31), (700, 601, 20),
                                   (1100, 1000, 19), (2500, 2000, 16)])
def test_real(ora, m, n, k, ta, tb):
    h = hsmm()
    A = W.uniform_f64((m, k) if ta == "N" else (k, m), 1 + m)
    B = W.uniform_f64((k, n) if tb == "N" else (n, k), 2 + n)
    C0 = W.uniform_f64((m, n), 3)
    C = dev_colmajor(C0, ld=m + 3)
    h.gemm(dev_colmajor(A, ld=A.shape[0] + 1), dev_colmajor(B), C, ta, tb, alpha=-1.5, beta=0.5)
    want = ora.gemm(A, B, ta, tb, -1.5, 0.5, C0)
    mag = 1.5 * ora.gemm(np.abs(A), np.abs(B), ta, tb) + 0.5 * np.abs(C0)
    err = np.abs(C.cpu().numpy() - want)
    assert (err <= 2 * (k + 3) * U * mag).all()      # both sides round


@pytest.mark.parametrize("ta,tb", [("N", "N"), ("C", "T"), ("T", "C")])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (9, 7, 17), (33, 65, 20), (130, 300, 18), (700, 500, 17)])
def test_complex(ora, m, n, k, ta, tb):
    h = hsmm()
    A = W.scaled_c128((m, k) if ta == "N" else (k, m), 5 + m, -1, 1)
    B = W.scaled_c128((k, n) if tb == "N" else (n, k), 6 + n, -1, 1)
    C = torch.full((n, m), float("nan"), dtype=torch.complex128, device="cuda").t()
    h.gemm(dev_colmajor(A), dev_colmajor(B), C, ta, tb, compute=h.COMPUTE_64F_NATIVE)
    op = {"N": lambda x: x, "T": lambda x: x.T, "C": lambda x: x.conj().T}
    a, b = op[ta](A), op[tb](B)
    want = a @ b
    mag = (np.abs(a.real) + np.abs(a.imag)) @ (np.abs(b.real) + np.abs(b.imag))
    got = C.cpu().numpy()
    bound = 2 * (2 * k + 3) * U * mag
    assert (np.abs(got.real - want.real) <= bound).all() and (np.abs(got.imag - want.imag) <= bound).all()
