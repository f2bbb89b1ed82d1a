"""The CPython call module passes every argument through (bound to C callbacks here, no GPU)."""
import ctypes
import glob
import importlib.util
import os

import pytest

from paper_cs_9809105_gb300 import build as B
from paper_cs_9809105_gb300 import hsmm as H


@pytest.fixture(scope="module")
def call():
    B.build()
    paths = glob.glob(os.path.join(os.path.dirname(H.LIB_PATH), "_hsmmcall*.so"))
    if not paths:
        pytest.skip("no Python headers: the binding uses ctypes")
    spec = importlib.util.spec_from_file_location("_hsmmcall", paths[0])
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def bind(call, code):
    """Bind recorders of hsmm_gemm and hsmm_gemv; the scalars are read as the compute type."""
    i64, vp, ci = ctypes.c_int64, ctypes.c_void_p, ctypes.c_int
    cfgp = ctypes.POINTER(H.Config)
    seen = []

    def scalar(p):
        t = {H.R_64F: ctypes.c_double, H.R_32I: ctypes.c_int32, H.C_64F: ctypes.c_double * 2}.get(code, ctypes.c_float)
        v = ctypes.cast(p, ctypes.POINTER(t))[0]
        return complex(v[0], v[1]) if code == H.C_64F else v

    def fields(c):
        c = c[0]
        return [c.a, c.b, c.c, c.compute, c.ozaki_slices, c.ozaki_bits, c.workspace, c.workspace_bytes, c.tile_n, c.ring_p,
                c.ring_k, list(c.reserved)]

    G = ctypes.CFUNCTYPE(ci, cfgp, ci, ci, i64, i64, i64, vp, vp, i64, vp, i64, vp, vp, i64, vp)
    V = ctypes.CFUNCTYPE(ci, cfgp, ci, i64, i64, vp, vp, i64, vp, i64, vp, vp, i64, vp)

    def gemm(c, ta, tb, m, n, k, al, A, lda, Bp, ldb, be, C, ldc, st):
        seen.append((fields(c), ta, tb, m, n, k, scalar(al), A, lda, Bp, ldb, scalar(be), C, ldc, st))
        return 3

    def gemv(c, t, m, n, al, A, lda, x, incx, be, y, incy, st):
        seen.append((fields(c), t, m, n, scalar(al), A, lda, x, incx, scalar(be), y, incy, st))
        return 2

    keep = (G(gemm), V(gemv))
    call.bind(*(ctypes.cast(f, vp).value for f in keep))
    return seen, keep


@pytest.mark.parametrize("code,alpha,beta", [(H.R_64F, 1.25, -3), (H.R_32F, 0.5, 2.0), (H.C_64F, 1 - 2j, 3.0)])
def test_gemm_arguments(call, code, alpha, beta):
    seen, keep = bind(call, code)
    big = 1 << 63
    args = [0, 1, 2, 3, 7, 6, big + 256, 4096, 128, 4, 2, code, ord("T"), ord("N"), 1 << 33, 5, 6, 0x1000, 11, 0x2000,
            12, 0x3000, 13, 0x4000]
    assert call.gemm(*args, alpha, beta) == 3
    cfg, *rest = seen[0]
    assert cfg == [0, 1, 2, 3, 7, 6, big + 256, 4096, 128, 4, 2, [0] * 5]
    assert rest == [ord("T"), ord("N"), 1 << 33, 5, 6, alpha, 0x1000, 11, 0x2000, 12, beta, 0x3000, 13, 0x4000]


def test_gemv_arguments(call):
    seen, keep = bind(call, H.R_32I)
    args = [H.R_8I, H.R_32I, 0x100, 64, ord("N"), 9, 10, 0x1000, 16, 0x2000, 2, 0x3000, 3, 0]
    assert call.gemv(*args, 2 ** 32 - 5, 3.9) == 2       # INT32: wraps, a float is truncated as int() does
    cfg, *rest = seen[0]
    assert cfg[:4] == [H.R_8I, H.R_8I, H.R_32I, 0] and cfg[6:8] == [0x100, 64]
    assert rest == [ord("N"), 9, 10, -5, 0x1000, 16, 0x2000, 2, 3, 0x3000, 3, None]


def test_bad_arguments_raise(call):
    bind(call, H.R_32F)
    with pytest.raises(TypeError):
        call.gemv(1, 2)
    with pytest.raises(TypeError):
        call.gemv(*([1.5] + [0] * 13), 1.0, 0.0)
    with pytest.raises(TypeError):
        call.gemv(*([1, 1] + [0] * 12), 1j, 0.0)
