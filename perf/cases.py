"""Performance cases of the library: what its users run, through the public entry points.

Every case is a dict of plain values with a "kind":

  precise   FP64-accurate product on the device (gemm, COMPUTE_64F_OZAKI), real or complex
  host      the same with A, B, C in page-locked host memory (gemm_host)
  native    product on the FP64 pipe (gemm, the default compute mode for FP64)
  train     forward and backward of one differentiable BF16 product (autograd.hsmm_matmul)
  linear    one row-major product of a layer at inference (matmul), BF16 or TF32
  gemv      matrix-vector products with one matrix, op = N and then op = T, FP32 or INT8
  grouped   many independent products in one launch, from a kept plan or described anew
  nbody     the two-array n^2 problem

Sizes of the largest cases are the workloads of ``workloads/`` (8192^3, 16384^2, 4096 x 2048 x
8192, 512 grouped problems); the others are generic, odd and ragged ones among them.
"""
from __future__ import annotations

import math
import random

import torch

import paper_cs_9809105_gb300 as h
from paper_cs_9809105_gb300.autograd import hsmm_matmul

DEV = "cuda"
SLICES = 7                              # digits per operand of the FP64-accurate form (the default)
PAIRS = SLICES * (SLICES + 1) // 2      # slice products it sums
NBODY_EPS2 = 1e-4


def listed():
    return [
        # the headline: a large FP64-accurate product with everything on the device
        dict(name="precise_8192", kind="precise", m=8192, n=8192, k=8192, ta="N", tb="N", alpha=1.0, beta=0.0,
             complex=False),
        # a small dense block of a solver: ragged, transposed, accumulated into C; launches count
        dict(name="precise_1000", kind="precise", m=1000, n=1200, k=900, ta="T", tb="N", alpha=1.5, beta=0.5,
             complex=False),
        # complex data, conjugate transpose (A^H B), odd sizes
        dict(name="zprecise_1500", kind="precise", m=1500, n=1100, k=2301, ta="C", tb="N", alpha=1.0, beta=0.0,
             complex=True),
        # the end-to-end call: operands and result in host memory
        dict(name="host_4096", kind="host", m=4096, n=4096, k=4096),
        # the default FP64 compute mode at a size of everyday linear algebra, odd leading dimension
        dict(name="native_700", kind="native", m=700, n=601, k=1000, ta="N", tb="T", complex=False),
        # a large training step of one layer, eager through the autograd engine
        dict(name="train_4096", kind="train", m=4096, k=2048, n=8192, graph=False),
        # a small one (few tokens, narrow layer), where a program captures the step in a CUDA graph
        dict(name="train_small", kind="train", m=520, k=1024, n=1280, graph=True),
        # a layer at inference with few rows: bound by reading the weights once
        dict(name="linear_16", kind="linear", m=16, k=4096, n=6144, dtype="bf16"),
        # an iterative solver's A x and A^T y on a large FP32 matrix: HBM streaming
        dict(name="gemv_f32_16384", kind="gemv", m=16384, n=16384, dtype="f32", pad=1),
        # the same on a small quantised matrix with ragged sizes, columns padded to 16 bytes
        dict(name="gemv_i8_2100", kind="gemv", m=2100, n=5300, dtype="i8", pad=16),
        # many uneven products in one launch from a kept plan
        dict(name="grouped_512", kind="grouped", count=512, lo=64, hi=2048, dtype="bf16", ta="N", tb="N", plan=True,
             shapes=7),
        # an n-body force evaluation of ordinary size
        dict(name="nbody_20000", kind="nbody", nx=20000, nz=20000),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _mult8(v):
    return max(8, (v + 4) // 8 * 8)


def draw(rng):
    kind = rng.choice(["precise", "precise", "host", "native", "train", "train", "linear", "linear", "gemv", "gemv",
                       "grouped", "nbody"])
    if kind == "precise":
        cplx = rng.random() < 0.3
        hi = 3000 if cplx else 8192
        ops = ["N", "T", "C"] if cplx else ["N", "T"]
        return dict(kind=kind, m=_logint(rng, 128, hi), n=_logint(rng, 128, hi), k=_logint(rng, 128, hi),
                    ta=rng.choice(ops), tb=rng.choice(ops), alpha=rng.choice([1.0, -0.75]),
                    beta=rng.choice([0.0, 0.5]), complex=cplx)
    if kind == "host":
        return dict(kind=kind, m=_logint(rng, 512, 4096), n=_logint(rng, 512, 4096), k=_logint(rng, 512, 4096))
    if kind == "native":
        cplx = rng.random() < 0.3
        hi = 700 if cplx else 2000
        return dict(kind=kind, m=_logint(rng, 64, hi), n=_logint(rng, 64, hi), k=_logint(rng, 64, hi),
                    ta=rng.choice(["N", "T"]), tb=rng.choice(["N", "T"]), complex=cplx)
    if kind == "train":
        m, k, n = _mult8(_logint(rng, 64, 4096)), _mult8(_logint(rng, 256, 2048)), _mult8(_logint(rng, 256, 8192))
        return dict(kind=kind, m=m, k=k, n=n, graph=m * k * n < 1 << 32)
    if kind == "linear":
        return dict(kind=kind, m=_logint(rng, 1, 2048), k=_mult8(_logint(rng, 512, 8192)),
                    n=_mult8(_logint(rng, 512, 8192)), dtype=rng.choice(["bf16", "bf16", "tf32"]))
    if kind == "gemv":
        dtype = rng.choice(["f32", "i8"])
        return dict(kind=kind, m=_logint(rng, 500, 16384), n=_logint(rng, 500, 16384), dtype=dtype,
                    pad=rng.choice([1, 4 if dtype == "f32" else 16]))
    if kind == "grouped":
        return dict(kind=kind, count=_logint(rng, 8, 512), lo=64, hi=rng.choice([512, 1024, 2048]),
                    dtype=rng.choice(["bf16", "bf16", "tf32"]), ta=rng.choice(["N", "T"]), tb=rng.choice(["N", "T"]),
                    plan=rng.random() < 0.6, shapes=rng.randrange(1 << 20))
    n = _logint(rng, 1000, 100000)
    return dict(kind=kind, nx=n, nz=rng.choice([n, _logint(rng, 1000, 100000)]))


# ---- inputs --------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _colmajor(rows, cols, dtype, ld=None):
    """Zero-filled column-major rows x cols tensor with leading dimension ld."""
    ld = max(1, rows) if ld is None else ld
    return torch.zeros((cols, ld), dtype=dtype, device=DEV).t()[:rows]


def _scaled_f64(rows, cols, g):
    """s 2^e with s ~ U(1, 2), a random sign and e uniform in [-12, 12], column-major."""
    out = torch.rand((cols, rows), dtype=torch.float64, device=DEV, generator=g).add_(1.0)
    out *= 1 - 2 * torch.randint(0, 2, (cols, rows), device=DEV, generator=g, dtype=torch.int8)
    e = torch.randint(-12, 13, (cols, rows), device=DEV, generator=g, dtype=torch.int8)
    return (out * torch.exp2(e.double())).t()


def _scaled(rows, cols, cplx, g):
    if not cplx:
        return _scaled_f64(rows, cols, g)
    re, im = _scaled_f64(rows, cols, g), _scaled_f64(rows, cols, g)
    return torch.complex(re.t().contiguous(), im.t().contiguous()).t()


def _shape(rows, cols, op):
    return (rows, cols) if op == "N" else (cols, rows)


def _op(x, op):
    return x if op == "N" else x.t() if op == "T" else x.t().conj()


def _pad(v, mult):
    return (v + mult - 1) // mult * mult


def _group_shapes(case):
    r = random.Random(case["shapes"])
    return [tuple(_logint(r, case["lo"], case["hi"]) for _ in range(3)) for _ in range(case["count"])]


def _precise_inputs(case, seed):
    g = _gen(seed)
    m, n, k, cplx = case["m"], case["n"], case["k"], case.get("complex", False)
    A = _scaled(*_shape(m, k, case.get("ta", "N")), cplx, g)
    B = _scaled(*_shape(k, n, case.get("tb", "N")), cplx, g)
    C = _colmajor(m, n, torch.complex128 if cplx else torch.float64)
    if case.get("beta", 0.0) != 0.0:
        C.copy_(_scaled(m, n, cplx, g))
    return A, B, C


def _native_inputs(case, seed):
    g = _gen(seed)
    dt = torch.complex128 if case["complex"] else torch.float64

    def uniform(rows, cols):
        x = torch.rand((cols, rows), dtype=torch.float64, device=DEV, generator=g).mul_(2).sub_(1)
        if case["complex"]:
            x = torch.complex(x, torch.rand((cols, rows), dtype=torch.float64, device=DEV, generator=g))
        return x.t()

    A = uniform(*_shape(case["m"], case["k"], case["ta"]))
    B = uniform(*_shape(case["k"], case["n"], case["tb"]))
    return A, B, _colmajor(case["m"], case["n"], dt)


def _train_inputs(case, seed):
    g = _gen(seed)
    m, k, n = case["m"], case["k"], case["n"]
    a = (torch.randn((m, k), device=DEV, generator=g) / math.sqrt(k)).bfloat16()
    b = (torch.randn((k, n), device=DEV, generator=g) / math.sqrt(k)).bfloat16()
    return a, b, torch.randn((m, n), device=DEV, generator=g).bfloat16()


def _linear_inputs(case, seed):
    g = _gen(seed)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    x = torch.randn((case["m"], case["k"]), device=DEV, generator=g)
    w = torch.randn((case["n"], case["k"]), device=DEV, generator=g) / math.sqrt(case["k"])
    return x.to(dt), w.to(dt)           # weights stored (out, in), as layers store them


def _gemv_inputs(case, seed):
    g = _gen(seed)
    m, n = case["m"], case["n"]
    if case["dtype"] == "f32":
        def make(shape):
            return torch.rand(shape, device=DEV, generator=g).mul_(2).sub_(1)
    else:
        def make(shape):
            return torch.randint(-128, 128, shape, device=DEV, generator=g, dtype=torch.int8)
    A = make((n, _pad(m, case["pad"]))).t()[:m]
    return A, make((n,)), make((m,))


def _grouped_inputs(case, seed):
    """Problems on flat buffers; every C is a column-major view of one flat tensor."""
    g = _gen(seed)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    align = 8 if dt == torch.bfloat16 else 4
    shapes = _group_shapes(case)

    def flat(sizes, dtype, fill):
        total = sum(c * _pad(r, align) for r, c in sizes)
        if fill:
            buf = torch.rand(total, device=DEV, generator=g).mul_(2).sub_(1).to(dtype)
        else:
            buf = torch.zeros(total, dtype=dtype, device=DEV)
        views, at = [], 0
        for r, c in sizes:
            ld = _pad(r, align)
            views.append(buf[at:at + c * ld].view(c, ld).t()[:r])
            at += c * ld
        return buf, views

    _, As = flat([_shape(m, k, case["ta"]) for m, n, k in shapes], dt, True)
    _, Bs = flat([_shape(k, n, case["tb"]) for m, n, k in shapes], dt, True)
    buf, Cs = flat([(m, n) for m, n, k in shapes], torch.float32, False)
    return buf, [(a, b, c, case["ta"], case["tb"]) for a, b, c in zip(As, Bs, Cs)]


def _nbody_inputs(case, seed):
    g = _gen(seed)

    def bodies(n):      # positions uniform in the unit ball, masses uniform in [0.5, 1.5] / n
        d = torch.randn((n, 3), device=DEV, generator=g)
        d /= d.norm(dim=1, keepdim=True)
        d *= torch.rand((n, 1), device=DEV, generator=g) ** (1.0 / 3.0)
        m = (torch.rand((n, 1), device=DEV, generator=g) + 0.5) / n
        return torch.cat([d, m], 1).contiguous()

    x = bodies(case["nx"])
    return x, x if case["nz"] == case["nx"] else bodies(case["nz"])


# ---- one pass ------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind in ("precise", "host"):
        s["A"], s["B"], s["C"] = _precise_inputs(case, seed)
        if kind == "host":
            for name in "ABC":          # column-major in page-locked host memory
                s[name] = s[name].t().contiguous().cpu().pin_memory().t()
            cfg = h.hsmm.make_config(h.R_64F, h.R_64F, h.R_64F, h.COMPUTE_64F_OZAKI)
            need = h.hsmm.gemm_host_workspace_size(cfg, "N", "N", case["m"], case["n"], case["k"])
        else:
            t = h.C_64F if case["complex"] else h.R_64F
            need = h.workspace_size(h.hsmm.make_config(t, t, t, h.COMPUTE_64F_OZAKI), case["ta"], case["tb"],
                                    case["m"], case["n"], case["k"])
        s["ws"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    elif kind == "native":
        s["A"], s["B"], s["C"] = _native_inputs(case, seed)
    elif kind == "train":
        a, b, g = _train_inputs(case, seed)
        s["a"], s["b"], s["g"] = a.requires_grad_(), b.requires_grad_(), g
        if case["graph"]:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                _train_step(s)
            torch.cuda.current_stream().wait_stream(side)
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                s["out"] = _train_step(s)
    elif kind == "linear":
        s["x"], s["w"] = _linear_inputs(case, seed)
    elif kind == "gemv":
        s["A"], s["x"], s["z"] = _gemv_inputs(case, seed)
        dt = torch.float32 if case["dtype"] == "f32" else torch.int32
        s["y"] = torch.zeros(case["m"], dtype=dt, device=DEV)
        s["v"] = torch.zeros(case["n"], dtype=dt, device=DEV)
        need = h.hsmm.gemv_workspace_size(h.R_32F if case["dtype"] == "f32" else h.R_8I, "N", case["m"], case["n"])
        s["ws"] = torch.empty(max(need, 16), dtype=torch.uint8, device=DEV)
    elif kind == "grouped":
        s["out"], s["problems"] = _grouped_inputs(case, seed)
        tf32 = case["dtype"] != "bf16"
        s["ab"] = h.R_32F if tf32 else h.R_16BF
        s["compute"] = h.COMPUTE_32F_FAST_TF32 if tf32 else h.COMPUTE_DEFAULT
        if case["plan"]:
            s["plan"] = h.GroupedPlan(s["problems"], s["ab"], h.R_32F, s["compute"])
        else:
            need = h.gemm_grouped_workspace_size(s["problems"], s["ab"], h.R_32F, s["compute"])
            s["ws"] = torch.empty(max(need, 256), dtype=torch.uint8, device=DEV)
    else:
        s["x"], s["z"] = _nbody_inputs(case, seed)
        s["out"] = torch.empty_like(s["x"])
    return s


def _train_step(s):
    s["a"].grad = None
    s["b"].grad = None
    y = hsmm_matmul(s["a"], s["b"])
    y.backward(s["g"])
    return [y.detach(), s["a"].grad, s["b"].grad]


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "precise":
        return h.gemm(s["A"], s["B"], s["C"], case["ta"], case["tb"], case["alpha"], case["beta"],
                      compute=h.COMPUTE_64F_OZAKI, workspace=s["ws"])
    if kind == "host":
        return h.gemm_host(s["A"], s["B"], s["C"], compute=h.COMPUTE_64F_OZAKI, workspace=s["ws"])
    if kind == "native":
        return h.gemm(s["A"], s["B"], s["C"], case["ta"], case["tb"])
    if kind == "train":
        if case["graph"]:
            s["graph"].replay()
            return s["out"]
        return _train_step(s)
    if kind == "linear":
        if case["dtype"] == "bf16":
            return h.matmul(s["x"], s["w"], trans_b=True, out_dtype=torch.bfloat16)
        return h.matmul(s["x"], s["w"], trans_b=True, compute=h.COMPUTE_32F_FAST_TF32)
    if kind == "gemv":
        h.gemv(s["A"], s["x"], s["y"], "N", workspace=s["ws"])
        h.gemv(s["A"], s["z"], s["v"], "T", workspace=s["ws"])
        return [s["y"], s["v"]]
    if kind == "grouped":
        if case["plan"]:
            s["plan"].launch()
        else:
            h.gemm_grouped(s["problems"], s["ab"], h.R_32F, s["compute"], workspace=s["ws"])
        return s["out"]
    return h.nbody(s["x"], s["z"], NBODY_EPS2, s["out"])


# ---- what a pass cannot do without ---------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("precise", "host", "native"):
        m, n, k = case["m"], case["n"], case["k"]
        z = 2 if case.get("complex", False) else 1
        flops = 2.0 * m * n * k * z * z
        if kind != "native":
            flops *= PAIRS              # BF16 slice products: the FP64 pipe is some 1500 times slower
        c = 2 if case.get("beta", 0.0) != 0.0 else 1
        return {"bytes": 8.0 * z * (m * k + k * n + c * m * n), "flops": flops}
    if kind == "train":
        m, k, n = case["m"], case["k"], case["n"]
        return {"bytes": 2.0 * (2 * m * k + 2 * k * n + 2 * m * n), "flops": 6.0 * m * k * n}
    if kind == "linear":
        m, k, n = case["m"], case["k"], case["n"]
        return {"bytes": (2.0 if case["dtype"] == "bf16" else 4.0) * (m * k + k * n + m * n),
                "flops": 2.0 * m * k * n}
    if kind == "gemv":
        m, n = case["m"], case["n"]     # the matrix is read once by each of the two products
        e = 4.0 if case["dtype"] == "f32" else 1.0
        return {"bytes": e * (2 * m * n + m + n) + 4.0 * (m + n), "flops": 4.0 * m * n}
    if kind == "grouped":
        e = 2.0 if case["dtype"] == "bf16" else 4.0
        shapes = _group_shapes(case)
        return {"bytes": sum(e * (m * k + k * n) + 4.0 * m * n for m, n, k in shapes),
                "flops": sum(2.0 * m * n * k for m, n, k in shapes)}
    nx, nz = case["nx"], case["nz"]     # 12 FP32 operations and a reciprocal square root a pair
    return {"bytes": 16.0 * (2 * nx + (0 if nz == nx else nz)), "flops": 20.0 * nx * nz}


# ---- the same in 64 bits -------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind in ("precise", "host", "native"):
        A, B, C = _native_inputs(case, seed) if kind == "native" else _precise_inputs(case, seed)
        P = _op(A, case.get("ta", "N")) @ _op(B, case.get("tb", "N"))
        P = case.get("alpha", 1.0) * P
        if case.get("beta", 0.0) != 0.0:
            P += case["beta"] * C
        return P
    if kind == "train":
        a, b, g = (x.double() for x in _train_inputs(case, seed))
        return [a @ b, g @ b.t(), a.t() @ g]
    if kind == "linear":
        x, w = (t.double() for t in _linear_inputs(case, seed))
        return x @ w.t()
    if kind == "gemv":
        A, x, z = _gemv_inputs(case, seed)
        if case["dtype"] == "i8":       # |sums| <= 2^28: exact in FP64
            A, x, z = A.double(), x.double(), z.double()
            return [(A @ x).to(torch.int32), (A.t() @ z).to(torch.int32)]
        cols = 2048                     # in column blocks: the matrix in 64 bits need not exist at once
        y = torch.zeros(case["m"], dtype=torch.float64, device=DEV)
        v = torch.zeros(case["n"], dtype=torch.float64, device=DEV)
        for j in range(0, case["n"], cols):
            Aj = A[:, j:j + cols].double()
            y += Aj @ x[j:j + cols].double()
            v[j:j + cols] = Aj.t() @ z.double()
        return [y, v]
    if kind == "grouped":
        buf, problems = _grouped_inputs(case, seed)
        out = torch.zeros(buf.numel(), dtype=torch.float64, device=DEV)
        at = 0
        for A, B, C, ta, tb in problems:
            m, n = C.shape
            ld = C.stride(1) if n > 1 else _pad(m, 8 if case["dtype"] == "bf16" else 4)
            out[at:at + n * ld].view(n, ld).t()[:m].copy_(_op(A.double(), ta) @ _op(B.double(), tb))
            at += n * ld
        return out
    x, z = (t.double() for t in _nbody_inputs(case, seed))
    out = torch.zeros((case["nx"], 4), dtype=torch.float64, device=DEV)
    rows = max(1, (1 << 25) // case["nz"])
    for i in range(0, case["nx"], rows):
        d = z[None, :, :3] - x[i:i + rows, None, :3]
        r2 = (d * d).sum(-1) + NBODY_EPS2
        out[i:i + rows, :3] = ((z[None, :, 3] * r2.pow(-1.5))[:, :, None] * d).sum(1)
    return out
