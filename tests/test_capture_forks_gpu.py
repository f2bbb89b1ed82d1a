"""Dependent launches behind something else than the kernel before them on their stream: copies, memsets
and joined branches, eager and captured.  Each call reads what the other branch wrote."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

N = 328


def _rand(dtype, seed, rows=N, cols=N):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.rand(cols, rows, device="cuda", dtype=torch.float64, generator=g) - 0.5).to(dtype).t()


def _gemv(h, s, st):
    h.gemv(st["A32"], st["x"], st["y"], "N", workspace=st["gws"], stream=s)
    h.gemv(st["A32"], st["x"], st["x2"], "T", workspace=st["gws"], stream=s)
    return [st["y"], st["x2"]]


def _native(h, s, st):
    h.gemm(st["A64"], st["B64"], st["C64"], stream=s)
    return [st["C64"]]


def _precise(h, s, st):
    h.gemm(st["A64"], st["B64"], st["C64"], "N", "T", compute=h.COMPUTE_64F_OZAKI, workspace=st["ws"], stream=s)
    return [st["C64"]]


def _nbody(h, s, st):
    h.nbody(st["bodies"], st["bodies"], 1e-2, st["out"], stream=s)
    return [st["out"]]


def _bf16(h, s, st):
    h.gemm(st["A16"], st["A16"], st["C32"], "T", "N", stream=s)
    return [st["C32"]]


def _plan(h, s, st):
    st["plan"].launch(stream=s)
    return [st["C32"]]


def _state(h):
    st = {"A32": _rand(torch.float32, 1), "x": _rand(torch.float32, 2, N, 1)[:, 0].contiguous(),
          "y": torch.zeros(N, device="cuda"), "x2": torch.zeros(N, device="cuda"), "A64": _rand(torch.float64, 3),
          "B64": _rand(torch.float64, 4), "C64": torch.zeros(N, N, dtype=torch.float64, device="cuda").t(),
          "bodies": _rand(torch.float32, 5, 4, N).t().contiguous().clone(), "out": torch.zeros(N, 4, device="cuda"),
          "A16": _rand(torch.bfloat16, 6), "C32": torch.zeros(N, N, device="cuda").t()}
    st["gws"] = torch.empty(max(16, h.hsmm.gemv_workspace_size(h.R_32F, "N", N, N)), dtype=torch.uint8, device="cuda")
    need = h.workspace_size(h.hsmm.make_config(h.R_64F, h.R_64F, h.R_64F, h.COMPUTE_64F_OZAKI), "N", "T", N, N, N)
    st["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    st["plan"] = h.GroupedPlan([(st["A16"], st["A16"], st["C32"], "N", "T")], h.R_16BF, h.R_32F)
    return st


INPUT = {_gemv: "A32", _native: "A64", _precise: "A64", _nbody: "bodies", _bf16: "A16", _plan: "A16"}


@pytest.mark.parametrize("call", list(INPUT), ids=lambda f: f.__name__[1:])
@pytest.mark.parametrize("captured", [False, True])
def test_calls_behind_other_work(call, captured):
    h = hsmm()
    st = _state(h)
    src = st[INPUT[call]]
    base, other = src.clone(), src.clone() * 0.5
    s, side = torch.cuda.Stream(), torch.cuda.Stream()

    def steps():
        outs = []
        src.copy_(base)                                   # behind a copy
        outs += [o.clone() for o in call(h, s, st)]
        src.zero_()                                       # behind a memset
        outs += [o.clone() for o in call(h, s, st)]
        side.wait_stream(s)                               # behind a joined branch that writes the input
        with torch.cuda.stream(side):
            src.copy_(other)
        s.wait_stream(side)
        outs += [o.clone() for o in call(h, s, st)]
        return outs

    want = []
    for x in (base, torch.zeros_like(base), other):
        src.copy_(x)
        torch.cuda.synchronize()
        want += [o.clone() for o in call(h, torch.cuda.current_stream(), st)]
        torch.cuda.synchronize()
    if captured:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            got = steps()
    for _ in range(3):
        with torch.cuda.stream(s):
            if captured:
                g.replay()
            else:
                got = steps()
        s.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got, strict=True))
    assert h.sync_status(s) == 0
