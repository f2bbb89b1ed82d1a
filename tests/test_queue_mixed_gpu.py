"""Kernels of different families queued behind one another, eager and in a CUDA graph: each call reads
what the one before wrote (matrix-vector and n^2 results as operands, products as matrices) and later
calls overwrite what earlier ones read.  The same calls with a synchronisation after each are the
reference, bit for bit."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


class Chain:
    def __init__(self, h, n):
        g = torch.Generator(device="cuda").manual_seed(n)

        def rand(rows, cols, dtype):
            return (torch.rand(cols, rows, device="cuda", dtype=torch.float64, generator=g) - 0.5).to(dtype).t()

        self.h, self.n = h, n
        self.a, self.b = rand(n, n, torch.bfloat16), rand(n, n, torch.bfloat16)
        self.c, self.f = rand(n, n, torch.float32), rand(n, n, torch.float32)
        self.t = rand(n, n, torch.bfloat16)
        self.x, self.y = rand(n, 1, torch.float32)[:, 0].contiguous(), torch.zeros(n, device="cuda")
        self.out = torch.zeros(n // 4, 4, device="cuda")
        self.d, self.e, self.m = (rand(n, n, torch.float64) for _ in range(3))
        need = h.workspace_size(h.hsmm.make_config(h.R_64F, h.R_64F, h.R_64F, h.COMPUTE_64F_OZAKI), "N", "N", n, n, n)
        self.ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        self.gws = torch.empty(max(16, h.hsmm.gemv_workspace_size(h.R_32F, "N", n, n)), dtype=torch.uint8, device="cuda")
        half = n // 16 * 8
        self.plan = h.GroupedPlan([(self.a, self.t[:, :half], self.f[:, :half], "N", "N"),
                                   (self.a, self.t[:, half:], self.f[:, half:], "T", "N")], h.R_16BF, h.R_32F)
        self.start = [t.clone() for t in self.state()]

    def state(self):
        return [self.c, self.f, self.t, self.x, self.y, self.out, self.d, self.e]

    def reset(self):
        for t, s in zip(self.state(), self.start):
            t.copy_(s)

    def run(self, stream, sync):
        h, tf32, oz = self.h, self.h.COMPUTE_32F_FAST_TF32, self.h.COMPUTE_64F_OZAKI
        bodies = self.y.view(-1, 4)
        for _ in range(3):
            for call in (lambda: h.gemm(self.a, self.b, self.c, stream=stream),
                         lambda: h.gemv(self.c, self.x, self.y, "T", workspace=self.gws, stream=stream),
                         lambda: h.nbody(bodies, bodies, 1.0, self.out, stream=stream),
                         lambda: h.gemv(self.c, self.out.view(-1), self.x, "N", 1e-3, 0.5, workspace=self.gws, stream=stream),
                         lambda: h.gemm(self.c, self.c, self.f, "T", "N", 1.0 / self.n, compute=tf32, stream=stream),
                         lambda: h.gemv(self.f, self.x, self.y, "N", 1.0, 1.0, workspace=self.gws, stream=stream),
                         lambda: self.plan.launch(stream=stream),
                         lambda: h.gemv(self.f, self.y, self.x, "T", 1e-3, workspace=self.gws, stream=stream),
                         lambda: h.gemm(self.a, self.a, self.t, "N", "T", 1.0 / self.n, stream=stream),
                         lambda: h.gemm(self.d, self.m, self.e, "N", "T", 1.0, 0.5, compute=oz, workspace=self.ws, stream=stream),
                         lambda: h.gemm(self.e, self.m, self.d, "T", "N", 1.0 / self.n, stream=stream),
                         lambda: h.gemm(self.m, self.d, self.e, "T", "N", 1.0, compute=oz, workspace=self.ws, stream=stream)):
                call()
                sync()


@pytest.mark.parametrize("n", [72, 520])
def test_mixed_calls_wait_for_each_other(n):
    h = hsmm()
    chain = Chain(h, n)
    s = torch.cuda.Stream()
    chain.run(s, s.synchronize)
    want = [t.clone() for t in chain.state()]
    assert all(torch.isfinite(t.float()).all() for t in want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        chain.run(s, lambda: None)
    for rep in range(4):
        chain.reset()
        torch.cuda.synchronize()
        if rep % 2:
            with torch.cuda.stream(s):
                graph.replay()
        else:
            chain.run(s, lambda: None)
        s.synchronize()
        assert h.sync_status(s) == 0
        for i, (w, t) in enumerate(zip(want, chain.state())):
            assert torch.equal(w, t), i
