"""Grouped calls without a plan, queued on one workspace without a synchronisation between them: every
call writes its own problems' TMA descriptors where the call before had those of other matrices, and
each product has to be formed from its own.  All sets have the same shapes and live as long as the
calls, so a stale descriptor would give a wrong value, not a bad address.  The entries are small
integers, so FP32 sums are exact and every value has one right answer."""
import pytest
import torch

from _gpu import hsmm, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

SHAPES = [(64, 64, 64), (300, 224, 136), (8, 256, 200), (513, 96, 1000)]


def _ints(rows, cols, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ld = (rows + 7) // 8 * 8
    return torch.randint(-3, 4, (cols, ld), device="cuda", generator=g).to(torch.bfloat16).t()[:rows]


def _problems(q, ta, tb):
    probs = []
    for i, (m, n, k) in enumerate(SHAPES):
        A, B = (_ints(*s, 100 * q + 2 * i + j) for j, s in
                enumerate([(m, k) if ta == "N" else (k, m), (k, n) if tb == "N" else (n, k)]))
        probs.append((A, B, torch.zeros(n, (m + 3) // 4 * 4, device="cuda").t()[:m], ta, tb))
    return probs


def _op(x, t):
    return x.double() if t == "N" else x.double().t()


@pytest.mark.parametrize("kernel", ["pair", "single"])
@pytest.mark.parametrize("ta,tb", [("N", "N"), ("T", "T")])
@pytest.mark.parametrize("captured", [False, True])
def test_one_workspace_for_many_problem_sets(captured, ta, tb, kernel, monkeypatch):
    monkeypatch.setenv("HSMM_GROUPED_KERNEL", kernel)
    h = hsmm()
    sets = [_problems(q, ta, tb) for q in range(4)]
    want = [[(_op(A, ta) @ _op(B, tb)).float() for A, B, _, ta, tb in p] for p in sets]
    ws = torch.empty(max(h.gemm_grouped_workspace_size(p) for p in sets), dtype=torch.uint8, device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())

    def queue():
        for r in range(3):
            for q in (0, 1, 2, 3, 1, 0, 3, 2):
                h.gemm_grouped(sets[q], alpha=float(r + 1), workspace=ws, stream=s)

    queue()                       # also sets the kernels' attributes before a capture
    s.synchronize()
    for _ in range(4):
        for p in sets:
            for prob in p:
                prob[2].fill_(float("nan"))
        s.wait_stream(torch.cuda.current_stream())
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                queue()
            with torch.cuda.stream(s):
                g.replay()
        else:
            queue()
        s.synchronize()
        assert h.sync_status(s) == 0
        for p, w in zip(sets, want):
            for prob, x in zip(p, w):
                assert torch.equal(prob[2], 3 * x), prob[2].shape
