"""Kernels that start while their predecessor runs, behind what is no kernel of the library: a wait for an event of
another stream, a copy, a memset, eager and captured in a graph.  The inputs arrive late, after a pause on the GPU."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PAUSE = 400000  # clocks, about 0.2 ms


def _calls(n):
    """name -> (call on (positions, other input, output), output shape, dtype)"""
    import paper_1112_4539_gb300 as bh
    ctx = bh.Context(n, max_systems=4, leaf_size=8, group_size=64, order=2, block_threads=64)
    assert bh.bh_batch_layout(ctx.h, np.array([0, n // 3, n // 2, n])) == 0

    def neighbours(x, h, out):
        ctx.build(x)
        assert bh.tree_neighbors(ctx.h, h, None, out) == 0

    def drift(x, v, out):
        out.copy_(x)
        ctx.kick_drift(out, v.repeat(4).view(4, n).t().contiguous(), x, 0.1, 0.2)

    return ctx, {
        "group": (lambda x, h, out: ctx.evaluate(x, 0.6, 0.01, out), (n, 4)),
        "particle": (lambda x, h, out: ctx.evaluate(x, 0.6, 0.01, out, walk="particle"), (n, 4)),
        "symmetrized": (lambda x, h, out: ctx.evaluate_symmetrized(x, h, 0.6, out), (n, 4)),
        "neighbours": (neighbours, (n,)),
        "drift": (drift, (n, 4)),
        "batched": (lambda x, h, out: bh.bh_force_batched(ctx.h, x, 0.6, 0.01, out), (n, 4)),
    }


@pytest.mark.parametrize("n", [3000, 20000])  # a build in one launch, and a chain of launches
@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("before", ["event", "copy", "host copy", "memset"])
def test_late_inputs(n, captured, before):
    pos = torch.from_numpy(workloads.plummer(n, seed=1)).cuda()
    old = torch.from_numpy(workloads.plummer(n, seed=2)).cuda()
    h = torch.full((n,), 0.2, device="cuda")
    pinned = pos.cpu().pin_memory()
    ctx, calls = _calls(n)
    side = torch.cuda.Stream()
    for name, (call, shape) in calls.items():
        want = torch.empty(shape, device="cuda")
        call(pos, h, want)
        torch.cuda.synchronize()
        x, out = torch.empty_like(pos), torch.empty(shape, device="cuda")

        def late():
            if before == "event":
                side.wait_stream(torch.cuda.current_stream())
                with torch.cuda.stream(side):
                    torch.cuda._sleep(PAUSE)
                    x.copy_(pos)
                torch.cuda.current_stream().wait_stream(side)
            else:
                torch.cuda._sleep(PAUSE)
                x.copy_(pinned if before == "host copy" else pos, non_blocking=True)
                if before == "memset":
                    out.zero_()
            call(x, h, out)

        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                late()
        for _ in range(3):
            x.copy_(old)
            out.fill_(-1.0)
            torch.cuda.synchronize()
            graph.replay() if captured else late()
            torch.cuda.synchronize()
            assert torch.equal(out, want), name
    assert ctx.status() == 0
    ctx.close()
