"""Moments of small sets (one launch for all levels) are those of a larger
set's launches: a system alone against the same system among others."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cfg", [dict(order=1, leaf_size=8), dict(order=2, leaf_size=16), dict(order=2, leaf_size=1),
                                 dict(order=2, leaf_size=64, fp64_node_threshold=100), dict(order=2, leaf_size=8, max_level=21),
                                 dict(order=1, leaf_size=8, fp64_node_threshold=1, curve=1)])
def test_same_forces_alone_and_among_others(cfg):
    import paper_1112_4539_gb300 as bh
    sizes = [1, 33, 700, 4097, 8192, 9000]
    parts = [workloads.clumpy(n, seed=k) if k % 2 else workloads.plummer(n, seed=k) for k, n in enumerate(sizes)]
    parts[3][100:200, :3] = parts[3][100, :3]  # a leaf of 100 particles
    offs = np.concatenate([[0], np.cumsum(sizes)])
    x = torch.from_numpy(np.concatenate(parts)).cuda()
    ctx = bh.Context(x.shape[0], max_systems=len(sizes), group_size=64, **cfg)
    assert bh.bh_batch_layout(ctx.h, offs) == 0
    out = torch.empty_like(x)
    assert bh.bh_force_batched(ctx.h, x, 0.6, 0.01, out) == 0 and ctx.status() == 0
    ctx.close()
    one = bh.Context(max(sizes), group_size=64, **cfg)
    for a, b in zip(offs[:-1], offs[1:]):
        alone = one.evaluate(x[a:b].contiguous(), 0.6, 0.01)
        assert one.status() == 0 and torch.equal(alone, out[a:b])
    one.close()
