"""The block-per-group walk (few groups) gives the bits and the counts of the
one-warp kernel, which a context with blocks_per_sm set runs at every size."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _both(pos, theta, eps, **cfg):
    import paper_1112_4539_gb300 as bh
    x = torch.from_numpy(pos).cuda()
    outs = []
    for grid in (0, 2):
        ctx = bh.Context(max(1, pos.shape[0]), blocks_per_sm=grid, **cfg)
        out = ctx.evaluate(x, theta, eps)
        assert ctx.status() == 0
        st = ctx.stats()
        outs.append((out, st["n_pp"], st["n_pc"], st["n_groups"]))
        ctx.close()
    assert outs[0][1:] == outs[1][1:]
    assert torch.equal(outs[0][0], outs[1][0])


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("G", [1, 32, 33, 64, 72, 96, 100, 128])
def test_slots_and_split_slots(G, order):
    _both(workloads.clumpy(7001, seed=5), 0.6, 1e-3, group_size=G, order=order, leaf_size=8)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 65, 130])
def test_tiny_sets(n):
    _both(workloads.plummer(n, seed=3), 0.5, 0.0, order=2, group_size=96, leaf_size=16)


@pytest.mark.parametrize("n,G", [(30011, 96), (60007, 96), (60007, 64), (40001, 32)])
@pytest.mark.parametrize("cfg", [dict(order=2, leaf_size=16), dict(order=1, leaf_size=64, curve=1),
                                 dict(order=2, leaf_size=8, max_level=21)])
def test_both_block_sizes(n, G, cfg):
    _both(workloads.plummer(n, seed=4), 0.55, 0.01, group_size=G, **cfg)


def test_oversized_leaf():
    # a knot of 5000 particles inside one level-10 cell: one leaf longer than the ring of pending sources
    pos = workloads.uniform_cube(9000, seed=6)
    pos[2000:7000, :3] = np.float32(0.30005) + np.float32(1e-5) * pos[2000:7000, :3]
    _both(pos, 0.5, 1e-3, order=2, group_size=96, leaf_size=16)
    _both(pos, 0.5, 1e-3, order=1, group_size=64, leaf_size=8)
