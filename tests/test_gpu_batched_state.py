"""After a batched call the context's tree has a root per system: tree_moments and the walks refuse it until the
next tree_build."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("order", [1, 2])
def test_moments_refuse_a_batched_tree(order):
    import paper_1112_4539_gb300 as bh
    pos = np.concatenate([workloads.plummer(500, seed=1), workloads.plummer(300, seed=2)])
    x = torch.from_numpy(pos).cuda()
    out = torch.zeros_like(x)
    ctx = bh.Context(800, max_systems=2, leaf_size=8, group_size=64, order=order)
    ref = ctx.evaluate(x, 0.5, 0.01, walk="particle").cpu().numpy()
    assert bh.bh_batch_layout(ctx.h, np.array([0, 500, 800])) == 0
    assert bh.bh_force_batched(ctx.h, x, 0.5, 0.01, out) == 0
    assert bh.tree_moments(ctx.h, 0.5) == bh.BH_ERR_STATE
    assert bh.tree_force(ctx.h, 0.01, out) == bh.BH_ERR_STATE
    assert bh.tree_force_particles(ctx.h, 0.01, out) == bh.BH_ERR_STATE
    count, rho = torch.empty(800, dtype=torch.int32, device="cuda"), torch.empty(800, device="cuda")
    assert bh.tree_neighbors(ctx.h, 0.2, count, rho) == 0  # (needs no moments and finds each group's root)
    np.testing.assert_array_equal(ctx.evaluate(x, 0.5, 0.01, walk="particle").cpu().numpy(), ref)
    assert ctx.status() == 0
    ctx.close()
