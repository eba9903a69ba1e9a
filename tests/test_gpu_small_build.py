"""The one-block build of small sets against the chain of launches (which a set
with one particle more takes) and the oracle: edges of the item counts, leaf and
group sizes, key widths, orders."""
import ctypes

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _export(bh, ctx, what, dtype, count):
    out = np.zeros(count, dtype=dtype)
    nb = ctypes.c_int64()
    assert bh.lib().bh_export(ctx.h, bh.EXPORT[what], out.ctypes.data_as(ctypes.c_void_p), out.nbytes,
                              ctypes.byref(nb), None) == 0
    return out[: nb.value // out.itemsize]


def _check(pos, n_leaf, G, curve=0, max_level=10):
    import oracle
    import paper_1112_4539_gb300 as bh
    n = pos.shape[0]
    ctx = bh.Context(n, leaf_size=n_leaf, group_size=G, curve=curve, max_level=max_level)
    ctx.build(torch.from_numpy(pos).cuda())
    assert ctx.status() == 0
    st = ctx.stats()
    b = oracle.Built(pos, n_leaf, G, 0.5, 1, curve, max_level)
    t = b.tree
    nn, ng = st["n_nodes"], st["n_groups"]
    assert nn == len(t.first) and ng == len(b.g_first)
    kt = np.uint64 if max_level > 10 else np.uint32
    np.testing.assert_array_equal(_export(bh, ctx, "keys", kt, n), b.skeys)
    np.testing.assert_array_equal(_export(bh, ctx, "perm", np.uint32, n), b.perm)
    np.testing.assert_array_equal(_export(bh, ctx, "spos", np.float32, 4 * n).reshape(-1, 4), b.spos)
    np.testing.assert_array_equal(_export(bh, ctx, "node_first", np.int32, nn), t.first)
    np.testing.assert_array_equal(_export(bh, ctx, "node_count", np.int32, nn), t.count)
    np.testing.assert_array_equal(_export(bh, ctx, "node_child", np.int32, nn), t.child_first)
    np.testing.assert_array_equal(_export(bh, ctx, "node_nchild", np.int32, nn), t.nchild)
    np.testing.assert_array_equal(_export(bh, ctx, "node_level", np.int32, nn), t.level)
    np.testing.assert_array_equal(_export(bh, ctx, "group_first", np.int32, ng), b.g_first)
    np.testing.assert_array_equal(_export(bh, ctx, "group_count", np.int32, ng), b.g_count)
    leaf = t.child_first < 0
    assert st["n_leaves"] == int(leaf.sum()) and st["max_leaf_count"] == int(t.count[leaf].max())
    ctx.close()


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 4095, 4096, 4097, 8191, 8192, 8193])
def test_sizes(n):
    _check(workloads.plummer(n, seed=n), 8, 64)


@pytest.mark.parametrize("n_leaf,G", [(1, 1), (1, 256), (2, 32), (16, 7), (64, 96), (64, 256)])
@pytest.mark.parametrize("curve,max_level,n", [(0, 10, 5003), (1, 10, 5003), (0, 21, 3001), (1, 21, 4096)])
def test_leaves_groups_and_keys(n_leaf, G, curve, max_level, n):
    _check(workloads.clumpy(n, seed=7), n_leaf, G, curve, max_level)


@pytest.mark.parametrize("max_level", [10, 21])
def test_equal_keys_keep_their_order(max_level):
    pos = workloads.uniform_cube(4000, seed=3)
    pos[100:3900, :3] = pos[50, :3]  # one cell of 3801 particles
    _check(pos, 8, 64, 0, max_level)
    _check(np.tile(pos[:1], (777, 1)), 8, 64, 0, max_level)


def test_nonfinite_input_is_reported():
    import paper_1112_4539_gb300 as bh
    pos = workloads.plummer(3000, seed=1)
    pos[1234, 2] = np.nan
    ctx = bh.Context(3000)
    ctx.build(torch.from_numpy(pos).cuda())
    assert ctx.status() == bh.BH_ERR_NONFINITE
    ctx.build(torch.from_numpy(workloads.plummer(3000, seed=1)).cuda())
    assert ctx.status() == 0
    ctx.close()
