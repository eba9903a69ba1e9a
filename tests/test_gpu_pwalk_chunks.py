"""The per-particle walk takes 32 particles per warp: chunk edges, masks and
oversized leaves against the oracle's walk of each particle."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 1e-5  # of max(|a|, 1e-3 median |a|, 0.1 sum of |terms|), on particles whose decisions have a margin of 1e-5


def _walk(pos, theta, eps, n_leaf, order, unsoftened=False, max_level=10, soft=None):
    import oracle
    import paper_1112_4539_gb300 as bh
    n = pos.shape[0]
    ctx = bh.Context(n, leaf_size=n_leaf, order=order, max_level=max_level)
    x = torch.from_numpy(pos).cuda()
    if soft is None:
        got = ctx.evaluate(x, theta, eps, walk="particle", unsoftened_cells=unsoftened)
        b = oracle.Built(pos, n_leaf, 32, theta, order, 0, max_level)
        ref = oracle.force_particles(b.spos, b.perm, b.tree, b.mom, eps, unsoftened_pc=unsoftened)
    else:
        got = ctx.evaluate_symmetrized(x, torch.from_numpy(soft).cuda(), theta, unsoftened_cells=unsoftened)
        ref, _ = oracle.tree_force_sym(pos, soft, theta, n_leaf=n_leaf, order=order, max_level=max_level,
                                       unsoftened_pc=unsoftened)
    assert ctx.status() == 0
    st = ctx.stats()
    ctx.close()
    got, out, ok = got.cpu().numpy().astype(np.float64), ref["out"], ref["margin"] >= 1e-5
    assert np.isfinite(got).all()
    if n == 1:
        assert (got == 0).all()
        return
    a = np.linalg.norm(out[:, :3], axis=1)
    den = np.maximum(np.maximum(a, 1e-3 * np.median(a)), 0.1 * ref["a_abs"])
    assert (np.linalg.norm(got[:, :3] - out[:, :3], axis=1) / den)[ok].max(initial=0) <= TOL
    assert (np.abs(got[:, 3] - out[:, 3]) / np.abs(out[:, 3]))[ok].max(initial=0) <= TOL
    if ok.all():
        assert st["n_pp"] == int(ref["n_pp"].sum()) and st["n_pc"] == int(ref["n_pc"].sum())


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 65, 97, 1000])
def test_chunk_edges(n, order):
    pos = workloads.plummer(n, seed=n)
    _walk(pos, 0.7, 0.01, 4, order)
    _walk(pos, 0.7, 0.01, 1, order, soft=workloads.softening_lengths(n, 0.01))


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("unsoftened", [False, True])
def test_no_softening_and_deep_trees(order, unsoftened):
    pos = workloads.clumpy(4001, seed=9)
    _walk(pos, 0.6, 0.0 if not unsoftened else 1e-3, 8, order, unsoftened)
    _walk(pos, 0.6, 1e-3, 2, order, unsoftened, max_level=21)
    _walk(pos, 0.6, 0.0, 8, order, unsoftened, soft=workloads.softening_lengths(4001, 1e-3))


def test_oversized_leaf():
    pos = workloads.uniform_cube(3000, seed=6)
    pos[500:2300, :3] = np.float32(0.30005) + np.float32(1e-5) * pos[500:2300, :3]
    _walk(pos, 0.5, 1e-3, 16, 2)
    _walk(pos, 0.5, 0.0, 16, 1, soft=workloads.softening_lengths(3000, 1e-3))
