"""Neighbour search with particles that have no finite place: nobody's neighbours, with a count of 0."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n,h", [(200, 0.3), (5001, 0.05), (5001, 2.0)])  # (few candidates, and a block per group)
def test_count_of_a_nonfinite_particle_is_zero(value, n, h):
    import oracle
    import paper_1112_4539_gb300 as bh
    pos = workloads.plummer(n, seed=7)
    bad = np.arange(3, n, 61)
    pos[bad, np.arange(len(bad)) % 3] = value
    pos[bad[0]:bad[0] + 40, :3] = value  # more than a warp of them
    good = np.isfinite(pos).all(1)
    for G in (1, 32, 96):
        ctx = bh.Context(n, leaf_size=8, group_size=G)
        count, rho = ctx.neighbors(torch.from_numpy(pos).cuda(), h)
        assert ctx.status() == bh.BH_ERR_NONFINITE
        ctx.close()
        c_ref, r_ref = oracle.sph_density(pos[good], np.full(good.sum(), h, np.float32))
        np.testing.assert_array_equal(count.cpu().numpy()[good], c_ref)
        np.testing.assert_allclose(rho.cpu().numpy()[good], r_ref, rtol=1e-5)
        assert (count.cpu().numpy()[~good] == 0).all() and (rho.cpu().numpy()[~good] == 0).all()
