"""Neighbour search where groups are listed as heavy (a block of warps each):
many candidates, many nodes, every slot count, and radii whose square underflows."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _search(pos, h, leaf, G, **cfg):
    import oracle
    import paper_1112_4539_gb300 as bh
    n = pos.shape[0]
    ctx = bh.Context(n, leaf_size=leaf, group_size=G, **cfg)
    count, rho = ctx.neighbors(torch.from_numpy(pos).cuda(), torch.from_numpy(h).cuda())
    again, rho2 = ctx.neighbors(torch.from_numpy(pos).cuda(), torch.from_numpy(h).cuda())
    assert ctx.status() == 0
    ctx.close()
    c_ref, r_ref = oracle.sph_density(pos, h)
    np.testing.assert_array_equal(count.cpu().numpy(), c_ref)
    np.testing.assert_allclose(rho.cpu().numpy(), r_ref, rtol=1e-5)  # FP32 sums of positive terms
    assert torch.equal(count, again) and torch.equal(rho, rho2)


@pytest.mark.parametrize("G", [1, 32, 64, 96, 128, 256])
def test_many_candidates(G):
    n = 6001
    pos = workloads.plummer(n, seed=3)
    h = np.full(n, 0.4, np.float32)
    h[::7] = 5.0
    _search(pos, h, 16, G)


@pytest.mark.parametrize("cfg", [dict(), dict(max_level=21), dict(curve=1)])
def test_analytic_radii(cfg):
    n = 20000  # the outskirts' radii reach over most of the tree
    pos = workloads.plummer(n, seed=4)
    _search(pos, workloads.plummer_search_radii(pos).astype(np.float32), 4, 32, **cfg)


def test_radius_whose_square_underflows():
    import paper_1112_4539_gb300 as bh
    pos = workloads.uniform_cube(500, seed=2)
    ctx = bh.Context(500, leaf_size=8, group_size=32)
    count, rho = ctx.neighbors(torch.from_numpy(pos).cuda(), 1e-30)
    assert ctx.status() == 0
    assert (count == 0).all() and (rho == float("inf")).all()  # m W(0), and 8 / (pi h^3) is beyond FP32
    ctx.close()
