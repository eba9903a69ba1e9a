"""Thousands of systems of a few particles per batched call: forces against direct 64-bit sums, and the time."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _systems(sizes, seed):
    off = np.concatenate([[0], np.cumsum(sizes)])
    pos = workloads.plummer(int(off[-1]), seed=seed)
    pos[:, 3] = np.repeat(1.0 / sizes, sizes)
    return off, torch.from_numpy(pos).cuda()


def _context(off, **cfg):
    import paper_1112_4539_gb300 as bh
    ctx = bh.Context(int(off[-1]), max_systems=len(off) - 1, block_threads=64, **cfg)
    assert bh.bh_batch_layout(ctx.h, off) == 0
    return bh, ctx


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("deep", [False, True])
def test_forces_of_tiny_systems(order, deep):
    """Up to 40 particles in leaves of up to 64: every term is a particle, so a plain FP32 sum of 40 terms of about 6
    roundings."""
    sizes = np.random.default_rng(1).integers(1, 41, 3000)
    off, x = _systems(sizes, 3)
    bh, ctx = _context(off, leaf_size=64, group_size=64, order=order, max_level=21 if deep else 10)
    out = torch.empty_like(x)
    assert bh.bh_force_batched(ctx.h, x, 0.5, 0.05, out) == 0 and ctx.status() == 0
    perm = ctx.export("perm")
    ctx.close()
    owner = np.repeat(np.arange(len(sizes)), sizes)
    np.testing.assert_array_equal(owner[perm], owner)  # sorted within each system
    p, s = x.double(), torch.from_numpy(owner).cuda()
    for i in torch.arange(x.shape[0], device="cuda").split(4000):
        same = (s[None, :] == s[i, None]) & (torch.arange(x.shape[0], device="cuda")[None, :] != i[:, None])
        d = p[None, :, :3] - p[i, None, :3]
        w = torch.where(same, p[None, :, 3], 0.0) / (d.square().sum(2) + 0.05 ** 2).sqrt()
        a = (w / (d.square().sum(2) + 0.05 ** 2))[:, :, None] * d
        want = torch.cat([a.sum(1), -w.sum(1)[:, None]], 1)
        mag = torch.cat([a.abs().sum(1), w.sum(1)[:, None]], 1)
        assert ((out[i].double() - want).abs() <= 46 * 2.0 ** -24 * mag).all()


def _ms(sizes, **cfg):
    off, x = _systems(sizes, 5)
    bh, ctx = _context(off, **cfg)
    out, ms = torch.empty_like(x), []
    for k in range(12):
        start, end = torch.cuda.Event(True), torch.cuda.Event(True)
        start.record()
        assert bh.bh_force_batched(ctx.h, x, 0.5, 0.01, out) == 0
        end.record()
        end.synchronize()
        ms.append(start.elapsed_time(end))
    ctx.close()
    return min(ms)


def test_time_of_the_sort():
    """20000 systems of 5, sorted with work for their own particles only 0.74 ms, with a full tile's 1.6 ms."""
    assert _ms(np.full(20000, 5), leaf_size=8, group_size=64, order=1) < 1.1
