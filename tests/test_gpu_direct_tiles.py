"""Direct sums at the edges of the source tiles and splits against long-double
sums on the host: both precisions, self terms anywhere, no softening."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _reference(src, tgt, idx, e2):
    """(sums, sums of magnitudes) in long double; e2[i, j]: squared softening of a pair."""
    s, t = src.astype(np.longdouble), tgt.astype(np.longdouble)
    d = s[None, :, :3] - t[:, None, :3]
    r2 = (d * d).sum(2) + e2
    m = np.broadcast_to(s[:, 3], r2.shape).copy()
    for k, j in enumerate(idx):
        if j >= 0:
            m[k, j], r2[k, j] = 0, 1
    w = m / np.sqrt(r2)
    a = (w / r2)[:, :, None] * d
    out = np.concatenate([a.sum(1), -w.sum(1)[:, None]], 1)
    mag = np.concatenate([np.abs(a).sum(1), w.sum(1)[:, None]], 1)
    return out, mag


# of the sum of magnitudes: plain sums of 256 (FP64) or 2 x 128 (FP32) terms of 4 roundings each, compensated across tiles
TOL = {64: (256 + 8) * 2.0 ** -53, 32: (128 + 8) * 2.0 ** -24}


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 513, 1025, 5000])
@pytest.mark.parametrize("kind", ["softened", "bare", "symmetrized"])
def test_tiles(n, precision, kind):
    import paper_1112_4539_gb300 as bh
    pos = workloads.plummer(n, seed=n)
    nt = min(n + 3, 700)
    tgt = np.concatenate([pos, workloads.plummer(3, seed=99)])[-nt:]
    idx = np.concatenate([np.arange(n), [-1, -1, -1]])[-nt:]
    eps = 0.0 if kind == "bare" else 0.01
    es, et = workloads.softening_lengths(n, 0.01), workloads.softening_lengths(nt, 0.01, seed=5)
    e2 = (0.5 * (es.astype(np.longdouble) ** 2)[None, :] + 0.5 * (et.astype(np.longdouble) ** 2)[:, None]
          if kind == "symmetrized" else np.longdouble(eps) ** 2)
    want, mag = _reference(pos, tgt, idx, e2)
    d = [torch.from_numpy(a).cuda() for a in (pos, tgt, idx.astype(np.int64), es, et)]
    out = torch.empty((nt, 4), device="cuda", dtype=torch.float64 if precision == 64 else torch.float32)
    rc = (bh.direct_force_sym(d[0], d[3], d[1], d[4], d[2], out, precision) if kind == "symmetrized"
          else bh.direct_force(d[0], d[1], d[2], eps, out, precision))
    assert rc == 0
    got = out.cpu().numpy().astype(np.longdouble)
    assert (np.abs(got - want) <= TOL[precision] * mag + np.longdouble(1e-300)).all()



@pytest.mark.parametrize("scale", [-120, -101, -37, 0, 23, 60])
def test_inverse_root(scale):
    """FP64, one source and one target per sum: every exponent and mantissa pattern of r^2, nothing to average over.
    With u = 2^-53, r^2 is off by at most 5 u (differences 2 u, three fused adds), its inverse root by 2.5 u + 1.5 u,
    the potential by 1 u more, the force by 3 x 4 u and 5 roundings."""
    import paper_1112_4539_gb300 as bh
    rng = np.random.Generator(np.random.Philox(key=scale + 500))
    n = 500
    src, tgt = np.zeros((1, 4), np.float32), np.zeros((n, 4), np.float32)
    src[0, 3] = 1.0
    tgt[:, :3] = np.ldexp(rng.uniform(-2, 2, (n, 3)), scale + rng.integers(-4, 5, (n, 1)))
    tgt[:4, :3] = np.ldexp(np.array([[1, 0, 0], [0, 2, 0], [1, 1, 0], [np.nextafter(np.float32(2), 0), 0, 0]]), scale)
    want, mag = _reference(src, tgt, np.full(n, -1), np.longdouble(0))
    d = [torch.from_numpy(a).cuda() for a in (src, tgt)]
    out = torch.empty((n, 4), device="cuda", dtype=torch.float64)
    assert bh.direct_force(d[0], d[1], torch.full((n,), -1, dtype=torch.int64, device="cuda"), 0.0, out, 64) == 0
    err = np.abs(out.cpu().numpy().astype(np.longdouble) - want) * 2.0 ** 53
    assert (err[:, :3] <= 18 * mag[:, :3]).all() and (err[:, 3] <= 6 * mag[:, 3]).all()


@pytest.mark.parametrize("n,nt", [(257, 77824), (257, 77825), (1025, 38912), (1025, 38656), (9000, 33)])
@pytest.mark.parametrize("kind", ["softened", "symmetrized"])
def test_wide(n, nt, kind):
    """FP64, 256 targets per block (full waves of them) and 32 with several tiles of sources."""
    import paper_1112_4539_gb300 as bh
    pos = workloads.plummer(n, seed=n)
    tgt = np.concatenate([pos, workloads.plummer(nt, seed=98)])[:nt]
    idx = np.where(np.arange(nt) < n, np.arange(nt), -1)
    at = np.unique(np.concatenate([np.arange(16), np.linspace(0, nt - 1, 200).astype(int)]))
    es, et = workloads.softening_lengths(n, 0.01), workloads.softening_lengths(nt, 0.01, seed=5)
    e2 = (0.5 * (es.astype(np.longdouble) ** 2)[None, :] + 0.5 * (et[at].astype(np.longdouble) ** 2)[:, None]
          if kind == "symmetrized" else np.longdouble(0.01) ** 2)
    want, mag = _reference(pos, tgt[at], idx[at], e2)
    d = [torch.from_numpy(a).cuda() for a in (pos, tgt, idx.astype(np.int64), es, et)]
    out = torch.empty((nt, 4), device="cuda", dtype=torch.float64)
    rc = (bh.direct_force_sym(d[0], d[3], d[1], d[4], d[2], out, 64) if kind == "symmetrized"
          else bh.direct_force(d[0], d[1], d[2], 0.01, out, 64))
    assert rc == 0
    assert (np.abs(out[torch.from_numpy(at).cuda()].cpu().numpy().astype(np.longdouble) - want) <= TOL[64] * mag).all()


@pytest.mark.parametrize("eps", [2e-162, 1e-160, 3.3e-157, 1e-155, 1.49e-154, 1.5e-154])
@pytest.mark.parametrize("nt", [1, 600])
def test_denormal_softening(eps, nt):
    """FP64, a source on the target: eps^2 is a denormal (a normal number from 1.4917e-154 on), its root within
    2 units of 2^-53 and the product with the mass 1 more."""
    import paper_1112_4539_gb300 as bh
    src = torch.tensor([[0.5, -1.0, 2.0, 3.0]], device="cuda")
    tgt = src.repeat(nt, 1).contiguous()
    out = torch.empty((nt, 4), device="cuda", dtype=torch.float64)
    assert bh.direct_force(src, tgt, None, eps, out, 64) == 0
    want = -3.0 / np.sqrt(np.longdouble(np.float64(eps) * np.float64(eps)))
    assert (np.abs(out[:, 3].cpu().numpy().astype(np.longdouble) / want - 1) <= 4 * 2.0 ** -53).all()


@pytest.mark.parametrize("n,nt", [(257, 1), (600, 33), (1000, 9000), (1024, 256), (1024, 40000)])
@pytest.mark.parametrize("kind", ["softened", "symmetrized"])
def test_few_sources_repeat(n, nt, kind):
    """FP64, up to 1024 sources (two to four partial sums per target): the same bits on every run."""
    import paper_1112_4539_gb300 as bh
    src, tgt = torch.from_numpy(workloads.plummer(n, seed=n)).cuda(), torch.from_numpy(workloads.plummer(nt, seed=98)).cuda()
    es, et = (torch.from_numpy(workloads.softening_lengths(k, 0.01)).cuda() for k in (n, nt))
    busy, out = torch.empty(1 << 22, device="cuda"), torch.empty((60, nt, 4), device="cuda", dtype=torch.float64)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for k in range(60):
        if k % 2:
            with torch.cuda.stream(side):  # (the blocks end in another order beside other work)
                busy.mul_(1.0)
        out[k].fill_(float(k))
        rc = (bh.direct_force_sym(src, es, tgt, et, None, out[k], 64) if kind == "symmetrized"
              else bh.direct_force(src, tgt, None, 0.01, out[k], 64))
        assert rc == 0
    torch.cuda.synchronize()
    assert (out == out[0]).all()
