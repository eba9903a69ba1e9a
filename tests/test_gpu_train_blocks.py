"""The gradient and the training step over their block shapes (32 or 64 samples
per block, one or several rows of partial sums) against PyTorch in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# FP32 sums of n products in runs of at most 64 and rows: the relative error of the
# gradient's 2-norm stays below (64 + 304 + 20) * 2^-24 = 2.3e-5 (worst case, no cancellation across samples)
TOL = 2.3e-5


def _data(n, seed):
    rng = np.random.Generator(np.random.Philox(key=seed))
    X = torch.from_numpy(rng.uniform(-1, 1, (n, 6)).astype(np.float32)).cuda()
    Y = torch.from_numpy(rng.uniform(-6, 0, n).astype(np.float32)).cuda()
    P = torch.from_numpy(rng.uniform(-0.4, 0.4, 1313).astype(np.float32)).cuda()
    return X, Y, P


def _loss64(P, X, Y):
    w1, b1, w2, b2, w3, b3 = torch.split(P, [192, 32, 1024, 32, 32, 1])
    h = torch.relu(X.double() @ w1.view(32, 6).T + b1)
    r = torch.relu(h @ w2.view(32, 32).T + b2) @ w3 + b3 - Y.double()
    return (torch.where(r < 0, 4.0, 1.0) * r * r).mean()


@pytest.mark.parametrize("n", [1, 5, 31, 32, 33, 63, 64, 65, 128, 1000, 4864, 4865, 20001])
def test_gradient(n):
    import paper_1112_4539_gb300 as bh
    X, Y, P = _data(n, n)
    grad = torch.full((bh.MLP_NPARAM,), float("nan"), device="cuda")
    loss = torch.full((1,), 0.5, device="cuda")
    work = torch.full((n * bh.MLP_ACT + 8,), 7.0, device="cuda")
    assert bh.bh_mlp_grad(P, X, Y, 4.0, work[: n * bh.MLP_ACT], grad, loss) == 0
    P64 = P.double().requires_grad_(True)
    want = _loss64(P64, X, Y)
    g, = torch.autograd.grad(want, P64)
    assert float((grad.double() - g).norm() / g.norm()) <= TOL
    assert abs(float(loss) - 0.5 - float(want.detach())) <= TOL * (0.5 + float(want.detach()))
    assert (work[n * bh.MLP_ACT:] == 7.0).all()


@pytest.mark.parametrize("n,batch", [(40, 1), (40, 32), (40, 33), (40, 64), (500, 65), (9000, 4864), (9000, 4865), (30000, 20000)])
def test_steps(n, batch):
    import paper_1112_4539_gb300 as bh
    steps = 3
    X, Y, P = _data(n, n + 1)
    order = torch.randperm(n, generator=torch.Generator().manual_seed(n)).to(torch.int32).cuda()
    p, m, v = P.clone(), torch.zeros_like(P), torch.zeros_like(P)
    size = batch * bh.MLP_ACT + bh.MLP_NPARAM
    work = torch.full((size + 8,), 7.0, device="cuda")
    loss = torch.zeros(steps, device="cuda")
    assert bh.bh_mlp_train(X, Y, order, p, m, v, work[:size], steps, batch, 1e-3, 4.0, loss, 0) == 0
    assert (work[size:] == 7.0).all()
    q = P.double().requires_grad_(True)
    for t in range(steps):
        at = order[(torch.arange(batch, device="cuda") + (t * batch) % n) % n].long()
        want = _loss64(q, X[at], Y[at])
        g, = torch.autograd.grad(want, q)
        assert abs(float(loss[t]) - float(want.detach())) <= 1e-4 * float(want.detach())
        if t == 0:
            m64, v64 = 0.1 * g, 0.001 * g * g
        else:
            m64, v64 = 0.9 * m64 + 0.1 * g, 0.999 * v64 + 0.001 * g * g
        with torch.no_grad():
            q -= 1e-3 * (m64 / (1 - 0.9 ** (t + 1))) / ((v64 / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
    # three steps of at most 1e-3 each; a gradient entry whose sign is rounding noise may differ by a whole step
    d = (p.double() - q).abs()
    assert float(d.max()) <= 6e-3 and float((d > 1e-5).float().mean()) <= 0.02
    assert float((m.double() - m64).norm() / m64.norm()) <= 1e-3
