"""The calls a user of this library makes, as cases with sizes, inputs and the
work that each one needs.

The library evaluates forces on particle sets held on the GPU.  Its users
call it once per orbit step (from a few thousand particles to tens of
millions), for many small systems at once, for particles with their own
softening, for neighbour densities, with the learned opening criterion (and
to train that criterion), and for direct sums, the judge of all of these.
Every case goes through the Python binding, as such a program does.
"""
import math

import numpy as np
import torch

import paper_1112_4539_gb300 as bh
from paper_1112_4539_gb300 import learned
from paper_1112_4539_gb300.leapfrog import Leapfrog

EPS = {"plummer": 0.01, "clumpy": 1e-3, "uniform": 0.01, "sphere": 0.01}
# learned criterion: threshold that gives p99 = 1e-3 on the set, as the benchmark calibrates it
TAU = {"plummer": 1.746e-4, "clumpy": 3.6e-5}
WEIGHTS = "paper_1112_4539_gb300/weights/mac_G96_l16_o2.npz"


def _evaluate(name, kind, shape, n, **kw):
    c = dict(name=name, kind=kind, shape=shape, n=n, order=2, leaf=16, group=96, theta=0.525, hilbert=False,
             max_level=10)
    c.update(kw)
    return c


def listed():
    return [
        # a small star cluster, the library's default configuration: one call is mostly launches
        _evaluate("eval_4k", "evaluate", "plummer", 4096, order=1, leaf=8, group=64, theta=0.5),
        # a galaxy model of ordinary size whose count is a multiple of nothing
        _evaluate("eval_100k", "evaluate", "clumpy", 100003),
        # the benchmark's single Plummer sphere
        _evaluate("eval_1m", "evaluate", "plummer", 1 << 20, theta=0.6),
        # one leapfrog step of the headline workload
        _evaluate("orbit_16m", "orbit", "clumpy", 1 << 24),
        # the paper's monopole tree on a dense core: 63-bit keys, Peano-Hilbert order
        _evaluate("deep_2m", "evaluate", "plummer", 2000003, order=1, leaf=8, group=64, theta=0.6, hilbert=True,
                  max_level=21),
        # the paper's own walk, a thread of control per particle (tighter criterion, fewer terms)
        _evaluate("particle_1m", "particle", "plummer", 1 << 20, theta=0.554),
        # particles of mixed mass resolution, each with its softening length
        _evaluate("symmetrized_262k", "symmetrized", "clumpy", 262147, theta=0.55),
        # neighbour counts and densities of a gas sphere, about 64 neighbours each
        dict(name="neighbors_1m", kind="neighbors", shape="plummer", n=1 << 20, leaf=16, group=32, ngb=64,
             each=True),
        # 512 clusters of 1k to 65k stars per call, replayed from a captured graph
        dict(name="batched_512", kind="batched", systems=512, nmin=1024, nmax=65536, order=1, leaf=8, group=96,
             theta=0.5, sizes=3),
        # the learned opening criterion with the shipped weights
        _evaluate("learned_4m", "learned", "clumpy", 1 << 22, theta=1.2),
        # the error judge: FP64 direct sums of sampled targets
        dict(name="judge_1m", kind="direct", precision=64, shape="plummer", n=1 << 20, targets=4096, each=False),
        # fitting the learned criterion: Adam steps on mini-batches
        dict(name="train_8k", kind="train", samples=1 << 20, batch=8192, steps=16),
    ]


def _size(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(lo, hi)))


def draw(rng):
    kind = rng.choice(["evaluate"] * 5 + ["orbit"] * 2 + ["particle"] * 2 + ["symmetrized", "neighbors", "neighbors",
                                                                            "batched", "learned", "direct", "train"])
    tree = dict(kind=kind, order=rng.choice([1, 2, 2]), leaf=rng.choice([8, 16]), group=rng.choice([32, 64, 96, 128]),
                theta=round(rng.uniform(0.5, 0.8), 3), hilbert=rng.random() < 0.25,
                max_level=21 if rng.random() < 0.25 else 10, shape=rng.choice(["plummer", "clumpy", "uniform", "sphere"]))
    if kind == "evaluate":
        return dict(tree, n=_size(rng, 10, 22))
    if kind == "orbit":
        return dict(tree, shape=rng.choice(["plummer", "clumpy"]), order=2, leaf=16, group=96, n=_size(rng, 12, 23))
    if kind == "particle":
        return dict(tree, n=_size(rng, 10, 20))
    if kind == "symmetrized":
        return dict(tree, n=_size(rng, 10, 19))
    if kind == "neighbors":
        return dict(kind=kind, shape=rng.choice(["plummer", "uniform"]), n=_size(rng, 11, 21), leaf=rng.choice([8, 16]),
                    group=rng.choice([32, 64]), ngb=rng.choice([32, 48, 64, 100]), each=rng.random() < 0.75)
    if kind == "batched":
        return dict(kind=kind, systems=_size(rng, 3, 9), nmin=rng.choice([256, 1024]), nmax=_size(rng, 12, 16),
                    order=rng.choice([1, 2]), leaf=rng.choice([8, 16]), group=rng.choice([64, 96]),
                    theta=round(rng.uniform(0.5, 0.7), 3), sizes=rng.randrange(1, 1000))
    if kind == "learned":
        return dict(tree, shape=rng.choice(["plummer", "clumpy"]), order=2, leaf=16, group=96, theta=1.2, hilbert=False,
                    max_level=10, n=_size(rng, 15, 22))
    if kind == "direct":
        return dict(kind=kind, precision=rng.choice([32, 32, 64]), shape=rng.choice(["plummer", "clumpy"]),
                    n=_size(rng, 10, 18), targets=_size(rng, 8, 14), each=rng.random() < 0.3)
    return dict(kind=kind, samples=_size(rng, 15, 21), batch=_size(rng, 9, 14), steps=rng.choice([8, 16, 32]))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _directions(g, n):
    z = 2.0 * _uniform(g, n) - 1.0
    ph = 2.0 * math.pi * _uniform(g, n)
    s = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    return torch.stack([s * torch.cos(ph), s * torch.sin(ph), z], dim=1)


def _particles(shape, n, seed):
    """(n, 4) float32 on the GPU: the distributions of the repository's workloads, equal masses, total mass 1."""
    g = _gen(seed)
    out = torch.empty((n, 4), device="cuda")
    out[:, 3] = 1.0 / n
    if shape == "plummer":  # unit Plummer sphere, truncated at r = 20
        x = _uniform(g, n).clamp(min=1e-12) * (20.0 ** 3 / (1.0 + 20.0 ** 2) ** 1.5)
        out[:, :3] = _directions(g, n) / torch.sqrt(x ** (-2.0 / 3.0) - 1.0)[:, None]
    elif shape == "uniform":
        out[:, :3] = _uniform(g, n, 3)
    elif shape == "sphere":
        out[:, :3] = _directions(g, n) * _uniform(g, n)[:, None] ** (1.0 / 3.0)
    else:  # 64 Hernquist clumps (80%) over a uniform background, in no order
        w = 10.0 ** _uniform(g, 64)
        centres = _uniform(g, 64, 3)
        clump = torch.searchsorted(torch.cumsum(w / w.sum(), 0), _uniform(g, n)).clamp(max=63)
        s = torch.sqrt(_uniform(g, n) * (20.0 / 21.0) ** 2)
        x = centres[clump] + _directions(g, n) * (0.05 * s / (1.0 - s))[:, None]
        out[:, :3] = torch.where((_uniform(g, n) < 0.2)[:, None], _uniform(g, n, 3), x)
    return out


def _softening(n, eps, seed):
    """Log-uniform lengths in [eps / 4, 4 eps]."""
    return (eps * torch.exp((2.0 * _uniform(_gen(seed + 1), n) - 1.0) * math.log(4.0))).float()


def _radii(case, pos):
    """Search radii that enclose about `ngb` neighbours, from the analytic density."""
    n, ngb = case["n"], case["ngb"]
    if case["shape"] == "plummer":
        r2 = pos[:, :3].double().square().sum(1)
        rho = 3.0 / (4.0 * math.pi) * (1.0 + r2) ** -2.5
        h = ((3.0 * ngb) / (4.0 * math.pi * rho * n)) ** (1.0 / 3.0)
    else:
        h = torch.full((n,), ((3.0 * ngb) / (4.0 * math.pi * n)) ** (1.0 / 3.0), device=pos.device, dtype=torch.float64)
    # one radius for all: that of the half-mass radius' density
    return h.float().contiguous() if case["each"] else float(h.median())


def _sizes(case):
    r = np.random.default_rng(case["sizes"])
    lo, hi = math.log2(case["nmin"]), math.log2(case["nmax"])
    return np.rint(2.0 ** r.uniform(lo, hi, case["systems"])).astype(np.int64)


def _features(case, seed):
    """Samples like the labelled pairs that the criterion is fitted to: six features and the log10 of an error."""
    g, n = _gen(seed), case["samples"]
    u = _uniform(g, n, 6)
    X = torch.stack([0.05 + 0.9 * u[:, 0], -6.0 * u[:, 1], 0.5 * u[:, 2] ** 2, 0.6 * u[:, 3], u[:, 4], u[:, 5]], 1)
    Y = 3.0 * torch.log10(X[:, 0]) + 0.6 * X[:, 1] + 0.5 * X[:, 2] + 0.3 * torch.randn(n, generator=g, device="cuda",
                                                                                 dtype=torch.float64)
    order = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    return X.float().contiguous(), Y.float().contiguous(), order


def _config(case):
    return dict(leaf_size=case["leaf"], group_size=case["group"], order=case["order"],
                curve=bh.CURVE_HILBERT if case.get("hilbert") else bh.CURVE_MORTON, max_level=case.get("max_level", 10))


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "train":
        X, Y, order = _features(case, seed)
        P = torch.from_numpy(learned.init_params(seed % 1000)).cuda()
        s.update(X=X, Y=Y, order=order, P=P, m=torch.zeros_like(P), v=torch.zeros_like(P), t=0,
                 work=torch.empty(case["batch"] * bh.MLP_ACT + bh.MLP_NPARAM + 64, device="cuda"))
        return s
    if kind == "batched":
        sizes = _sizes(case)
        offs = np.concatenate([[0], np.cumsum(sizes)])
        n = int(offs[-1])
        pos = _particles("plummer", n, seed)
        pos[:, 3] = torch.from_numpy(np.repeat(1.0 / sizes, sizes)).float().cuda()
        s["pos"], s["out"] = pos, torch.empty_like(pos)
        s["ctx"] = bh.Context(n, max_systems=case["systems"], leaf_size=case["leaf"], group_size=case["group"],
                              order=case["order"], block_threads=64)
        if bh.bh_batch_layout(s["ctx"].h, offs) != 0:
            raise RuntimeError("bh_batch_layout")
        s["graph"] = bh.BatchedGraph(s["ctx"], pos, case["theta"], EPS["plummer"], s["out"])
        return s
    s["pos"] = pos = _particles(case["shape"], case["n"], seed)
    s["eps"] = EPS[case["shape"]]
    if kind == "direct":
        pick = torch.randperm(case["n"], generator=_gen(seed + 2), device="cuda")[: case["targets"]]
        s["index"] = torch.sort(pick).values
        s["tgt"] = pos[s["index"]].contiguous()
        if case["each"]:
            s["lengths"] = _softening(case["n"], s["eps"], seed)
            s["tgt_lengths"] = s["lengths"][s["index"]].contiguous()
        return s
    if kind == "orbit":
        s["orbit"] = Leapfrog(pos, dt=1e-4, theta=case["theta"], eps=s["eps"], **_config(case))
        return s
    if kind == "neighbors":
        s["ctx"] = bh.Context(case["n"], leaf_size=case["leaf"], group_size=case["group"])
        s["h"] = _radii(case, pos)
        return s
    s["ctx"] = bh.Context(case["n"], **_config(case))
    s["out"] = torch.empty_like(pos)
    if kind == "symmetrized":
        s["lengths"] = _softening(case["n"], s["eps"], seed)
    if kind == "learned":
        params, fmin, fmax, _ = learned.load(WEIGHTS)
        if bh.bh_mac_set(s["ctx"].h, params, fmin, fmax, TAU[case["shape"]], 0.5) != 0:
            raise RuntimeError("bh_mac_set")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("evaluate", "learned"):
        return s["ctx"].evaluate(s["pos"], case["theta"], s["eps"], s["out"])
    if kind == "particle":
        return s["ctx"].evaluate(s["pos"], case["theta"], s["eps"], s["out"], walk="particle")
    if kind == "symmetrized":
        return s["ctx"].evaluate_symmetrized(s["pos"], s["lengths"], case["theta"], s["out"])
    if kind == "orbit":
        s["orbit"].step()
        return {"pos": s["orbit"].pos, "vel": s["orbit"].vel, "acc": s["orbit"].acc}
    if kind == "neighbors":
        return s["ctx"].neighbors(s["pos"], s["h"])
    if kind == "batched":
        s["graph"].launch()
        return s["out"]
    if kind == "direct":
        out = torch.empty((case["targets"], 4), device="cuda",
                          dtype=torch.float64 if case["precision"] == 64 else torch.float32)
        if case["each"]:
            rc = bh.direct_force_sym(s["pos"], s["lengths"], s["tgt"], s["tgt_lengths"], s["index"], out,
                                     case["precision"])
        else:
            rc = bh.direct_force(s["pos"], s["tgt"], s["index"], s["eps"], out, case["precision"])
        if rc != 0:
            raise RuntimeError("direct_force: %d" % rc)
        return out
    loss = torch.zeros(case["steps"], device="cuda")
    rc = bh.bh_mlp_train(s["X"], s["Y"], s["order"], s["P"], s["m"], s["v"], s["work"], case["steps"], case["batch"],
                         1e-3, 4.0, loss, s["t"])
    if rc != 0:
        raise RuntimeError("bh_mlp_train: %d" % rc)
    s["t"] += case["steps"]
    return {"params": s["P"], "m": s["m"], "v": s["v"], "loss": loss}


# ---------------------------------------------------------------- work
def _terms(n, theta, kind):
    """Interactions per particle, about: a line in log2 n over theta^2, fitted to the counts that the library reports
    for its benchmark sets; the walk per particle needs half of the group walk's, the learned criterion 0.6 of those
    at the angle of the same accuracy."""
    if kind == "learned":
        theta = 0.54
    per = 69.0 * max(1.0, math.log2(n) - 5.4) / theta ** 2.08
    per *= {"particle": 0.5, "symmetrized": 0.5, "learned": 0.6}.get(kind, 1.0)
    return min(per, n - 1)


def work(case):
    kind = case["kind"]
    if kind == "train":
        # forward, backward and the weights' gradient: 6 flops per weight and sample
        return {"bytes": case["steps"] * (case["batch"] * 32 + bh.MLP_NPARAM * 24),
                "flops": case["steps"] * (case["batch"] * 6 * bh.MLP_NPARAM + bh.MLP_NPARAM * 12)}
    if kind == "direct":
        wide = 32 if case["precision"] == 64 else 16
        return {"bytes": case["n"] * 16 + case["targets"] * (24 + wide), "flops": 19 * case["n"] * case["targets"]}
    if kind == "neighbors":
        # each particle and its neighbours: the pair rule and the kernel
        return {"bytes": case["n"] * (16 + 4 + 8), "flops": case["n"] * (case["ngb"] + 1) * 20}
    flop = 19 if case["order"] == 1 else 40  # a quadrupole term takes 54; three of five terms are cells
    if kind == "batched":
        sizes = _sizes(case)
        return {"bytes": int(sizes.sum()) * 32,
                "flops": float(sum(k * _terms(k, case["theta"], kind) for k in sizes.tolist())) * flop}
    move = {"orbit": 80, "symmetrized": 36}.get(kind, 32)
    return {"bytes": case["n"] * move, "flops": case["n"] * _terms(case["n"], case["theta"], kind) * flop}


# ---------------------------------------------------------------- 64-bit results
PAIRS = 4e10  # pairs that plain 64-bit arithmetic sums in a few seconds


def _direct64(src, tgt, index, eps2_src, eps2_tgt):
    """Eq. (1) in 64 bits: pair softening eps2_src + eps2_tgt, the source `index` of each target left out."""
    src, tgt = src.double(), tgt.double()
    out = torch.empty((tgt.shape[0], 4), device="cuda", dtype=torch.float64)
    step = max(1, int(4e7 // max(1, src.shape[0])))
    for i in range(0, tgt.shape[0], step):
        j = min(tgt.shape[0], i + step)
        d = [src[None, :, k] - tgt[i:j, k, None] for k in range(3)]
        w = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2_src[None, :] + eps2_tgt[i:j, None]).rsqrt_()
        m = src[:, 3].expand(j - i, -1).clone()
        m[torch.arange(j - i, device="cuda"), index[i:j]] = 0.0
        w = torch.where(m == 0, torch.zeros_like(w), w)
        out[i:j, 3] = -(m * w).sum(1)
        m *= w * w * w
        for k in range(3):
            out[i:j, k] = (m * d[k]).sum(1)
    return out


def _density64(pos, h):
    """Densities in 64 bits over the neighbours that the FP32 rule names."""
    n = pos.shape[0]
    hh = torch.full((n,), float(h), device="cuda") if not torch.is_tensor(h) else h
    x, h64 = pos.double(), hh.double()
    rho = torch.empty(n, device="cuda", dtype=torch.float64)
    step = max(1, int(3e7 // n))
    for i in range(0, n, step):
        j = min(n, i + step)
        r2 = sum((x[None, :, k] - x[i:j, k, None]).square() for k in range(3))
        q = r2.sqrt() / h64[i:j, None]
        w = torch.where(q <= 0.5, 1.0 - 6.0 * q * q * (1.0 - q), 2.0 * (1.0 - q).clamp(min=0.0) ** 3)
        rho[i:j] = (w * x[None, :, 3]).sum(1) * 8.0 / (math.pi * h64[i:j] ** 3)
    return rho


def _train64(case, s):
    X, Y = s["X"].double(), s["Y"].double()
    P = s["P"].double().clone().requires_grad_(True)
    m, v, losses = torch.zeros_like(P), torch.zeros_like(P), []
    n, B = case["samples"], case["batch"]
    for t in range(case["steps"]):
        at = s["order"][(torch.arange(B, device="cuda") + (t * B) % n) % n].long()
        w1, b1, w2, b2, w3, b3 = torch.split(P, [192, 32, 1024, 32, 32, 1])
        h = torch.relu(X[at] @ w1.view(32, 6).T + b1)
        y = torch.relu(h @ w2.view(32, 32).T + b2) @ w3 + b3
        r = y - Y[at]
        loss = (torch.where(r < 0, 4.0, 1.0) * r * r).mean()
        g, = torch.autograd.grad(loss, P)
        losses.append(loss.detach())
        with torch.no_grad():
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            P -= 1e-3 * (m / (1 - 0.9 ** (t + 1))) / ((v / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
    return {"params": P.detach(), "m": m, "v": v, "loss": torch.stack(losses)}


def exact(case, seed):
    """Forces: Eq. (1) summed directly, so the tree's own truncation at theta is part of the distance from it."""
    kind = case["kind"]
    if kind == "train":
        X, Y, order = _features(case, seed)
        return _train64(case, dict(X=X, Y=Y, order=order, P=torch.from_numpy(learned.init_params(seed % 1000)).cuda()))
    if kind == "batched":
        sizes = _sizes(case)
        if float((sizes.astype(np.float64) ** 2).sum()) > PAIRS:
            return None
        offs = np.concatenate([[0], np.cumsum(sizes)])
        pos = _particles("plummer", int(offs[-1]), seed)
        pos[:, 3] = torch.from_numpy(np.repeat(1.0 / sizes, sizes)).float().cuda()
        e2 = torch.full((int(sizes.max()),), 0.5 * EPS["plummer"] ** 2, device="cuda", dtype=torch.float64)
        parts = []
        for a, b in zip(offs[:-1], offs[1:]):
            x = pos[a:b]
            parts.append(_direct64(x, x, torch.arange(b - a, device="cuda"), e2[: b - a], e2[: b - a]))
        return torch.cat(parts)
    n = case["n"]
    if float(n) * case.get("targets", n) > PAIRS:
        return None
    pos = _particles(case["shape"], n, seed)
    if kind == "neighbors":
        return [None, _density64(pos, _radii(case, pos))]
    eps = EPS[case["shape"]]
    e2 = torch.full((n,), 0.5 * eps * eps, device="cuda", dtype=torch.float64)
    if kind == "symmetrized" or (kind == "direct" and case["each"]):
        e2 = 0.5 * _softening(n, eps, seed).double() ** 2
    if kind == "direct":
        pick = torch.randperm(n, generator=_gen(seed + 2), device="cuda")[: case["targets"]]
        index = torch.sort(pick).values
        return _direct64(pos, pos[index], index, e2, e2[index])
    acc = _direct64(pos, pos, torch.arange(n, device="cuda"), e2, e2)
    if kind != "orbit":
        return acc
    vel = torch.zeros_like(acc)
    vel[:, :3] = acc[:, :3] * 0.5e-4
    new = pos.double()
    new[:, :3] += 1e-4 * vel[:, :3]
    return {"pos": new, "vel": vel, "acc": acc}
