"""The work that users of this package have it do, as cases that can be timed
and compared: force evaluations (tree build, group walk, force sum), leapfrog
steps, captured steps of one system and of batches, the learned opening angle
and its training, the brute-force sum, the FP64 judge and the neighbour
search, each through the package's public entry points.

A case is a dict of plain values; `prepare` makes its inputs (on the GPU, from
a seed) and the context a program would keep; `run` is one pass; `exact` is
the same pass in FP64 by plain torch, without this package's code.
"""
import math

import numpy as np
import torch

import paper_0909_0541_gb300 as nb

DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest force evaluation of the tree / brute-force crossover sweep:
        # all launches and waits
        dict(name="force_sphere_1000", kind="force", dist="sphere", n=1000, eps=1 / 64, theta=0.6,
             n_crit=32, precision="fp32", order="morton", quad=False),
        # one eager step of the 16k Plummer sphere, the ordinary small simulation
        dict(name="step_plummer_16384", kind="step", dist="plummer", n=16384, eps=1 / 64,
             theta=0.75, n_crit=64, dt=1 / 128, precision="fp32"),
        # one force evaluation of a 2M clustered set at the wide opening angle
        dict(name="force_halos_2m", kind="force", dist="halos", n=1 << 21, eps=1e-3, theta=1.0,
             n_crit=256, precision="fp32", order="morton", quad=False),
        # compensated sums in Peano-Hilbert order, an odd mid-size set
        dict(name="force_halos_500003_comp", kind="force", dist="halos", n=500003, eps=5e-4,
             theta=0.6, n_crit=200, precision="fp32_comp", order="hilbert", quad=False),
        # quadrupole cells at the angle that meets a 1e-3 error with them
        dict(name="force_halos_500k_quad", kind="force", dist="halos", n=500000, eps=5e-4,
             theta=0.98, n_crit=256, precision="fp32", order="morton", quad=True),
        # the production run: captured steps of the 2.87M halo mix
        dict(name="graph_halos_2870k", kind="graph", dist="halos", n=2870000, systems=1, eps=5e-4,
             theta=0.6, n_crit=256, dt=1 / 1024, steps=2),
        # captured steps of 512 independent systems of uneven size
        dict(name="graph_batch_512", kind="graph", dist="mixed", n=7660000, systems=512, eps=1 / 64,
             theta=0.75, n_crit=256, dt=1 / 128, steps=2),
        # force evaluation with the learned per-group opening angle
        dict(name="learned_halos_1m", kind="learned", dist="halos", n=1 << 20, eps=5e-4, n_crit=256,
             mode=1),
        # training the opening-angle network, the size of a labelled set
        dict(name="train_10527", kind="train", n=10527, batch=256, epochs=4),
        # brute force in the crossover sweep
        dict(name="direct_sphere_100k", kind="direct", dist="sphere", n=100003, eps=1 / 64,
             precision="fp32"),
        # the FP64 judge of a sample of targets
        dict(name="judge_halos_4096", kind="judge", dist="halos", n=524288, targets=4096, eps=5e-4),
        # fixed-radius neighbours, about 48 each
        dict(name="neigh_sphere_300k", kind="neigh", dist="sphere", n=300000, mean=48.0, n_crit=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "step", "graph", "batch", "learned", "train",
                       "direct", "judge", "neigh"])
    dist = rng.choice(["sphere", "plummer", "halos"])
    eps = rng.choice([1 / 64, 1e-3, 5e-4])
    theta = round(rng.uniform(0.5, 1.0), 3)
    n_crit = rng.choice([32, 64, 100, 128, 200, 256, 512])
    if kind == "force":
        quad = rng.random() < 0.25
        return dict(kind="force", dist=dist, n=_log_int(rng, 1000, 1 << 21), eps=eps, theta=theta,
                    n_crit=n_crit, precision=rng.choice(["fp32", "fp32", "fp32_comp"]),
                    order=rng.choice(["morton", "morton", "hilbert"]), quad=quad)
    if kind == "step":
        return dict(kind="step", dist=dist, n=_log_int(rng, 1000, 300000), eps=1 / 64, theta=theta,
                    n_crit=n_crit, dt=1 / 1024, precision=rng.choice(["fp32", "fp32_comp"]))
    if kind == "graph":
        return dict(kind="graph", dist=dist, n=_log_int(rng, 4096, 2870000), systems=1, eps=eps,
                    theta=theta, n_crit=n_crit, dt=1 / 4096, steps=rng.randint(1, 4))
    if kind == "batch":
        systems = _log_int(rng, 4, 256)
        return dict(kind="graph", dist="mixed", n=15000 * systems + rng.randint(0, 999),
                    systems=systems, eps=1 / 64, theta=theta, n_crit=n_crit, dt=1 / 128,
                    steps=rng.randint(1, 4))
    if kind == "learned":
        return dict(kind="learned", dist="halos", n=_log_int(rng, 30000, 1 << 20), eps=eps,
                    n_crit=rng.choice([128, 200, 256]), mode=rng.randint(0, 1))
    if kind == "train":
        return dict(kind="train", n=_log_int(rng, 1000, 20000),
                    batch=rng.choice([64, 100, 128, 256, 512]), epochs=rng.randint(1, 6))
    if kind == "direct":
        return dict(kind="direct", dist=dist, n=_log_int(rng, 1000, 130000), eps=eps,
                    precision=rng.choice(["fp32", "fp32_comp"]))
    if kind == "judge":
        return dict(kind="judge", dist=dist, n=_log_int(rng, 1000, 524288),
                    targets=_log_int(rng, 500, 4096), eps=eps)
    return dict(kind="neigh", dist=rng.choice(["sphere", "plummer"]), n=_log_int(rng, 3000, 300000),
                mean=float(_log_int(rng, 8, 100)), n_crit=rng.choice([32, 64, 100]))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _unit(g, n):
    z = 2.0 * _uniform(g, n) - 1.0
    ph = 2.0 * math.pi * _uniform(g, n)
    s = torch.sqrt((1.0 - z * z).clamp_min(0.0))
    return torch.stack([s * torch.cos(ph), s * torch.sin(ph), z], 1)


def _interp(x, xp, fp):
    """Piecewise linear f(x) through the ascending points (xp, fp)."""
    i = torch.searchsorted(xp, x.contiguous()).clamp(1, xp.numel() - 1)
    x0, x1 = xp[i - 1], xp[i]
    w = ((x - x0) / (x1 - x0).clamp_min(1e-300)).clamp(0.0, 1.0)
    return fp[i - 1] + w * (fp[i] - fp[i - 1])


def _sphere(g, n):
    """Uniform sphere of radius 1 at rest."""
    r = _uniform(g, n) ** (1.0 / 3.0)
    return r[:, None] * _unit(g, n), torch.zeros(n, 3, dtype=torch.float64, device=DEV)


def _plummer(g, n):
    """Plummer sphere (scale radius 1, mass 1, cut at 20) in equilibrium."""
    u = _uniform(g, n).clamp_min(1e-12) * (400.0 / 401.0) ** 1.5
    r = 1.0 / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
    q = torch.linspace(0.0, 1.0, 4097, device=DEV, dtype=torch.float64)
    cdf = torch.cumsum(q * q * (1.0 - q * q) ** 3.5, 0)
    speed = _interp(_uniform(g, n) * cdf[-1], cdf, q) * math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    return r[:, None] * _unit(g, n), speed[:, None] * _unit(g, n)


def _hernquist(g, n):
    """Hernquist sphere (scale radius 1, mass 1, cut at 20), Jeans dispersion."""
    su = torch.sqrt(_uniform(g, n).clamp_min(1e-12) * (20.0 / 21.0) ** 2)
    r = su / (1.0 - su)
    t = 12.0 * r * (1.0 + r) ** 3 * torch.log1p(1.0 / r)
    u = r / (1.0 + r) * (25.0 + 52.0 * r + 42.0 * r * r + 12.0 * r ** 3)
    sig = torch.sqrt(((t - u) / 12.0).clamp_min(0.0))
    vel = torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64) * sig[:, None]
    cap = 0.95 * torch.sqrt(2.0 / (r + 1.0))
    return r[:, None] * _unit(g, n), vel * (cap / vel.norm(dim=1).clamp_min(1e-30)).clamp_max(
        1.0)[:, None]


def _halos(g, n):
    """NFW halos (dN/dM ~ M^-1.9, 80 % of the mass, about 1400 particles each)
    on a uniform background in a unit sphere; the halos' particles have random
    velocities near their halo's virial speed."""
    k = max(8, n // 1435)
    e = -0.9
    mh = (1e-6 ** e + _uniform(g, k) * (1e-2 ** e - 1e-6 ** e)) ** (1.0 / e)
    mh = 0.8 * mh / mh.sum()
    conc = 5.0 + 10.0 * _uniform(g, k)
    centre = _sphere(g, k)[0]
    rvir = (mh / 200.0) ** (1.0 / 3.0)
    nh = int(0.8 * n)
    cum = torch.cumsum(mh, 0)
    h = torch.searchsorted(cum, _uniform(g, nh) * cum[-1]).clamp_max(k - 1)
    x = torch.cat([torch.zeros(1, device=DEV, dtype=torch.float64),
                   torch.logspace(-6, math.log10(15.0), 2048, device=DEV, dtype=torch.float64)])
    mu = torch.log1p(x) - x / (1.0 + x)
    c = conc[h]
    r = _interp(_uniform(g, nh) * (torch.log1p(c) - c / (1.0 + c)), mu, x) * rvir[h] / c
    pos = torch.cat([centre[h] + r[:, None] * _unit(g, nh), _sphere(g, n - nh)[0]])
    sig = 0.6 * torch.sqrt(mh / rvir)[h]
    vel = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    vel[:nh] = torch.randn(nh, 3, generator=g, device=DEV, dtype=torch.float64) * sig[:, None]
    perm = torch.randperm(n, generator=g, device=DEV)
    return pos[perm].contiguous(), vel[perm].contiguous()


def _offsets(g, n, systems):
    """Row offsets of `systems` systems, sizes log-uniform over 1:64, n in all."""
    w = 64.0 ** _uniform(g, systems)
    size = (w / w.sum() * n).floor().long().clamp_min(16)
    size[size.argmax()] += n - size.sum()
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(size, 0)])


def _particles(case, seed):
    """pos, vel (n x 3 float64), mass (n float32), offsets (batches) or None."""
    g = _gen(seed)
    n, dist = case["n"], case["dist"]
    if dist != "mixed":
        pos, vel = dict(sphere=_sphere, plummer=_plummer, halos=_halos)[dist](g, n)
        return pos, vel, torch.full((n,), 1.0 / n, dtype=torch.float32, device=DEV), None
    off = _offsets(g, n, case["systems"])
    size = off[1:] - off[:-1]
    sid = torch.repeat_interleave(torch.arange(size.numel(), device=DEV), size)
    a, b = _plummer(g, n), _hernquist(g, n)
    even = (sid % 2 == 0)[:, None]
    return (torch.where(even, a[0], b[0]), torch.where(even, a[1], b[1]),
            (1.0 / size.double())[sid].float(), off)


def _network(g):
    """Parameters of the opening-angle network: random weights about theta 0.65,
    feature means and spreads of a clustered set (the layout of include/nb.h)."""
    def normal(*s):
        return torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)
    p = torch.zeros(nb.MLP_NPARAM, dtype=torch.float64, device=DEV)
    w1 = torch.zeros(64, 16, dtype=torch.float64, device=DEV)
    w1[:, :12] = normal(64, 12) * math.sqrt(2 / 12)
    p[0:1024] = w1.reshape(-1)
    p[1088:5184] = (normal(64, 64) * math.sqrt(2 / 64)).reshape(-1)
    p[5248:9344] = (normal(64, 64) * math.sqrt(2 / 64)).reshape(-1)
    w4 = normal(64)   # away from zero, where Adam's first steps would be rounding noise
    p[9408:9472] = torch.where(w4 < 0, w4 - 2.0, w4 + 2.0) * 0.03
    p[9920] = -0.45
    p[9928:9940] = torch.tensor([4, -4, -4, -4, 16, -1, 7, 0.5, -3, -2, -1, 0.4])
    p[9944:9960] = 1.0
    p[9944:9956] = torch.tensor([1, 1, 1, 1, 3, 1, 1, 0.2, 1, 1, 1, 0.1])
    return p.float()


def _used(p):
    """The trained parameters without the layout's unused slots."""
    return [p[:9472], p[9920:9921]]


def _training_set(case, seed):
    """(params, feature rows, labels, shuffles): labels a smooth function of
    standardised features with scatter, on the 0.05 grid as measured labels are."""
    g = _gen(seed)
    n = case["n"]
    feat = torch.zeros(n, 16, device=DEV)
    feat[:, :12] = torch.randn(n, 12, generator=g, device=DEV)
    w = torch.randn(12, generator=g, device=DEV)
    z = feat[:, :12] @ w / 3 + 0.2 * torch.randn(n, generator=g, device=DEV)
    labels = (0.3 + torch.round(18 * torch.sigmoid(z)) * 0.05).float()
    params = _network(g)
    params[9928:9940] = 0.0
    params[9944:9960] = 1.0
    order = torch.stack([torch.randperm(n, generator=g, device=DEV) for _ in range(case["epochs"])])
    return params, feat, labels, order.int().contiguous()


def _radius(case):
    """The radius with about `mean` neighbours at the middle of the set."""
    if case["dist"] == "sphere":
        return (case["mean"] / case["n"]) ** (1 / 3)
    # the Plummer sphere's density at its half-mass radius (1.3)
    rho = 3 / (4 * math.pi) * (1 + 1.3 ** 2) ** -2.5
    return (case["mean"] / case["n"] / (4 / 3 * math.pi * rho)) ** (1 / 3)


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.kind = case, case["kind"]
    if s.kind == "train":
        s.params, s.feat, s.labels, s.order = _training_set(case, seed)
        return s
    s.pos, s.vel, s.mass, s.off = _particles(case, seed)
    n = case["n"]
    if s.kind == "direct":
        s.work = torch.empty(max(1, nb.direct_f32_workspace_size(n)), dtype=torch.uint8, device=DEV)
    elif s.kind == "judge":
        s.targets = torch.randperm(n, generator=_gen(seed + 1), device=DEV)[:case["targets"]]
    elif s.kind == "neigh":
        s.ctx = nb.NBody(n, n_crit=case["n_crit"])
        # the table a program keeps its neighbours in, with room to spare
        s.table = torch.full((int(4 * n * case["mean"]),), -1, dtype=torch.int32, device=DEV)
    elif s.kind in ("force", "learned"):
        s.ctx = nb.NBody(n, eps=case["eps"], n_crit=case["n_crit"])
        if s.kind == "learned":
            s.params = _network(_gen(seed + 1))
            s.ctx.set_feature_mode(case["mode"])
        else:
            s.ctx.set_key_order(case["order"])
            s.ctx.set_quadrupole(case["quad"])
        s.acc = torch.empty(n, 3, dtype=torch.float32, device=DEV)
        s.pot = torch.empty(n, dtype=torch.float32, device=DEV)
    elif s.kind == "step":
        s.ctx = nb.NBody(n, eps=case["eps"], theta=case["theta"], n_crit=case["n_crit"],
                         precision=case["precision"])
    else:
        # a captured sequence of steps needs a stream of its own and one
        # synchronising step, which sizes the lists; its replays then queue
        torch.cuda.synchronize()
        s.stream = torch.cuda.Stream()
        s.ctx = nb.NBody(n, eps=case["eps"], theta=case["theta"], n_crit=case["n_crit"],
                         stream=s.stream, max_systems=case["systems"])
        if s.off is None:
            s.ctx.leapfrog_step(s.pos, s.vel, s.mass, case["dt"])
        else:
            s.ctx.leapfrog_step_batched(s.pos, s.vel, s.mass, s.off, case["dt"])
        s.ctx.graph_capture_leapfrog(s.pos, s.vel, s.mass, case["dt"], case["steps"],
                                     offsets=s.off)
        s.ctx.set_sync_checks(False)
    return s


def run(s):
    c = s.case
    if s.kind == "force":
        s.ctx.build_tree(s.pos, s.mass)
        s.ctx.walk_groups(c["theta"], c["n_crit"])
        s.ctx.forces(c["eps"], s.acc, s.pot, c["precision"])
        return [s.acc, s.pot]
    if s.kind == "learned":
        s.ctx.build_tree(s.pos, s.mass)
        s.ctx.walk_groups_learned(c["n_crit"], s.params)
        s.ctx.forces(c["eps"], s.acc, s.pot)
        return [s.acc, s.pot]
    if s.kind == "step":
        s.ctx.leapfrog_step(s.pos, s.vel, s.mass, c["dt"])
        return [s.pos, s.vel]
    if s.kind == "graph":
        s.ctx.graph_launch()
        return [s.pos, s.vel]
    if s.kind == "train":
        params = s.params.clone()
        loss = nb.mlp_train(params, s.feat, s.labels, s.order, c["epochs"], c["batch"], 2e-3)
        return _used(params) + [loss]
    if s.kind == "direct":
        return list(nb.direct_f32(s.pos, s.mass, c["eps"], c["precision"], work=s.work))
    if s.kind == "judge":
        return list(nb.direct_sum(s.pos, s.mass, c["eps"], s.targets))
    s.ctx.build_tree(s.pos, s.mass)
    off, idx = s.ctx.neighbours(_radius(c), c["n_crit"])
    s.table[:idx.numel()] = idx
    return [off, s.table]


# ---------------------------------------------------------------- work
def _interactions(case):
    """Force evaluations of one force pass, within about a quarter: per particle
    the list grows with log n and falls as a power of theta (coefficients counted
    on these sets), and the group adds its own members."""
    n, theta = case["n"] / case.get("systems", 1), case.get("theta", 0.65)
    c = dict(sphere=29.0, halos=50.0, plummer=68.0, mixed=75.0)[case["dist"]]
    per = c * math.log2(max(n, 64) / 32) * theta ** -1.85 + 0.4 * min(case["n_crit"], n)
    return case["n"] * min(n, per)


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "train":
        # forward, backward and weight gradients: 3 products per weight and sample
        flops = 6 * (64 * 12 + 2 * 64 * 64 + 64) * n * case["epochs"]
        return dict(bytes=n * (case["epochs"] * 4 + 52) + 8 * nb.MLP_NPARAM, flops=flops)
    if kind == "direct":
        return dict(bytes=44 * n, flops=20.0 * n * n)
    if kind == "judge":
        return dict(bytes=28 * n + 40 * case["targets"], flops=20.0 * n * case["targets"])
    if kind == "neigh":
        return dict(bytes=28 * n + 8 * n + 4 * n * case["mean"], flops=8.0 * n * case["mean"])
    quad = 1.6 if case.get("quad") else 1.0
    flops = 20.0 * _interactions(case) * quad
    if kind in ("force", "learned"):
        return dict(bytes=44 * n, flops=flops)
    return dict(bytes=100 * n, flops=flops * case.get("steps", 1))


def tolerance(case):
    kind = case["kind"]
    if kind == "neigh":
        return "exact"
    if kind == "judge":      # FP64 sums in another order
        return {"rel": 1e-14}
    if kind == "train":      # BF16 operands; the difference grows over the steps
        return {"rel": 3e-3}
    if kind == "direct":
        return {"rel": 2e-6}
    # FP32 coordinates and sums; after a drift a key or an opening test may fall
    # the other way for a few groups, which "max" leaves room for
    return {"rel": 4e-6, "max": 1e-2 if kind in ("step", "graph") else 1e-3}


# ---------------------------------------------------------------- exact
def _spread3(v):
    x = v & 0x1FFFFF
    x = (x | x << 32) & 0x1F00000000FFFF
    x = (x | x << 16) & 0x1F0000FF0000FF
    x = (x | x << 8) & 0x100F00F00F00F00F
    x = (x | x << 4) & 0x10C30C30C30C30C3
    return (x | x << 2) & 0x1249249249249249


CHUNK = 1 << 25   # pairs held at a time


class _Tree:
    """The method in FP64: the oct-tree's cells as runs of particles sharing a
    key prefix, level by level, and the group walk with its FP32 opening test."""

    def __init__(self, pos, mass, off, n_crit, quad):
        n, dev = pos.shape[0], pos.device
        if off is None:
            off = torch.tensor([0, n], device=dev)
        S = off.numel() - 1
        sid = torch.repeat_interleave(torch.arange(S, device=dev), off[1:] - off[:-1])
        at = sid[:, None].expand(n, 3)
        lo = torch.full((S, 3), math.inf, dtype=torch.float64, device=dev).scatter_reduce(
            0, at, pos, "amin")
        hi = torch.full((S, 3), -math.inf, dtype=torch.float64, device=dev).scatter_reduce(
            0, at, pos, "amax")
        self.L = (hi - lo).amax(1) * (1.0 + 2.0 ** -20)
        self.L = torch.where(self.L > 0, self.L, torch.ones_like(self.L))
        self.centre = 0.5 * (lo + hi)
        self.corner = self.centre - 0.5 * self.L[:, None]
        q = ((pos - self.corner[sid]) * (2097152.0 / self.L)[sid, None]).floor().clamp(
            0, 2097151).long()
        key = _spread3(q[:, 0]) << 2 | _spread3(q[:, 1]) << 1 | _spread3(q[:, 2])
        order = torch.sort(key, stable=True)[1]
        order = order[torch.sort(sid[order], stable=True)[1]]
        self.order, self.sid, self.q, key = order, sid[order], q[order], key[order]
        self.x, self.m, self.quad, self.n = pos[order], mass.double()[order], quad, n
        self.nid = []
        for d in range(23):
            p = key >> (63 - 3 * d) if d < 22 else torch.arange(n, device=dev)
            new = torch.ones(n, dtype=torch.bool, device=dev)
            new[1:] = (p[1:] != p[:-1]) | (self.sid[1:] != self.sid[:-1])
            self.nid.append((torch.cumsum(new, 0) - 1).int())
        # groups: the cells of at most n_crit particles under larger ones
        gf, gc, gd = [], [], []
        parent = None
        for d in range(23):
            first, count = self.nodes(d)
            ok = count <= n_crit
            if parent is not None:
                ok &= parent[self.nid[d - 1][first].long()] > n_crit
            parent = count
            gf.append(first[ok])
            gc.append(count[ok])
            gd.append(torch.full_like(first[ok], d))
        gf, gc, gd = torch.cat(gf), torch.cat(gc), torch.cat(gd)
        o = torch.argsort(gf)
        self.gf, self.gc, self.gd = gf[o], gc[o], gd[o]
        G = self.gf.numel()
        gid = torch.repeat_interleave(torch.arange(G, device=dev), self.gc)[:, None].expand(n, 3)
        x32 = self.x.float()
        self.lo = torch.full((G, 3), math.inf, device=dev).scatter_reduce(0, gid, x32, "amin")
        self.hi = torch.full((G, 3), -math.inf, device=dev).scatter_reduce(0, gid, x32, "amax")

    def nodes(self, d):
        nid = self.nid[d]
        new = torch.ones(self.n, dtype=torch.bool, device=nid.device)
        new[1:] = nid[1:] != nid[:-1]
        first = new.nonzero()[:, 0]
        return first, torch.diff(first, append=torch.tensor([self.n], device=nid.device))

    def moments(self, d, first):
        nid, dev = self.nid[d].long(), self.x.device
        M = torch.zeros(first.numel(), dtype=torch.float64, device=dev).index_add_(0, nid, self.m)
        mx = torch.zeros(first.numel(), 3, dtype=torch.float64, device=dev).index_add_(
            0, nid, self.m[:, None] * self.x)
        com = mx / M[:, None]
        l = self.L[self.sid[first]] * 2.0 ** -d
        g = self.corner[self.sid[first]] + (2 * (self.q[first] >> (21 - d)) + 1) * (0.5 * l)[:, None]
        Q = None
        if self.quad:
            r = self.x - com[nid]
            r2 = (r * r).sum(1)
            Q = torch.zeros(first.numel(), 6, dtype=torch.float64, device=dev)
            for k, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                Q[:, k].index_add_(0, nid, self.m * (3 * r[:, a] * r[:, b] - (r2 if a == b else 0)))
        return M, com, l.float(), (com - g).norm(dim=1).float(), Q

    def walk(self, theta, emit):
        """emit(groups, source particle or None, masses, places, quadrupoles) for
        every level's list entries; theta: one opening angle or one per group."""
        dev = self.x.device
        G = self.gf.numel()
        th = torch.full((G,), theta, device=dev) if not torch.is_tensor(theta) else theta
        inv = (1.0 / th.float().double()).float()
        g = torch.arange(G, device=dev)
        node = self.nid[0][self.gf].long()
        for d in range(23):
            if g.numel() == 0:
                break
            first, count = self.nodes(d)
            M = com = None
            if d < 22:
                M, com, l, s, Q = self.moments(d, first)
                child = self.nid[d + 1][first].long()
                nchild = self.nid[d + 1][first + count - 1].long() + 1 - child
            ng, nn = [], []
            for a in range(0, g.numel(), CHUNK):
                gg, u = g[a:a + CHUNK], node[a:a + CHUNK]
                f, c = first[u], count[u]
                own = (self.gd[gg] == d) & (f == self.gf[gg])
                gg, u, f, c = gg[~own], u[~own], f[~own], c[~own]
                leaf = c == 1
                j = f[leaf]
                emit(gg[leaf], j, self.m[j], self.x[j], None)
                gg, u, f, c = gg[~leaf], u[~leaf], f[~leaf], c[~leaf]
                if gg.numel() == 0:
                    continue
                if d == 22:
                    raise AssertionError("a cell below the last level")
                holds = (f <= self.gf[gg]) & (self.gf[gg] + self.gc[gg] <= f + c)
                h = com.float()[u]
                e = torch.maximum(self.lo[gg] - h, h - self.hi[gg]).clamp_min(0.0)
                e = e * e
                d2 = e[:, 0] + e[:, 1]
                d2 = d2 + e[:, 2]
                w = l[u] * inv[gg]
                w = w + s[u]
                far = ~holds & (d2 > w * w)
                emit(gg[far], None, M[u[far]], com[u[far]], Q[u[far]] if self.quad else None)
                gg, u = gg[~far], u[~far]
                k = nchild[u]
                start = torch.cumsum(k, 0) - k
                rep = torch.repeat_interleave(torch.arange(u.numel(), device=dev), k)
                ng.append(gg[rep])
                nn.append(child[u][rep] + torch.arange(rep.numel(), device=dev) - start[rep])
            g = torch.cat(ng) if ng else g[:0]
            node = torch.cat(nn) if nn else node[:0]

    def forces(self, theta, eps):
        """Accelerations and potentials in caller order."""
        dev = self.x.device
        eps2 = float(np.float32(eps)) ** 2
        X = [self.x[:, k].contiguous() for k in range(3)]
        A = [torch.zeros(self.n, dtype=torch.float64, device=dev) for _ in range(4)]

        def add(g, src, m, p, Q):
            if g.numel() == 0:
                return
            c = self.gc[g]
            end = torch.cumsum(c, 0)
            total, a = int(end[-1]), 0
            while a < g.numel():
                base = int(end[a - 1]) if a else 0
                b = g.numel() if total - base <= CHUNK else max(
                    a + 1, int(torch.searchsorted(end, base + CHUNK)))
                k = c[a:b]
                t = torch.repeat_interleave(torch.arange(b - a, device=dev), k)
                at = self.gf[g[a:b]] - (end[a:b] - k - base)
                tgt = at[t] + torch.arange(t.numel(), device=dev)
                D = [p[a:b, q].contiguous()[t] - X[q][tgt] for q in range(3)]
                r2 = D[0] * D[0] + D[1] * D[1] + D[2] * D[2] + eps2
                ok = r2 > 0
                if src is not None:
                    ok &= src[a:b][t] != tgt
                ri = torch.where(ok, r2, 1.0).rsqrt()
                mr = torch.where(ok, m[a:b][t], 0.0) * ri
                pot = mr
                ri2 = ri * ri
                w = mr * ri2
                if Q is not None:
                    q = [Q[a:b, i].contiguous()[t] for i in range(6)]
                    v = [q[0] * D[0] + q[3] * D[1] + q[4] * D[2],
                         q[3] * D[0] + q[1] * D[1] + q[5] * D[2],
                         q[4] * D[0] + q[5] * D[1] + q[2] * D[2]]
                    dqd = v[0] * D[0] + v[1] * D[1] + v[2] * D[2]
                    ri5 = ri2 * ri2 * ri
                    pot = pot + 0.5 * dqd * ri5
                    w = w + 2.5 * dqd * ri5 * ri2
                for i in range(3):
                    A[i].index_add_(0, tgt, w * D[i] - (v[i] * ri5 if Q is not None else 0.0))
                A[3].index_add_(0, tgt, -pot)
                a = b

        self.walk(theta, add)
        # a group's own members
        g = torch.repeat_interleave(torch.arange(self.gf.numel(), device=dev), self.gc)
        j = torch.arange(self.n, device=dev)
        add(g, j, self.m, self.x, None)
        acc = torch.empty(self.n, 3, dtype=torch.float64, device=dev)
        acc[self.order] = torch.stack(A[:3], 1)
        pot = torch.empty(self.n, dtype=torch.float64, device=dev)
        pot[self.order] = A[3]
        return acc, pot

    def features(self, mode):
        """The network's inputs of every group, FP64."""
        G, dev = self.gf.numel(), self.x.device
        s = self.sid[self.gf]
        L = self.L[s]
        side = (self.hi.double() - self.lo.double()) / L[:, None]
        mid = 0.5 * (self.lo.double() + self.hi.double())
        F = torch.zeros(G, 12, dtype=torch.float64, device=dev)
        F[:, 0] = torch.log(self.gc.double())
        F[:, 1:4] = torch.log(side + 1e-7)
        F[:, 4] = F[:, 0] - torch.log(side + 1e-4).sum(1)
        F[:, 5] = torch.log((mid - self.centre[s]).norm(dim=1) / L + 1e-6)
        F[:, 11] = self.gd.double() / 22.0
        if mode == 0:   # statistics of a walk at theta 1.2
            z = torch.zeros(G, dtype=torch.float64, device=dev)
            length, cells, total, far, near = z.clone(), z.clone(), z.clone(), z.clone(), z + 1e300

            def note(g, src, m, p, Q):
                one = torch.ones(g.numel(), dtype=torch.float64, device=dev)
                length.index_add_(0, g, one)
                if src is None and g.numel():
                    r = (p - mid[g]).norm(dim=1)
                    cells.index_add_(0, g, one)
                    total.index_add_(0, g, r)
                    far.scatter_reduce_(0, g, r, "amax")
                    near.scatter_reduce_(0, g, r, "amin")

            self.walk(1.2, note)
            some = cells > 0
            F[:, 6] = torch.log(length + 1.0)
            F[:, 7] = torch.where(length > 0, cells / length.clamp_min(1), z)
            F[:, 8] = torch.log(torch.where(some, near, z) / L + 1e-7)
            F[:, 9] = torch.log(torch.where(some, total / cells.clamp_min(1), z) / L + 1e-7)
            F[:, 10] = torch.log(far / L + 1e-7)
        return F


def _bf16(x):
    return x.float().bfloat16().double()


def _gelu(x):
    return 0.5 * x * (1.0 + torch.erf(x / math.sqrt(2.0)))


def _gelu_grad(x):
    return 0.5 * (1.0 + torch.erf(x / math.sqrt(2.0))) + x * torch.exp(-0.5 * x * x) / math.sqrt(
        2.0 * math.pi)


def _net(p, x):
    """theta and the activations: BF16 operands, FP64 sums."""
    W = [p[0:1024].view(64, 16), p[1088:5184].view(64, 64), p[5248:9344].view(64, 64)]
    b = [p[1024:1088], p[5184:5248], p[9344:9408]]
    z = torch.zeros(x.shape[0], 16, dtype=torch.float64, device=x.device)
    z[:, :12] = (x[:, :12] - p[9928:9940]) / p[9944:9956]
    a, Z = [_bf16(z)], []
    for k in range(3):
        Z.append(a[k] @ _bf16(W[k]).T + b[k])
        h = _gelu(Z[k])
        a.append(_bf16(h))
    s = torch.sigmoid(h @ p[9408:9472] + p[9920])
    return 0.3 + 0.9 * s, (W, a, Z, h, s)


def _train(case, seed):
    params, feat, labels, order = _training_set(case, seed)
    p, x, y = params.double(), feat.double(), labels.double()
    m, v, hist, t = torch.zeros_like(p), torch.zeros_like(p), [], 0
    B = case["batch"]
    for e in range(case["epochs"]):
        loss = 0.0
        for k in range(case["n"] // B):
            i = order[e, k * B:(k + 1) * B].long()
            th, (W, a, Z, h3, s) = _net(p, x[i])
            d = th - y[i]
            up = d.clamp_min(0.0)
            loss = loss + (d * d + 4.0 * up * up).sum()
            dz = (2.0 * d + 8.0 * up) / B * 0.9 * s * (1.0 - s)
            g = torch.zeros_like(p)
            g[9408:9472] = dz @ h3
            g[9920] = dz.sum()
            D = dz[:, None] * p[9408:9472] * _gelu_grad(Z[2])
            for q, (wo, bo) in ((2, (5248, 9344)), (1, (1088, 5184)), (0, (0, 1024))):
                r = _bf16(D)
                gw = r.T @ a[q]
                g[wo:wo + gw.numel()] = gw.reshape(-1)
                g[bo:bo + 64] = D.sum(0)
                if q:
                    D = (r @ _bf16(W[q])) * _gelu_grad(Z[q - 1])
            t += 1
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            p = p - 2e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        hist.append(loss)
    return _used(p) + [torch.stack(hist)]


def _pairs(pos, mass, eps, targets):
    """The direct sum at the targets."""
    nt, n = targets.numel(), pos.shape[0]
    acc = torch.empty(nt, 3, dtype=torch.float64, device=DEV)
    pot = torch.empty(nt, dtype=torch.float64, device=DEV)
    X = [pos[:, k].contiguous() for k in range(3)]
    step = max(1, CHUNK // n)
    j = torch.arange(n, device=DEV)
    for a in range(0, nt, step):
        t = targets[a:a + step]
        D = [X[k][None, :] - X[k][t][:, None] for k in range(3)]
        r2 = D[0] * D[0] + D[1] * D[1] + D[2] * D[2] + eps * eps
        ok = (r2 > 0) & (j[None, :] != t[:, None])
        ri = torch.where(ok, r2, 1.0).rsqrt()
        mr = torch.where(ok, mass[None, :], 0.0) * ri
        pot[a:a + step] = -mr.sum(1)
        w = mr * ri * ri
        for k in range(3):
            acc[a:a + step, k] = (w * D[k]).sum(1)
    return acc, pot


def exact(case, seed):
    kind = case["kind"]
    if kind == "neigh":
        return None
    if kind == "train":
        return _train(case, seed)
    pos, vel, mass, off = _particles(case, seed)
    if kind == "direct":
        return list(_pairs(pos.float().double(), mass.double(), float(np.float32(case["eps"])),
                           torch.arange(case["n"], device=DEV)))
    if kind == "judge":
        t = torch.randperm(case["n"], generator=_gen(seed + 1), device=DEV)[:case["targets"]]
        return list(_pairs(pos, mass.double(), case["eps"], t))

    def tree(x):
        return _Tree(x, mass, off, case["n_crit"], case.get("quad", False))
    if kind == "force":
        return list(tree(pos).forces(float(np.float32(case["theta"])), case["eps"]))
    if kind == "learned":
        T = tree(pos)
        theta = _net(_network(_gen(seed + 1)).double(), T.features(case["mode"]))[0]
        return list(T.forces(theta, case["eps"]))
    theta, dt = float(np.float32(case["theta"])), case["dt"]
    acc = tree(pos).forces(theta, case["eps"])[0]
    for _ in range(1 if kind == "step" else 1 + case["steps"]):
        vel = vel + acc * (0.5 * dt)
        pos = pos + vel * dt
        acc = tree(pos).forces(theta, case["eps"])[0]
        vel = vel + acc * (0.5 * dt)
    return [pos, vel]
