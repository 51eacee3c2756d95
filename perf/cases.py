"""The work that users of this library have it do, as measurable cases.

One case is one call sequence of a simulation step through the entry points of
``paper_2609_17658_gb300.og``, on inputs made from a seed:

* ``step``    a new tree and its short-range accelerations (og_tree_build,
              og_tree_force, og_tree_free), the library's main use;
* ``refit``   drifted positions on a kept tree, then the force;
* ``batch``   many independent periodic boxes in one og_batch_force call;
* ``pot``     the force with the potential output (energy diagnostics);
* ``active``  the force on the active particles of an individual-time-step
              scheme, previous accelerations known;
* ``pm``      the long-range mesh force of a kept tree;
* ``sph``     the SPH density at given smoothing lengths, on a kept tree;
* ``serve``   a handful of requests of mixed size through the serving loop.

Particles are Poisson-uniform, or 70 % in NFW haloes and 30 % uniform; box 1,
total mass 1.  Lengths follow the workloads of the benchmark: softening
1 / (50 N^(1/3)), split scale ``rs_cells`` / N^(1/3), cutoff 4.5 split scales.

Everything is made on the GPU with torch; nothing here calls the library
outside prepare() and run().
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_17658_gb300 import og

BH, REL = 0, 1
# serve: the kick is small enough that a halo core's positions do not amplify
# rounding over the steps
SERVE_STEPS, SERVE_KICK, SERVE_SIGMA = 4, 1e-7, 1e-4
# direct sums (exact) up to this many particles
DIRECT_MAX = 131_072


def listed():
    return [
        # the smallest systems: a step is a chain of short launches; the caller
        # holds numpy arrays (zoom regions, tests of an integrator, halo finders)
        dict(name="step-4k-host", kind="step", n=4096, dist="uniform", opening=BH, rs_cells=0.625, host=True,
             a_old=False, masses="equal"),
        # the 32^3 Poisson-uniform box, Barnes-Hut, with the interaction counts
        dict(name="step-uniform-32k", kind="step", n=32768, dist="uniform", opening=BH, rs_cells=0.625, host=False,
             a_old=False, masses="equal"),
        # an ordinary step inside a run: the previous step's accelerations are
        # known, so one pass with the relative criterion; two particle species
        dict(name="step-halo-100k-aold", kind="step", n=100_003, dist="halo", opening=REL, rs_cells=0.625, host=False,
             a_old=True, masses="mixed"),
        # the 128^3 clustered box: first step of a run, a Barnes-Hut pass
        # supplies the accelerations of the relative criterion
        dict(name="step-halo-2m", kind="step", n=128 ** 3, dist="halo", opening=REL, rs_cells=0.625, host=False,
             a_old=False, masses="equal"),
        # the 256^3 clustered box: the largest single system
        dict(name="step-halo-16m", kind="step", n=256 ** 3, dist="halo", opening=REL, rs_cells=0.625, host=False,
             a_old=False, masses="equal"),
        # a drift step that keeps the tree
        dict(name="refit-halo-200k", kind="refit", n=200_000, dist="halo", opening=BH, rs_cells=0.625,
             sigma=2e-4, masses="equal"),
        # many independent boxes of uneven size at once
        dict(name="batch-128", kind="batch", boxes=128, sizes=1, n_lo=4096, n_hi=262144, rs_cells=0.625),
        # energy diagnostics of an ordinary system
        dict(name="pot-halo-120k", kind="pot", n=120_001, dist="halo", opening=BH, rs_cells=0.625, masses="mixed"),
        # individual time steps: one particle in sixteen is active, most of them
        # in the haloes
        dict(name="active-halo-2m", kind="active", n=128 ** 3, dist="halo", opening=REL, rs_cells=0.625,
             active=1.0 / 16.0, masses="equal"),
        # the long-range half of a TreePM step
        dict(name="pm-halo-2m-256", kind="pm", n=128 ** 3, dist="halo", mesh=256, rs_cells=0.625, masses="equal"),
        # the density loop of an SPH step
        dict(name="sph-halo-2m", kind="sph", n=128 ** 3, dist="halo", ngb=32, rs_cells=0.625, masses="equal"),
        # a serving process: eight requests of mixed size, four kick-drift steps each
        dict(name="serve-8", kind="serve", requests=8, sizes=1, n_lo=10_000, n_hi=400_000, rs_cells=0.625),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "refit", "batch", "pot", "active", "pm", "sph", "serve"])
    dist = rng.choice(["uniform", "halo", "halo"])
    masses = rng.choice(["equal", "mixed"])
    opening = rng.choice([BH, REL])
    if kind == "step":
        host = rng.random() < 0.25
        n = _log_uniform(rng, 4096, 500_000 if host else 8_000_000)
        return dict(kind=kind, n=n, dist=dist, opening=opening, rs_cells=rng.choice([0.625, 1.25]), host=host,
                    a_old=opening == REL and rng.random() < 0.5, masses=masses)
    if kind == "refit":
        return dict(kind=kind, n=_log_uniform(rng, 10_000, 2_000_000), dist=dist, opening=BH, rs_cells=0.625,
                    sigma=rng.choice([5e-5, 2e-4]), masses=masses)
    if kind == "batch":
        return dict(kind=kind, boxes=_log_uniform(rng, 8, 256), sizes=rng.randrange(1, 10000), n_lo=4096, n_hi=rng.choice([32768, 131072, 262144]),
                    rs_cells=0.625)
    if kind == "pot":
        return dict(kind=kind, n=_log_uniform(rng, 4096, 2_000_000), dist=dist, opening=BH,
                    rs_cells=rng.choice([0.625, 1.25]), masses=masses)
    if kind == "active":
        return dict(kind=kind, n=_log_uniform(rng, 50_000, 4_000_000), dist=dist, opening=opening, rs_cells=0.625,
                    active=rng.choice([1.0 / 64.0, 1.0 / 16.0, 1.0 / 4.0]), masses=masses)
    if kind == "pm":
        mesh = rng.choice([64, 128, 256, 512])
        return dict(kind=kind, n=_log_uniform(rng, 30_000, 8_000_000), dist=dist, mesh=mesh, rs_cells=0.625,
                    masses=masses)
    if kind == "sph":
        return dict(kind=kind, n=_log_uniform(rng, 10_000, 4_000_000), dist=dist, ngb=rng.choice([32, 64]),
                    rs_cells=0.625, masses=masses)
    return dict(kind="serve", requests=rng.randint(2, 12), sizes=rng.randrange(1, 10000), n_lo=10_000, n_hi=rng.choice([100_000, 400_000]),
                rs_cells=0.625)


# ---- inputs -----------------------------------------------------------------

def _nfw_mu(x):
    return torch.log1p(x) - x / (1.0 + x)


def _halo_counts(r, n_halo, total, n_max):
    """Halo particle counts from dN/dn ~ n^-1.9 on [32, n_max], rescaled to sum to total."""
    a = -0.9
    raw = (32.0 ** a + r.random(n_halo) * (float(n_max) ** a - 32.0 ** a)) ** (1.0 / a)
    scaled = raw * (total / raw.sum())
    counts = np.floor(scaled).astype(np.int64)
    order = np.argsort(-(scaled - counts), kind="stable")
    counts[order[: total - int(counts.sum())]] += 1
    return counts


def _particles(n, dist, masses, seed):
    """(pos [n,3] f64, mass [n] f64, a [n,3] f32) on the GPU: positions in the unit box, masses of
    sum about 1, and the haloes' own analytic accelerations (what a previous step would have
    left, to a factor of a few)."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 17)
    f64 = dict(dtype=torch.float64, device=dev, generator=g)
    n_in = int(round(0.7 * n)) if dist == "halo" else 0
    n_halo = max(1, min(int(round(2000 * n / 128 ** 3)), n_in // 32)) if n_in >= 32 else 0
    if n_halo == 0:
        n_in = 0
    out = n - n_in
    pos = torch.rand((n, 3), **f64)
    acc = torch.randn((n, 3), dtype=torch.float32, device=dev, generator=g)
    if n_in:
        r = np.random.Generator(np.random.PCG64(int(seed)))
        counts = torch.from_numpy(_halo_counts(r, n_halo, n_in, max(64, n // 20))).to(dev)
        m_h = counts.double() / n
        r200 = (3.0 * m_h / (4.0 * math.pi * 200.0)) ** (1.0 / 3.0)
        owner = torch.repeat_interleave(torch.arange(n_halo, device=dev), counts)
        mu_c = math.log1p(10.0) - 10.0 / 11.0
        target = torch.rand((n_in,), **f64) * mu_c
        lo, hi = torch.zeros_like(target), torch.full_like(target, 10.0)
        for _ in range(45):
            mid = 0.5 * (lo + hi)
            below = _nfw_mu(mid) < target
            lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
        x = (0.5 * (lo + hi)).clamp_(min=1e-6)
        rs = (r200 / 10.0)[owner]
        u = torch.randn((n_in, 3), **f64)
        u /= u.norm(dim=1, keepdim=True)
        centre = torch.rand((n_halo, 3), **f64)
        pos[out:] = centre[owner] + u * (x * rs)[:, None]
        amag = m_h[owner] * _nfw_mu(x) / mu_c / (x * rs) ** 2
        acc[out:] -= (u * amag[:, None]).float()
        order = torch.randperm(n, device=dev, generator=g)
        pos, acc = pos[order], acc[order]
    pos = torch.remainder(pos, 1.0)
    pos[pos >= 1.0] = 0.0
    mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device=dev)
    if masses == "mixed":  # two species in the cosmic baryon ratio
        mass *= torch.where(torch.rand((n,), **f64) < 0.5, 0.3125, 1.6875)
    return pos.contiguous(), mass, acc.contiguous()


def _smoothing(pos, ngb):
    """Smoothing lengths that hold about ngb neighbours: from the number density of the finest
    grid cell around each particle that holds at least ngb particles."""
    h = torch.full((pos.shape[0],), 0.2, dtype=torch.float64, device=pos.device)
    for level in range(2, 13):
        side = 1 << level
        i = (pos * side).to(torch.int64)
        _, at, count = torch.unique((i[:, 0] * side + i[:, 1]) * side + i[:, 2], return_inverse=True, return_counts=True)
        held = count[at].double()
        here = (3.0 * ngb / (4.0 * math.pi * held)) ** (1.0 / 3.0) / side
        h = torch.where(held >= ngb, here, h)
    return h.clamp_(max=0.2).float().contiguous()


def _params(n, opening, rs_cells):
    side = n ** (1.0 / 3.0)
    return dict(box=1.0, G=1.0, eps=1.0 / (50.0 * side), r_s=rs_cells / side, rcut_over_rs=4.5, opening=opening,
                theta=0.5, alpha=0.0025 if n > 8_000_000 else 0.005, theta_first_pass=0.5)


def _box_sizes(case):
    """Sizes of the systems of a batch or stream, log-uniform over the range; the seed of the
    inputs does not change them."""
    r = np.random.Generator(np.random.PCG64(int(case["sizes"])))
    count = case.get("boxes") or case["requests"]
    # one size in each part of the range
    q = (np.arange(count) + r.random(count)) / count
    sizes = np.exp(np.log(case["n_lo"]) + q * (np.log(case["n_hi"]) - np.log(case["n_lo"])))
    r.shuffle(sizes)
    return [int(round(x)) for x in sizes], (r.random(count) < 0.5).tolist()


_held = {}


def _context():
    """The one context and stream that a program keeps."""
    if not _held:
        _held["stream"] = torch.cuda.Stream()
        _held["ctx"] = og.Context(torch.cuda.current_device())
        og.og_set_stream(_held["ctx"].h, _held["stream"].cuda_stream)
    return _held["ctx"], _held["stream"]


class _State:
    """Inputs, output buffers and the tree (if kept) of one case."""

    def __init__(self, case):
        self.case = dict(case)
        self.tree = None

    def __del__(self):
        if self.tree is not None:
            og.og_tree_free(self.tree)


def prepare(case, seed):
    ctx, stream = _context()
    s = _State(case)
    s.ctx = ctx
    kind = case["kind"]
    with torch.cuda.stream(stream):
        if kind == "batch":
            sizes, halo = _box_sizes(case)
            total = sum(sizes)
            dev = torch.device("cuda")
            s.acc = torch.zeros((total, 3), dtype=torch.float32, device=dev)
            s.n_pp = torch.zeros(total, dtype=torch.int32, device=dev)
            s.n_pn = torch.zeros(total, dtype=torch.int32, device=dev)
            s.boxes, o = [], 0
            for k, n in enumerate(sizes):
                pos, mass, _ = _particles(n, "halo" if halo[k] else "uniform", "equal", int(seed) * 1009 + k)
                s.boxes.append(dict(pos=pos, mass=mass, params=_params(n, BH, case["rs_cells"]), acc=s.acc[o:o + n],
                                    n_pp=s.n_pp[o:o + n], n_pn=s.n_pn[o:o + n]))
                o += n
        elif kind == "serve":
            sizes, _ = _box_sizes(case)
            r = np.random.Generator(np.random.PCG64(int(seed) + 1))
            s.requests = []
            for k, n in enumerate(sizes):
                pos, mass, _ = _particles(n, "halo", "equal", int(seed) * 1009 + k)
                s.requests.append(dict(pos=pos.cpu().numpy(), vel=r.normal(0.0, SERVE_SIGMA, (n, 3)),
                                       mass=mass.cpu().numpy(), params=_params(n, BH, case["rs_cells"]),
                                       acc=np.zeros((n, 3), np.float32), out=np.zeros((n, 3))))
        else:
            n = case["n"]
            s.pos, s.mass, a_old = _particles(n, case["dist"], case["masses"], seed)
            s.prm = _params(n, case.get("opening", BH), case["rs_cells"])
            dev = s.pos.device
            s.acc = torch.zeros((n, 3), dtype=torch.float32, device=dev)
            s.a_old = a_old if case.get("a_old") or (kind == "active" and case["opening"] == REL) else None
            # the counts, where the first pass's rounding cannot move them
            counts = s.prm["opening"] == BH or s.a_old is not None
            s.n_pp = torch.zeros(n, dtype=torch.int32, device=dev) if counts else None
            s.n_pn = torch.zeros(n, dtype=torch.int32, device=dev) if counts else None
            if case.get("host"):
                s.pos, s.mass, s.acc = s.pos.cpu().numpy(), s.mass.cpu().numpy(), s.acc.cpu().numpy()
                s.a_old = None if s.a_old is None else s.a_old.cpu().numpy()
                s.n_pp = np.zeros(n, np.uint32) if counts else None
                s.n_pn = np.zeros(n, np.uint32) if counts else None
            if kind == "pot":
                s.pot = torch.zeros(n, dtype=torch.float32, device=dev)
            if kind == "active":
                g = torch.Generator(device=dev)
                g.manual_seed(int(seed) + 3)
                # the deepest particles first, with some scatter
                key = a_old.norm(dim=1) * torch.exp(torch.randn(n, device=dev, generator=g))
                s.active = (key >= torch.topk(key, max(1, int(n * case["active"]))).values[-1]).to(torch.uint8)
            if kind == "sph":
                s.h = _smoothing(s.pos, case["ngb"])
                s.rho = torch.zeros(n, dtype=torch.float32, device=dev)
                s.n_ngb = torch.zeros(n, dtype=torch.int32, device=dev)
            if kind in ("refit", "active", "pm", "sph"):
                s.tree = og.og_tree_build(ctx.h, s.pos, s.mass, s.prm)
            if kind == "refit":
                g = torch.Generator(device=dev)
                g.manual_seed(int(seed) + 5)
                s.pos = torch.remainder(s.pos + case["sigma"] * torch.randn((n, 3), dtype=torch.float64, device=dev,
                                                                            generator=g), 1.0).contiguous()
    return s


def _counted(s, **more):
    out = dict(acc=s.acc, **more)
    if s.n_pp is not None:
        out.update(n_pp=s.n_pp, n_pn=s.n_pn)
    return out


def run(s):
    kind = s.case["kind"]
    if kind == "step":
        t = og.og_tree_build(s.ctx.h, s.pos, s.mass, s.prm)
        og.og_tree_force(t, s.acc, s.a_old, s.n_pp, s.n_pn)
        og.og_tree_free(t)
        return _counted(s)
    if kind == "refit":
        og.og_tree_refit(s.tree, s.pos)
        og.og_tree_force(s.tree, s.acc, None, s.n_pp, s.n_pn)
        return _counted(s)
    if kind == "batch":
        og.og_batch_force(s.ctx.h, s.boxes)
        return dict(acc=s.acc, n_pp=s.n_pp, n_pn=s.n_pn)
    if kind == "pot":
        t = og.og_tree_build(s.ctx.h, s.pos, s.mass, s.prm)
        og.og_tree_force_pot(t, s.acc, s.pot, None, s.n_pp, s.n_pn)
        og.og_tree_free(t)
        return _counted(s, pot=s.pot)
    if kind == "active":
        og.og_tree_force_active(s.tree, s.active, s.acc, s.a_old, s.n_pp, s.n_pn)
        return _counted(s)
    if kind == "pm":
        og.og_tree_pm_force(s.tree, s.case["mesh"], s.acc)
        return dict(acc=s.acc)
    if kind == "sph":
        og.og_tree_sph_density(s.tree, s.h, s.rho, s.n_ngb)
        return dict(rho=s.rho, n_ngb=s.n_ngb)
    tickets = [og.og_serve_submit(s.ctx.h, q["pos"], q["vel"], q["mass"], q["params"], SERVE_STEPS, SERVE_KICK, 1.0,
                                  acc_out=q["acc"], pos_out=q["out"]) for q in s.requests]
    for t in tickets:
        og.og_serve_poll(s.ctx.h, t, -1)
    return dict(acc=[q["acc"] for q in s.requests], pos=[q["out"] for q in s.requests])


# interactions a particle (list entries evaluated) of one pass, as the library
# counts them: 45 operations each
def _interactions(n, dist, opening):
    if dist == "uniform":
        return 500.0
    return (1300.0 if n > 8_000_000 else 980.0 if opening == REL else 650.0)


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        sizes, _ = _box_sizes(case)
        n = sum(sizes)
        if kind == "batch":
            return dict(bytes=n * (32 + 12 + 8), flops=45.0 * 575.0 * n)
        return dict(bytes=n * (56 + 12 + 24), flops=45.0 * 650.0 * n * SERVE_STEPS)
    n = case["n"]
    if kind == "pm":
        m = case["mesh"] ** 3
        return dict(bytes=n * (12 + 4 + 12 + 4), flops=5.0 * m * math.log2(m) + 300.0 * n)
    if kind == "sph":
        return dict(bytes=n * (12 + 4 + 4 + 4 + 4), flops=20.0 * case["ngb"] * n)
    per = _interactions(n, case["dist"], case["opening"])
    passes = 2 if case["opening"] == REL and not case.get("a_old") and kind == "step" else 1
    if kind == "active":
        return dict(bytes=n * 1 + n * case["active"] * (12 + 12 + 8), flops=45.0 * per * n * case["active"])
    nbytes = n * (32 + 12 + 8) + (12 * n if case.get("a_old") else 0) + (4 * n if kind == "pot" else 0)
    return dict(bytes=nbytes, flops=45.0 * per * passes * n)


# ---- the same in 64 bits ------------------------------------------------------

def _grid(pos):
    """Positions on the library's 32-bit grid, as exact 64-bit integers."""
    return torch.remainder(torch.floor(pos * 4294967296.0), 4294967296.0).to(torch.int64)


def _direct(pos, mass, prm, want_pot):
    """Direct sum of the split, softened pair force: what the tree approximates."""
    q = _grid(pos)
    n = q.shape[0]
    s = 2.0 ** -32
    h, rs = 2.8 * prm["eps"], prm["r_s"]
    rc2 = (prm["rcut_over_rs"] * rs) ** 2
    acc = torch.zeros((n, 3), dtype=torch.float64, device=q.device)
    pot = torch.zeros(n, dtype=torch.float64, device=q.device)
    # targets in order of x: the sources of a block are those within the cutoff in x
    order = torch.argsort(q[:, 0])
    q, m = q[order], mass[order]
    x = q[:, 0].contiguous()
    reach = int(math.ceil(math.sqrt(rc2) / s)) + 1
    rows = 512
    for b in range(0, n, rows):
        t = q[b:b + rows]
        lo, hi = int(t[0, 0]) - reach, int(t[-1, 0]) + reach
        if hi - lo >= 2 ** 32:
            src, ms = q, m
        else:
            edges = torch.tensor([lo, hi + 1, lo + 2 ** 32, hi + 1 - 2 ** 32], device=q.device)
            e = torch.searchsorted(x, edges).tolist()
            parts = [slice(e[0], e[1])]
            if lo < 0:
                parts.append(slice(e[2], n))
            if hi >= 2 ** 32:
                parts.append(slice(0, e[3]))
            src = torch.cat([q[p] for p in parts])
            ms = torch.cat([m[p] for p in parts])
        for c in range(0, src.shape[0], 16384):
            d = src[None, c:c + 16384] - t[:, None]
            d = (torch.remainder(d + 2 ** 31, 2 ** 32) - 2 ** 31).double() * s
            r2 = (d * d).sum(2)
            i, j = torch.nonzero((r2 < rc2) & (r2 > 0.0), as_tuple=True)
            r2, d, w = r2[i, j], d[i, j], ms[c:c + 16384][j]
            r = r2.sqrt()
            u = r / h
            g = torch.where(u < 0.5, (32.0 / 3.0 - 38.4 * u ** 2 + 32.0 * u ** 3) / h ** 3,
                            (64.0 / 3.0 - 48.0 * u + 38.4 * u ** 2 - 32.0 / 3.0 * u ** 3 - 1.0 / (15.0 * u ** 3)) /
                            h ** 3)
            g = torch.where(u < 1.0, g, r ** -3)
            v = r / (2.0 * rs)
            ec = torch.erfc(v)
            f = w * g * (ec + 2.0 / math.sqrt(math.pi) * v * torch.exp(-v * v))
            acc.index_add_(0, order[b + i], f[:, None] * d)
            if want_pot:
                psi = torch.where(
                    u < 0.5, (2.8 - 16.0 / 3.0 * u ** 2 + 9.6 * u ** 4 - 6.4 * u ** 5) / h,
                    (3.2 - 1.0 / (15.0 * u) - 32.0 / 3.0 * u ** 2 + 16.0 * u ** 3 - 9.6 * u ** 4 +
                     32.0 / 15.0 * u ** 5) / h)
                psi = torch.where(u < 1.0, psi, 1.0 / r)
                pot.index_add_(0, order[b + i], -w * psi * ec)
    return acc * prm["G"], pot * prm["G"]


def _mesh_force(pos, mass, ng, rs):
    """Cloud-in-cell mesh force with the deconvolved Green's function, in 64 bits."""
    dev = pos.device
    x = _grid(pos).double() * (ng / 4294967296.0)
    i0 = x.floor()
    f = x - i0
    i0 = i0.to(torch.int64)
    rho = torch.zeros(ng ** 3, dtype=torch.float64, device=dev)
    corners = [(a, b, c) for a in (0, 1) for b in (0, 1) for c in (0, 1)]

    def corner(a, b, c):
        w = (f[:, 0] if a else 1 - f[:, 0]) * (f[:, 1] if b else 1 - f[:, 1]) * (f[:, 2] if c else 1 - f[:, 2])
        i = torch.remainder(i0 + torch.tensor([a, b, c], device=dev), ng)
        return w, (i[:, 0] * ng + i[:, 1]) * ng + i[:, 2]

    for a in corners:
        w, at = corner(*a)
        rho.index_add_(0, at, mass * w)
    rho = rho.view(ng, ng, ng) * ng ** 3
    k = 2.0 * math.pi * torch.fft.fftfreq(ng, 1.0 / ng, dtype=torch.float64, device=dev)
    kz = 2.0 * math.pi * torch.fft.rfftfreq(ng, 1.0 / ng, dtype=torch.float64, device=dev)
    win = torch.exp(-(k * rs) ** 2) / torch.sinc(k / (2.0 * math.pi * ng)) ** 4
    winz = torch.exp(-(kz * rs) ** 2) / torch.sinc(kz / (2.0 * math.pi * ng)) ** 4
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    green = -4.0 * math.pi * (win[:, None, None] * win[None, :, None] * winz[None, None, :]) / k2
    green[0, 0, 0] = 0.0
    phi = torch.fft.irfftn(torch.fft.rfftn(rho) * green, s=(ng, ng, ng))
    acc = torch.zeros_like(pos)
    for axis in range(3):
        grad = (8.0 * (phi.roll(-1, axis) - phi.roll(1, axis)) - (phi.roll(-2, axis) - phi.roll(2, axis))) * (ng / 12.0)
        flat = grad.reshape(-1)
        for a in corners:
            w, at = corner(*a)
            acc[:, axis] -= w * flat[at]
    return acc


def _density(pos, mass, h):
    """Cubic-spline density, all pairs within a slab of the largest smoothing length."""
    q = _grid(pos)
    n = q.shape[0]
    order = torch.argsort(q[:, 0])
    q, m, hs = q[order], mass[order], h.double()[order]
    x = q[:, 0].contiguous()
    rho = torch.zeros(n, dtype=torch.float64, device=q.device)
    rows = 512
    for b in range(0, n, rows):
        t, ht = q[b:b + rows], hs[b:b + rows]
        reach = int(float(ht.max()) * 4294967296.0) + 2
        lo, hi = int(t[0, 0]) - reach, int(t[-1, 0]) + reach
        if hi - lo >= 2 ** 32:
            src, ms = q, m
        else:
            edges = torch.tensor([lo, hi + 1, lo + 2 ** 32, hi + 1 - 2 ** 32], device=q.device)
            e = torch.searchsorted(x, edges).tolist()
            parts = [slice(e[0], e[1])]
            if lo < 0:
                parts.append(slice(e[2], n))
            if hi >= 2 ** 32:
                parts.append(slice(0, e[3]))
            src = torch.cat([q[p] for p in parts])
            ms = torch.cat([m[p] for p in parts])
        for c in range(0, src.shape[0], 16384):
            d = src[None, c:c + 16384] - t[:, None]
            d = (torch.remainder(d + 2 ** 31, 2 ** 32) - 2 ** 31).double() * 2.0 ** -32
            i, j = torch.nonzero((d * d).sum(2) < (ht * ht)[:, None], as_tuple=True)
            u = d[i, j].norm(dim=1) / ht[i]
            w = torch.where(u < 0.5, 1.0 - 6.0 * u ** 2 + 6.0 * u ** 3, 2.0 * (1.0 - u) ** 3)
            rho.index_add_(0, order[b + i], ms[c:c + 16384][j] * w * (8.0 / math.pi) / ht[i] ** 3)
    return rho


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve", "refit", "active"):
        return None
    n = case["n"]
    pos, mass, _ = _particles(n, case["dist"], case["masses"], seed)
    if kind == "pm":
        # the library's masses are 32-bit from here on
        return dict(acc=_mesh_force(pos, mass.float().double(), case["mesh"], case["rs_cells"] / n ** (1.0 / 3.0)))
    if n > DIRECT_MAX:
        return None
    if kind == "sph":
        return dict(rho=_density(pos, mass, _smoothing(pos, case["ngb"])), n_ngb=None)
    prm = _params(n, case["opening"], case["rs_cells"])
    acc, pot = _direct(pos, mass, prm, kind == "pot")
    out = dict(acc=acc)
    if kind == "pot":
        out["pot"] = pot
    if prm["opening"] == BH or case.get("a_old"):
        out.update(n_pp=None, n_pn=None)
    return out
