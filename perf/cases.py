"""Performance cases of the framework: the calls a simulation makes, over the range it makes them.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` others of
the same ranges; ``prepare`` makes what a program holds before the call (particles, buffers,
the context), ``run`` is one pass through the public entry points, ``work`` counts what a
pass cannot do without, and ``exact`` evaluates the same outputs in 64 bits with plain torch.

Particle sets are the synthetic ones of the package (uniform; half uniform and half in NFW
halos; a Zel'dovich-displaced grid with halos replacing grid particles), drawn on the GPU,
with distances in units of the box side ``L`` and the cutoff in mean particle spacings.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0910_0121_gb300 import greem, synth

CELLS = 1 << 21          # finest cells per axis


# --------------------------------------------------------------------------- the cases
def _force(name, pset, n, **kw):
    c = dict(op="force", set=pset, n=n, L=1.0, rc=3.0, theta=0.5, n_crit=64, n_leaf=10, eps=0.0, theta0=0.0,
             precision="f32", quad=False, species=1, keep_acc=True)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # A small box (16^3, the lower end of the batched workload): launches and latency; the
        # call allocates its result.
        _force("uniform_4k", "uniform", 16 ** 3, keep_acc=False),
        # The smallest configuration of the package, called in a loop with buffers that are kept.
        _force("uniform_32k", "uniform", 32 ** 3),
        # A ragged clustered set in a box whose side is no power of two: softened, two particle
        # masses, the distance-dependent opening angle (a zoom or a merger run).
        _force("ragged_100k", "nfw", 100003, L=100.0, eps=0.02, theta=0.7, theta0=0.25, n_crit=128, species=2),
        # The clustered 128^3 configuration.
        _force("nfw_128", "nfw", 128 ** 3),
        # The benchmark's configuration: 256^3, the step of a production run.
        _force("zel_256", "zel", 256 ** 3, n_crit=192),
        # Many independent boxes in one call (ensembles, parameter scans).
        dict(name="batched_64", op="batched", nbox=64, nlo=16 ** 3, nhi=96 ** 3, theta=0.5, n_crit=64),
        # The double-precision form: reference forces for accuracy studies.
        _force("f64_nfw_64", "nfw", 64 ** 3, precision="f64"),
        # Second-order terms at a wide opening angle: accurate forces at fewer interactions.
        _force("quad_1m", "nfw", 1000003, theta=0.7, n_crit=128, quad=True),
        # One whole TreePM time step of a 128^3 run: drift, force (PP + PM), kick, timestep.
        dict(name="treepm_step_128", op="step", set="zel", n=128 ** 3, L=1.0, rc=3.0, theta=0.5, n_crit=128, n_pm=128,
             assign="tsc", eps=0.05),
        # The mesh part alone at the benchmark's size (large-scale field, PM-only runs).
        dict(name="pm_256", op="pm", set="zel", n=256 ** 3, L=1.0, n_pm=256, rc=3.0, assign="tsc"),
        # Snapshots in host memory, streamed through the GPU one after another.
        dict(name="host_4x300k", op="host", set="nfw", nstep=4, n=300007, L=1.0, rc=3.0, theta=0.5, n_crit=96),
        # One process's part of an eight-process step: particles packed by destination, the
        # tree of its own particles, the local essential trees for the seven others.
        dict(name="domain_8x500k", op="domain", set="nfw", n=4000037, L=1.0, rc=3.0, theta=0.5, n_crit=64,
             grid="2x2x2", rank=0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above; about two in three are single-box FP32 forces, as in use."""
    kind = rng.choice(["force"] * 6 + ["batched", "f64", "quad", "step", "pm", "host", "domain"])
    theta = rng.choice([0.3, 0.5, 0.5, 0.5, 0.7])
    n_crit = rng.choice([32, 64, 64, 96, 128, 192])
    L = rng.choice([1.0, 1.0, 64.0, 100.0])
    pset = rng.choice(["uniform", "nfw", "nfw", "zel"])
    if kind == "force":
        n = _logint(rng, 4096, 6_000_000)
        if pset == "zel":
            n = max(16, round(n ** (1.0 / 3.0))) ** 3
        soft = rng.random() < 0.3
        return _force("", pset, n, L=L, rc=rng.choice([2.5, 3.0, 3.0, 3.5]), theta=theta, n_crit=n_crit,
                      eps=0.02 if soft else 0.0, theta0=rng.choice([0.0, 0.0, 0.0, 0.25]),
                      species=rng.choice([1, 1, 2]), keep_acc=rng.random() < 0.7)
    if kind == "batched":
        return dict(op="batched", nbox=rng.randint(2, 48), nlo=rng.randint(500, 4096), nhi=_logint(rng, 20000, 400000),
                    theta=theta, n_crit=n_crit)
    if kind == "f64":
        return _force("", rng.choice(["uniform", "nfw"]), _logint(rng, 4096, 200_000), L=L, theta=max(theta, 0.5),
                      n_crit=rng.choice([32, 64]), eps=rng.choice([0.0, 0.02]), precision="f64")
    if kind == "quad":
        return _force("", rng.choice(["uniform", "nfw"]), _logint(rng, 4096, 1_500_000), L=L,
                      theta=rng.choice([0.5, 0.7]), n_crit=n_crit, quad=True)
    if kind == "step":
        k = _logint(rng, 24, 144)
        return dict(op="step", set="zel", n=k ** 3, L=L, rc=3.0, theta=theta, n_crit=n_crit,
                    n_pm=max(16, k // rng.choice([2, 4]) * 2), assign=rng.choice(["tsc", "tsc", "cic"]), eps=0.05)
    if kind == "pm":
        k = _logint(rng, 32, 240)
        return dict(op="pm", set="zel", n=k ** 3, L=L, n_pm=rng.choice([32, 64, 96, 128, 192, 256]), rc=3.0,
                    assign=rng.choice(["tsc", "cic"]))
    if kind == "host":
        return dict(op="host", set=rng.choice(["uniform", "nfw"]), nstep=rng.randint(2, 6),
                    n=_logint(rng, 10000, 600_000), L=L, rc=3.0, theta=theta, n_crit=n_crit)
    return dict(op="domain", set=rng.choice(["uniform", "nfw"]), n=_logint(rng, 60_000, 4_000_000), L=1.0, rc=3.0,
                theta=theta, n_crit=n_crit, grid=rng.choice(["2x1x1", "2x2x1", "2x2x2", "3x2x2"]),
                rank=rng.randint(0, 1))


# --------------------------------------------------------------------------- particle sets
def _dev():
    return torch.device("cuda")


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) * 2654435761 % (1 << 62))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=_dev(), dtype=torch.float64)


def _halos(sizes, n_total, g):
    """Particles of NFW halos with the given sizes in a unit box of n_total particles."""
    sizes = torch.as_tensor(np.asarray(sizes, np.int64), device=_dev())
    nh = sizes.shape[0]
    centre = _rand(g, nh, 3)
    conc = 5.0 + 10.0 * _rand(g, nh)
    r200 = (3.0 * sizes.double() / n_total / (800.0 * math.pi)) ** (1.0 / 3.0)
    owner = torch.repeat_interleave(torch.arange(nh, device=_dev()), sizes)
    c = conc[owner]
    y = _rand(g, owner.shape[0]) * (torch.log1p(c) - c / (1.0 + c))
    lo, hi = torch.zeros_like(c), c.clone()
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        below = torch.log1p(mid) - mid / (1.0 + mid) < y
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    r = 0.5 * (lo + hi) * r200[owner] / c
    v = torch.randn(owner.shape[0], 3, generator=g, device=_dev(), dtype=torch.float64)
    v /= v.norm(dim=1, keepdim=True)
    return torch.remainder(centre[owner] + v * r[:, None], 1.0)


def _zeldovich(k, rms, g):
    """k^3 grid displaced by a Zel'dovich field with P(k) ~ k^-2, rms in grid spacings."""
    k1 = 2.0 * math.pi * torch.fft.fftfreq(k, d=1.0 / k, device=_dev(), dtype=torch.float64)
    kz = 2.0 * math.pi * torch.fft.rfftfreq(k, d=1.0 / k, device=_dev(), dtype=torch.float64)
    ks = (k1[:, None, None], k1[None, :, None], kz[None, None, :])
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    d = torch.randn(*k2.shape, 2, generator=g, device=_dev(), dtype=torch.float64)
    d = torch.view_as_complex(d) / torch.sqrt(k2)
    d[0, 0, 0] = 0.0
    psi = torch.stack([torch.fft.irfftn(1j * a * d / k2, s=(k, k, k)) for a in ks], dim=-1).reshape(-1, 3)
    psi *= (rms / k) / torch.sqrt((psi * psi).sum(1).mean())
    q = (torch.arange(k, device=_dev(), dtype=torch.float64) + 0.5) / k
    grid = torch.stack(torch.meshgrid(q, q, q, indexing="ij"), dim=-1).reshape(-1, 3)
    return torch.remainder(grid + psi, 1.0)


def _set(pset, n, seed):
    """Positions [n,3] in the unit box."""
    g, rng = _gen(seed), np.random.default_rng(seed)
    if pset == "uniform":
        return _rand(g, n, 3)
    nh = max(1, round(1000 * n / 128 ** 3))
    sizes = synth.powerlaw_sizes(nh, rng, hi=min(1e5, max(200.0, n / 20.0)))
    if pset == "nfw":
        return torch.cat([_rand(g, n - n // 2, 3), _halos(synth.integer_sizes(sizes, n // 2), n, g)])
    k = round(n ** (1.0 / 3.0))
    pos = _zeldovich(k, 0.5, g)
    halo = _halos(synth.integer_sizes(sizes, n // 4), n, g)
    pos[torch.randperm(n, generator=g, device=_dev())[: halo.shape[0]]] = halo
    return pos


def _particles(case, seed, n=None):
    n = case["n"] if n is None else n
    pos = (_set(case["set"], n, seed) * case["L"]).contiguous()
    mass = torch.full((n,), 1.0 / n, device=_dev(), dtype=torch.float32)
    if case.get("species", 1) == 2:  # every eighth particle eight times heavier
        mass[::8] *= 8.0
    return pos, mass


def _spacing(case, n=None):
    return case["L"] / (case["n"] if n is None else n) ** (1.0 / 3.0)


def _params(case, n=None, **kw):
    sp = _spacing(case, n)
    flags = 0
    if case.get("theta0", 0.0):
        flags |= greem.FLAG_THETA_EQ12
        kw["theta0"] = case["theta0"]
    if case.get("quad"):
        flags |= greem.FLAG_QUADRUPOLE
    if case["op"] == "step":
        flags |= greem.FLAG_ADD_PM
        kw.update(n_pm=case["n_pm"], assign=_scheme(case))
    return greem.params(L=case["L"], r_cut=case["rc"] * sp, theta=case["theta"], n_crit=case["n_crit"],
                        n_leaf=case.get("n_leaf", 10), eps=case.get("eps", 0.0) * sp,
                        precision=greem.F64 if case.get("precision") == "f64" else greem.F32_REL, flags=flags, **kw)


def _scheme(case):
    return greem.ASSIGN_TSC if case["assign"] == "tsc" else greem.ASSIGN_CIC


def _box_sizes(case):
    rng = np.random.default_rng(case["nbox"] * 7919 + case["nhi"])
    return np.rint(np.exp(rng.uniform(math.log(case["nlo"]), math.log(case["nhi"]), case["nbox"]))).astype(np.int64)


def _boxes_of(case, seed):
    """The batched boxes: (positions, masses, offsets, per-box cases)."""
    nb = _box_sizes(case)
    sub = [dict(op="force", set="nfw", n=int(n), L=1.0, rc=3.0, theta=case["theta"], n_crit=case["n_crit"])
           for n in nb]
    parts = [_particles(c, seed * 1009 + b) for b, c in enumerate(sub)]
    off = np.zeros(len(nb) + 1, np.int64)
    off[1:] = np.cumsum(nb)
    return torch.cat([p for p, _ in parts]), torch.cat([m for _, m in parts]), off, sub


def _momenta(case, n, seed):
    """Velocities that move a particle about a tenth of a spacing per unit time."""
    return (0.1 * _spacing(case) * torch.randn(n, 3, generator=_gen(seed + 77), device=_dev())).contiguous()


def _domain_set(case, seed):
    """The boxes of a decomposition and the particles of one of them, after a drift that has
    carried some across its faces: (boxes int32 [ndom,6], pos, mass, ids).  How many items go
    where depends on the positions alone, so the set of positions belongs to the case; the
    seed draws the masses and where in the set the process's order starts."""
    pos, _ = _particles(case, case["n"])
    cells = (pos * (CELLS / case["L"])).long().clamp_(0, CELLS - 1).int()
    grid = [int(v) for v in case["grid"].split("x")]
    rng = np.random.default_rng(case["n"])
    pick = torch.from_numpy(np.sort(rng.choice(case["n"], max(64, case["n"] // 2500), replace=False))).to(_dev())
    boxes = greem.domain_boxes(cells[pick].cpu().numpy(), grid)
    b = torch.from_numpy(boxes[case["rank"]]).to(_dev())
    mine = ((cells >= b[0::2]) & (cells < b[1::2])).all(1).nonzero()[:, 0]
    pos = torch.remainder(pos[mine] + 0.1 * _spacing(case) * torch.randn(
        mine.shape[0], 3, generator=_gen(case["n"] + 78), device=_dev(), dtype=torch.float64), case["L"])
    turn = int(np.random.default_rng(seed).integers(1, mine.shape[0]))
    pos, ids = torch.roll(pos, turn, 0), torch.roll(mine, turn, 0)
    mass = (0.5 + torch.rand(mine.shape[0], generator=_gen(seed), device=_dev())) / case["n"]
    return boxes, pos.contiguous(), mass.contiguous(), ids.contiguous()


# --------------------------------------------------------------------------- the calls
F_KICK, F_DRIFT = 0.25, 0.5


def prepare(case, seed):
    op = case["op"]
    st = dict(case=case)
    if op == "host":
        sets = [_particles(case, seed * 31 + k) for k in range(case["nstep"])]
        st["pos"] = [p.cpu().pin_memory() for p, _ in sets]
        st["mass"] = [m.cpu().pin_memory() for _, m in sets]
        st["acc"] = [torch.empty(case["n"], 3).pin_memory() for _ in sets]
        st["p"] = _params(case)
    elif op == "batched":
        st["pos"], st["mass"], st["off"], sub = _boxes_of(case, seed)
        st["p"] = [_params(c) for c in sub]
        st["acc"] = torch.empty_like(st["pos"], dtype=torch.float32)
    elif op == "domain":
        st["boxes"], st["pos"], st["mass"], st["ids"] = _domain_set(case, seed)
        st["p"] = _params(case)
    else:
        st["pos"], st["mass"] = _particles(case, seed)
        dt = torch.float64 if case.get("precision") == "f64" else torch.float32
        st["acc"] = torch.empty_like(st["pos"], dtype=dt) if case.get("keep_acc", True) else None
        if op == "step":
            st["vel"] = _momenta(case, case["n"], seed)
            st["pos1"], st["vel1"] = torch.empty_like(st["pos"]), torch.empty_like(st["vel"])
        if op != "pm":
            st["p"] = _params(case)
    st["ctx"] = greem.Context()
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    op = case["op"]
    if op == "force":
        return ctx.short_force(st["pos"], st["mass"], st["p"], st["acc"])
    if op == "batched":
        return ctx.short_force_batched(st["pos"], st["mass"], st["off"], st["p"], st["acc"])
    if op == "pm":
        return ctx.pm_force(st["pos"], st["mass"], case["L"], case["n_pm"], case["rc"] * _spacing(case), _scheme(case),
                            st["acc"])
    if op == "host":
        return ctx.short_force_host(st["pos"], st["mass"], st["p"], st["acc"])
    if op == "step":  # the state before the step is kept
        pos, vel = st["pos1"].copy_(st["pos"]), st["vel1"].copy_(st["vel"])
        ctx.drift(pos, vel, case["L"], F_DRIFT)
        acc = ctx.short_force(pos, st["mass"], st["p"], st["acc"])
        ctx.kick(vel, acc, F_KICK)
        dt = ctx.timestep(vel, acc, case["eps"] * _spacing(case), 0.1)
        return dict(pos=pos, vel=vel, acc=acc, dt=dt)
    # domain: the particles that stay are this process's share of the packed ones
    po, mo, io, counts = ctx.domain_pack(st["pos"], st["mass"], st["ids"], case["L"], st["boxes"])
    b = int(counts[: case["rank"]].sum())
    e = b + int(counts[case["rank"]])
    ctx.build_tree(po[b:e], mo[b:e], st["p"])
    lp, lm, _, lc = ctx.let_export(st["boxes"], case["rank"])
    return dict(pos=po, mass=mo, ids=io, counts=counts, let_pos=lp, let_mass=lm, let_counts=lc)


def work(case):
    """Each input read once, each output written once; the operations of Eq. 1-2 (42 a pair)
    over the particles within r_cut at the mean density, and of the mesh part's transforms."""
    op = case["op"]

    def pairs(n, rc):
        return n * 4.0 / 3.0 * math.pi * rc ** 3

    if op == "batched":
        n = case["nbox"] * (case["nhi"] - case["nlo"]) / math.log(case["nhi"] / case["nlo"])
        return dict(bytes=40.0 * n, flops=42.0 * pairs(n, 3.0))
    n = float(case["n"])
    mesh = 0.0
    if op in ("pm", "step"):
        g = float(case["n_pm"]) ** 3
        mesh = 4 * 2.5 * g * math.log2(g) + n * 4 * 2 * (27 if case["assign"] == "tsc" else 8)
    if op == "force":
        return dict(bytes=(28.0 + (24 if case["precision"] == "f64" else 12)) * n, flops=42.0 * pairs(n, case["rc"]))
    if op == "pm":
        return dict(bytes=40.0 * n, flops=mesh)
    if op == "step":  # and the state copied and moved: positions and velocities in and out
        return dict(bytes=(40.0 + 72.0) * n, flops=42.0 * pairs(n, case["rc"]) + mesh)
    if op == "host":
        return dict(bytes=40.0 * n * case["nstep"], flops=42.0 * pairs(n, case["rc"]) * case["nstep"])
    ndom = math.prod(int(v) for v in case["grid"].split("x"))
    return dict(bytes=72.0 * n / ndom, flops=0.0)


# --------------------------------------------------------------------------- exact values
# The method as the header states it, in 64-bit torch: the tree over Morton-sorted particles,
# the groups, the opening test on exact integer cells, Eq. 1-2 over every entry.
P22, H21 = 1 << 22, 1 << 21


def _wrap(x, L):
    r = x - L * torch.floor(x / L)
    r = torch.where(r < 0, r + L, r)
    r = torch.where(r >= L, r - L, r)
    return torch.where((r >= 0) & (r < L), r, torch.zeros_like(r))


def _cell(r, L):
    return torch.floor((r / L) * float(CELLS)).long().clamp_(0, CELLS - 1)


def _spread(v):
    for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F), (4, 0x10C30C30C30C30C3),
                 (2, 0x1249249249249249)):
        v = (v | (v << s)) & m
    return v


def _expand(start, count):
    """Row index and element index of the concatenated ranges [start, start + count)."""
    row = torch.repeat_interleave(torch.arange(start.shape[0], device=start.device), count)
    first = torch.cumsum(count, 0) - count
    return row, start[row] + torch.arange(row.shape[0], device=start.device) - first[row]


class _Tree:
    def __init__(self, pos, mass, L, r_cut, n_leaf, n_crit):
        w = _wrap(pos, L)
        cell = _cell(w, L)
        key = (_spread(cell[:, 0]) << 2) | (_spread(cell[:, 1]) << 1) | _spread(cell[:, 2])
        key, self.perm = torch.sort(key, stable=True)
        self.x, self.m, self.cell = w[self.perm], mass[self.perm].double(), cell[self.perm]
        self.L, self.r_cut, self.u = L, r_cut, L / float(P22)
        n = key.shape[0]
        dev = key.device
        self.lmin = next(k for k in range(22) if L * 2.0 ** -k < 0.5 * L - r_cut)
        self.lv, groups = [], []
        b, e = torch.zeros(1, dtype=torch.long, device=dev), torch.full((1,), n, dtype=torch.long, device=dev)
        free = torch.ones(1, dtype=torch.bool, device=dev)
        for k in range(22):
            cnt = e - b
            split = (cnt >= n_leaf) | (k < self.lmin) if k < 21 else torch.zeros_like(free)
            lev = dict(b=b, e=e, leaf=~split, c=(2 * (self.cell[b] >> (21 - k)) + 1) << (21 - k))
            self.lv.append(lev)
            g = free & ((cnt <= n_crit) | ~split) if k >= self.lmin else torch.zeros_like(free)
            gi = g.nonzero()[:, 0]
            groups.append((b[gi], e[gi], lev["c"][gi], torch.full_like(b[gi], 1 << (21 - k))))
            si = split.nonzero()[:, 0]
            if si.numel() == 0:
                break
            row, idx = _expand(b[si], cnt[si])
            pre = key[idx] >> (60 - 3 * k)
            head = torch.ones_like(pre, dtype=torch.bool)
            head[1:] = (pre[1:] != pre[:-1]) | (row[1:] != row[:-1])
            hb = head.nonzero()[:, 0]
            nb, par = idx[hb], row[hb]
            ne = torch.cat([idx[hb[1:] - 1] + 1, idx[-1:] + 1])
            lev["nchild"] = torch.zeros_like(b).index_copy_(0, si, torch.bincount(par, minlength=si.numel()))
            lev["child"] = torch.cumsum(lev["nchild"], 0) - lev["nchild"]
            free = (free & ~g)[si][par]
            b, e = nb, ne
        gb, ge, gc, gh = (torch.cat([g[i] for g in groups]) for i in range(4))
        o = torch.argsort(gb)
        self.gb, self.ge, self.gc, self.gh = gb[o], ge[o], gc[o], gh[o]
        below = None
        for lev in reversed(self.lv):  # moments, bottom up
            self._moments(lev, below)
            below = lev

    def _moments(self, lev, below):
        nn = lev["b"].shape[0]
        dev = lev["b"].device
        cen = lev["c"].double() * self.u
        M, D = torch.zeros(nn, dtype=torch.float64, device=dev), torch.zeros(nn, 3, dtype=torch.float64, device=dev)
        Q = torch.zeros(nn, 6, dtype=torch.float64, device=dev)
        li = lev["leaf"].nonzero()[:, 0]
        row, j = _expand(lev["b"][li], (lev["e"] - lev["b"])[li])
        parts = [(li[row], self.m[j], self.x[j], None)]
        if below is not None:
            par = torch.repeat_interleave(torch.arange(nn, device=dev), lev["nchild"])
            parts.append((par, below["M"], below["com"], below["Q"]))
        for row, m, x, _ in parts:
            M.index_add_(0, row, m)
            D.index_add_(0, row, m[:, None] * (x - cen[row]))
        com = cen + D / M[:, None]
        for row, m, x, q in parts:
            s = x - com[row]
            t = m[:, None] * torch.stack([s[:, 0] * s[:, 0], s[:, 1] * s[:, 1], s[:, 2] * s[:, 2], s[:, 0] * s[:, 1],
                                          s[:, 0] * s[:, 2], s[:, 1] * s[:, 2]], 1)
            Q.index_add_(0, row, t if q is None else t + q)
        lev["M"], lev["com"], lev["Q"] = M, com, Q


def _g(R):
    """Eq. 2, both branches as printed."""
    inner = 1.0 - (224.0 * R ** 3 - 224.0 * R ** 5 + 70.0 * R ** 6 + 48.0 * R ** 7 - 21.0 * R ** 8) / 140.0
    outer = 1.0 - (12.0 - 224.0 * R ** 2 + 896.0 * R ** 3 - 840.0 * R ** 4 + 224.0 * R ** 5 + 70.0 * R ** 6 -
                   48.0 * R ** 7 + 7.0 * R ** 8) / 140.0
    return torch.where(R < 1.0, inner, torch.where(R < 2.0, outer, torch.zeros_like(R)))


def _theta2(sd, theta, theta0, u_over_eta):
    if not theta0:
        return theta * theta
    R = torch.sqrt(sd.double()) * u_over_eta
    rg = R * _g(R)
    t2 = torch.where(rg > 0, theta0 * theta0 / rg.clamp_min(1e-300), torch.full_like(rg, theta * theta))
    return t2.clamp_max(theta * theta)


def _half_wrap(d):
    return torch.where(d >= H21, d - P22, torch.where(d < -H21, d + P22, d))


def _walk(t, cen, half, bc, bh, theta, theta0):
    """The entries of every receiver: opening tests against (cen, half), pruning against the
    box (bc, bh), in u.  Returns the accepted nodes (receiver, first particle, centre of mass,
    mass, second moments) and the particles of opened leaves (receiver, particle)."""
    G = cen.shape[0]
    dev = cen.device
    uu, rc2 = t.u * t.u, t.r_cut * t.r_cut
    g = torch.arange(G, device=dev)
    nd = torch.zeros(G, dtype=torch.long, device=dev)
    nodes, leaves = [], []
    for k, lev in enumerate(t.lv):
        hn = 1 << (21 - k)
        d = _half_wrap(lev["c"][nd] - cen[g])
        gap = ((d - (bc - cen)[g]).abs() - hn - bh[g]).clamp_min_(0)
        keep = ~((gap * gap).sum(1).double() * uu > rc2)
        g, nd, d = g[keep], nd[keep], d[keep]
        e = (d.abs() - half[g]).clamp_min_(0)
        sd = (e * e).sum(1)
        acc = torch.zeros_like(keep[: g.shape[0]])
        if k >= t.lmin:
            acc = float((2 * hn) ** 2) < _theta2(sd, theta, theta0, t.u / (0.5 * t.r_cut)) * sd.double()
        nodes.append((g[acc], lev["b"][nd[acc]], lev["com"][nd[acc]], lev["M"][nd[acc]], lev["Q"][nd[acc]]))
        op = ~acc
        g, nd, d = g[op], nd[op], d[op]
        lf = lev["leaf"][nd]
        row, j = _expand(lev["b"][nd[lf]], (lev["e"] - lev["b"])[nd[lf]])
        if row.numel():
            gl = g[lf][row]
            # a group's entries keep the leaf's image; a domain box takes each particle's nearest
            dj = d[lf][row] + (2 * t.cell[j] + 1 - lev["c"][nd[lf]][row])
            dj = _half_wrap(dj) if bc is cen else dj - (bc - cen)[gl]
            dj = (dj.abs() - 1 - bh[gl]).clamp_min_(0)
            kp = ~((dj * dj).sum(1).double() * uu > rc2)
            leaves.append((gl[kp], j[kp]))
        g, nd = g[~lf], nd[~lf]
        if g.numel() == 0:
            break
        row, ch = _expand(lev["child"][nd], lev["nchild"][nd])
        g, nd = g[row], ch
    lg, lj = (torch.cat([v[i] for v in leaves]) if leaves else g[:0] for i in range(2))
    return [torch.cat([v[i] for v in nodes]) for i in range(5)] + [lg, lj]


def _pair(d, m, q, eta, eps):
    """Eq. 1 (and the second-order terms for entries with moments) summed over the last axis."""
    r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    r = torch.sqrt(r2)
    R = r / eta
    v, w = (2.0 - R).clamp_min_(0), (1.0 - R).clamp_min_(0)
    # Eq. 2 factored at its zeros, without the cancellation of the printed form
    pc, pp = ((7.0 * R + 22.0) * R + 10.0) * R + 4.0, (7.0 * R + 18.0) * R + 3.0
    g = v ** 5 * pc / 140.0 + w ** 6 * pp / 35.0
    s2 = r2 + eps * eps
    zero = r2 == 0
    f = torch.where(zero, torch.zeros_like(r2), m * g / (s2 * torch.sqrt(s2)))
    out = [f * d[c] for c in range(3)]
    if q is not None:
        dpc, dpp = (21.0 * R + 44.0) * R + 10.0, 14.0 * R + 18.0
        g1 = (v ** 5 * dpc - 5.0 * v ** 4 * pc) / 140.0 + (w ** 6 * dpp - 6.0 * w ** 5 * pp) / 35.0
        g2 = (v ** 5 * (42.0 * R + 44.0) - 10.0 * v ** 4 * dpc + 20.0 * v ** 3 * pc) / 140.0 + \
             (w ** 6 * 14.0 - 12.0 * w ** 5 * dpp + 30.0 * w ** 4 * pp) / 35.0
        g1, g2 = g1 / eta, g2 / (eta * eta)
        B = torch.where(zero, torch.zeros_like(r), g1 / r ** 4 - 3.0 * g / r ** 5)
        C = torch.where(zero, torch.zeros_like(r), g2 / r ** 5 - 7.0 * g1 / r ** 6 + 15.0 * g / r ** 7)
        Qd = [q[0] * d[0] + q[3] * d[1] + q[4] * d[2], q[3] * d[0] + q[1] * d[1] + q[5] * d[2],
              q[4] * d[0] + q[5] * d[1] + q[2] * d[2]]
        a = 0.5 * B * (q[0] + q[1] + q[2]) + 0.5 * C * (d[0] * Qd[0] + d[1] * Qd[1] + d[2] * Qd[2])
        out = [out[c] + a * d[c] + B * Qd[c] for c in range(3)]
    return [o.sum(-1) for o in out]


def _exact_force(case, pos, mass):
    L, rc = case["L"], case["rc"] * _spacing(case)
    eps, theta, theta0 = case.get("eps", 0.0) * _spacing(case), case["theta"], case.get("theta0", 0.0)
    t = _Tree(pos, mass, L, rc, case.get("n_leaf", 10), case["n_crit"])
    ng = t.gb.shape[0]
    n = pos.shape[0]
    dev = pos.device
    gid = torch.repeat_interleave(torch.arange(ng, device=dev), t.ge - t.gb)[:, None].expand(n, 3)
    lo = torch.full((ng, 3), CELLS, dtype=torch.long, device=dev).scatter_reduce_(0, gid, t.cell, "amin")
    hi = torch.full((ng, 3), -1, dtype=torch.long, device=dev).scatter_reduce_(0, gid, t.cell, "amax")
    acc = torch.zeros(n, 3, dtype=torch.float64, device=dev)
    step = 16384
    for g0 in range(0, ng, step):
        s = slice(g0, min(ng, g0 + step))
        G = s.stop - g0
        gn, _, gx, gm, gq, lg, lj = _walk(t, t.gc[s], t.gh[s][:, None], (lo + hi + 1)[s], (hi - lo + 1)[s], theta,
                                          theta0)
        quad = bool(case.get("quad"))
        for sets in ((gn, gx, gm, gq if quad else None), (lg, t.x[lj], t.m[lj], None)):
            o = torch.argsort(sets[0], stable=True)
            x, m = sets[1][o].T.contiguous(), sets[2][o]
            q = None if sets[3] is None else sets[3][o].T.contiguous()
            ln = torch.bincount(sets[0], minlength=G)
            _group_sums(t, acc, s, ln, x, m, q, 0.5 * rc, eps)
    out = torch.empty_like(acc)
    out[t.perm] = acc
    return out


def _group_sums(t, acc, s, ln, x, m, q, eta, eps):
    """acc += the force of each group's entries, by dense tiles of groups of like sizes."""
    if m.numel() == 0:
        return
    first = torch.cumsum(ln, 0) - ln
    nb = (t.ge - t.gb)[s]
    key = torch.ceil(torch.log2(nb.double()) * 2).long() * (1 << 40) + ln
    order = torch.argsort(key)
    nbo, lno = nb[order].tolist(), ln[order].tolist()
    a = 0
    while a < len(nbo):
        b, nm, lm = a, 0, 0
        while b < len(nbo):
            n2, l2 = max(nm, nbo[b]), max(lm, lno[b])
            if b > a and (b + 1 - a) * n2 * l2 > (1 << 24):
                break
            nm, lm, b = n2, l2, b + 1
        gi = order[a:b]
        a = b
        if lm == 0:
            continue
        li = torch.arange(lm, device=m.device)
        ok = li < ln[gi][:, None]
        e = torch.where(ok, first[gi][:, None] + li, torch.zeros_like(li))
        ii = torch.arange(nm, device=m.device)
        iok = ii < nb[gi][:, None]
        i = torch.where(iok, t.gb[s][gi][:, None] + ii, t.gb[s][gi][:, None])
        d = []
        for c in range(3):
            dc = x[c][e][:, None, :] - t.x[i, c][:, :, None]
            d.append(dc - t.L * torch.round(dc / t.L))
        qe = None if q is None else [(q[c][e] * ok)[:, None, :] for c in range(6)]
        f = _pair(d, (m[e] * ok)[:, None, :], qe, eta, eps)
        for c in range(3):
            acc[:, c].index_add_(0, i[iok], f[c][iok])


def _mesh_weights(s, tsc):
    if not tsc:
        i = torch.floor(s)
        f = s - i
        return [i.long(), i.long() + 1], [1.0 - f, f]
    i = torch.floor(s + 0.5)
    d = s - i
    i = i.long()
    return [i - 1, i, i + 1], [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]


def _exact_pm(pos, mass, L, n, r_cut, tsc):
    """Assignment, Green's function of the complement of Eq. 2, spectral gradient, interpolation."""
    dev = pos.device
    dl = L / n
    s = _wrap(pos, L) / dl
    axes = [_mesh_weights(s[:, c], tsc) for c in range(3)]
    pts = [(((a % n) * n + b % n) * n + c % n, wa * wb * wc) for a, wa in zip(*axes[0]) for b, wb in zip(*axes[1])
           for c, wc in zip(*axes[2])]
    rho = torch.zeros(n ** 3, dtype=torch.float64, device=dev)
    for i, w in pts:
        rho.index_add_(0, i, mass.double() * w)
    rk = torch.fft.rfftn(rho.view(n, n, n) / dl ** 3)
    k1 = 2.0 * math.pi * torch.fft.fftfreq(n, d=dl, device=dev, dtype=torch.float64)
    kz = 2.0 * math.pi * torch.fft.rfftfreq(n, d=dl, device=dev, dtype=torch.float64)
    ks = [k1[:, None, None], k1[None, :, None], kz[None, None, :]]
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    xi = torch.sqrt(k2) * (0.5 * r_cut)
    big = xi.clamp_min(1e-2)
    S = torch.where(xi < 1e-2, 1.0 - xi * xi / 15.0 + xi ** 4 / 560.0,
                    12.0 * (2.0 - 2.0 * torch.cos(big) - big * torch.sin(big)) / big ** 4)
    W = 1.0
    for a in ks:
        W = W * torch.sinc(a * dl / (2.0 * math.pi)) ** (3 if tsc else 2)
    k2[0, 0, 0] = 1.0
    G = -4.0 * math.pi * S * S / (k2 * W * W)
    G[0, 0, 0] = 0.0
    phi = G * rk
    acc = torch.zeros_like(pos)
    for c in range(3):
        ka = torch.where((ks[c].abs() * dl - math.pi).abs() < 1e-9, torch.zeros_like(ks[c]), ks[c])
        grid = torch.fft.irfftn(-1j * ka * phi, s=(n, n, n)).reshape(-1)
        for i, w in pts:
            acc[:, c] += w * grid[i]
    return acc


def _exact_domain(case, seed):
    boxes, pos, mass, ids = _domain_set(case, seed)
    L, rank = case["L"], case["rank"]
    w = _wrap(pos, L)
    cell = _cell(w, L)
    bx = torch.from_numpy(boxes.astype(np.int64)).to(pos.device)
    dom = torch.full((pos.shape[0],), -1, dtype=torch.long, device=pos.device)
    for d in range(bx.shape[0]):
        dom[((cell >= bx[d, 0::2]) & (cell < bx[d, 1::2])).all(1)] = d
    _, o = torch.sort(dom, stable=True)
    counts = torch.bincount(dom, minlength=bx.shape[0])
    mine = (dom == rank).nonzero()[:, 0]
    t = _Tree(w[mine], mass[mine], L, case["rc"] * _spacing(case), 10, case["n_crit"])
    cen, half = bx[:, 0::2] + bx[:, 1::2], bx[:, 1::2] - bx[:, 0::2]
    g, b, x, m, _, lg, lj = _walk(t, cen, half, cen, half, case["theta"], 0.0)
    rows = [torch.cat(v) for v in ((g, lg), (b, lj), (x, t.x[lj]), (m, t.m[lj]))]
    rows = [v[rows[0] != rank] for v in rows]
    k = torch.argsort(rows[0] * (1 << 32) + rows[1])
    lc = torch.bincount(rows[0], minlength=bx.shape[0])
    return dict(pos=w[o], mass=mass[o].double(), ids=ids[o], counts=counts.cpu().numpy(), let_pos=rows[2][k],
                let_mass=rows[3][k], let_counts=lc.cpu().numpy())


def exact(case, seed):
    op = case["op"]
    if op == "domain":
        return _exact_domain(case, seed)
    if op == "host":
        return [_exact_force(case, *_particles(case, seed * 31 + k)).cpu() for k in range(case["nstep"])]
    if op == "batched":
        pos, mass, off, sub = _boxes_of(case, seed)
        return torch.cat([_exact_force(c, pos[a:b], mass[a:b]) for c, a, b in zip(sub, off[:-1], off[1:])])
    pos, mass = _particles(case, seed)
    if op == "force":
        return _exact_force(case, pos, mass)
    rc = case["rc"] * _spacing(case)
    if op == "pm":
        return _exact_pm(pos, mass, case["L"], case["n_pm"], rc, case["assign"] == "tsc")
    vel = _momenta(case, case["n"], seed)
    p1 = _wrap(pos + F_DRIFT * vel.double(), case["L"])
    acc = _exact_force(case, p1, mass)
    acc += _exact_pm(p1, mass, case["L"], case["n_pm"], rc, case["assign"] == "tsc")
    v1 = vel.double() + F_KICK * acc
    eps = case["eps"] * _spacing(case)
    dt = 0.1 * min(math.sqrt(eps / float(acc.norm(dim=1).max())), eps / float(v1.norm(dim=1).max()))
    return dict(pos=p1, vel=v1, acc=acc, dt=dt)
