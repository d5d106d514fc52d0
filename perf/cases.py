"""What a user of this framework has it do, as cases that can be timed.

Every case is one pass of the force path through the Python entry points: a
whole step (tree build, mesh where there is one, forces, release) on particles
that just moved, or forces on some of the particles of a resident tree.  The
sizes and parameters are those of the repository's workloads (Plummer 8192,
Hernquist 2^20, the periodic Zel'dovich box, two species, time bins, served
systems) and sizes between and below them, odd ones among them.  The particles
are drawn on the device from the seed; |a| of the previous step, which the
relative criterion needs, is the closed form of the profile (the linear-theory
acceleration in the periodic box), so that it does not depend on the code that
is measured.
"""
import math

import numpy as np
import torch

import paper_1909_04667_gb300 as tpm

DEV = "cuda:0"

# Interactions per particle of the per-particle walk (particle-node plus
# particle-particle, rounded means of the counts that the force call returns),
# for the work of a case: relative criterion at the parameters below, geometric
# criterion at theta = 0.7 (it grows as theta^-3).  "dense" is the part of a
# halo that short time steps select.
INTERACTIONS = {"hernquist/rel": 720, "hernquist/bh": 810, "plummer/rel": 850, "plummer/bh": 580, "dense/rel": 1490,
                "dense/bh": 1100, "two/rel": 735, "two/bh": 800, "iso/rel": 680, "iso/bh": 700, "box/rel": 90,
                "box/bh": 73, "ewald/rel": 3500, "ewald/bh": 270}


def listed():
    return [
        # a small isolated system, the geometric criterion of a first force: launches and latency count
        dict(name="plummer_8192", kind="step", profile="plummer", n=8192, crit="bh", theta=0.7, bucket=8),
        # the main workload: one step of a 2^20 halo, everything active, |a| of the last step at hand
        dict(name="hernquist_1m", kind="step", profile="hernquist", n=1 << 20, crit="rel", alpha=0.0025, bucket=16),
        # a program that keeps its particles in page-locked host arrays, first force, a ragged size
        dict(name="hernquist_300k_host", kind="host", profile="hernquist", n=300007, crit="bh", theta=0.5, bucket=8),
        # the cosmological box: short-range walk and mesh
        dict(name="box_128", kind="box", ngrid=128, pm_n=256, grad="fd4", crit="rel", alpha=0.005, bucket=8),
        # a small box with the spectral mesh gradient, first force
        dict(name="box_40_spectral", kind="box", ngrid=40, pm_n=64, grad="ik", crit="bh", theta=0.5, bucket=8),
        # the same kind of box without a mesh: the Ewald-corrected tree
        dict(name="box_32_ewald", kind="ewald", ngrid=32, crit="rel", alpha=0.005, bucket=8),
        # an isolated halo with the zero-padded mesh
        dict(name="hernquist_500k_mesh", kind="iso", profile="hernquist", n=500009, pm_n=64, asmth=2.5, crit="rel",
             alpha=0.0025, bucket=16),
        # halo and stars, each with its own softening
        dict(name="two_species", kind="step", profile="two", n=(1 << 20) + (1 << 18), crit="rel", alpha=0.0025,
             bucket=16),
        # a served request: a few particles, anywhere in a resident tree
        dict(name="active_1000", kind="active", profile="hernquist", n=1 << 20, active=1000, crit="rel",
             alpha=0.0025, bucket=16),
        # a local time step: the particles due at a tick, a new tree, their forces
        dict(name="substep", kind="substep", profile="hernquist", n=1 << 20, tick=8, crit="rel", alpha=0.0025,
             bucket=16),
        # time-bin requests of many substeps on one tree, in one batched call
        dict(name="timebin_batch", kind="timebins", profile="hernquist", n=1 << 20, ids=1 << 20, crit="rel",
             alpha=0.0025, bucket=16),
        # a round of a force server: requests on several resident systems in one batched call
        dict(name="served_round", kind="round", systems=12, nmin=1 << 12, nmax=1 << 17, crit="rel", alpha=0.0025,
             bucket=8),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the ranges above."""
    kind = rng.choice(["step", "step", "two", "host", "box", "ewald", "iso", "active", "substep", "timebins", "round"])
    bucket = rng.choice([4, 8, 16])
    crit = dict(crit="rel", alpha=0.0025) if rng.random() < 0.6 else dict(crit="bh", theta=rng.choice([0.5, 0.6, 0.7]))
    if kind == "step":
        return dict(kind="step", profile=rng.choice(["plummer", "hernquist"]), n=_logint(rng, 4096, 900000),
                    bucket=bucket, **crit)
    if kind == "two":
        return dict(kind="step", profile="two", n=_logint(rng, 8192, 900000), bucket=bucket, **crit)
    if kind == "host":
        return dict(kind="host", profile=rng.choice(["plummer", "hernquist"]), n=_logint(rng, 4096, 500000),
                    bucket=bucket, **crit)
    if kind == "box":
        ngrid = rng.randint(20, 120)
        pm_n = 32
        while pm_n * 1.5 < ngrid * 2:  # the power of two nearest to two mesh points per mean spacing
            pm_n *= 2
        crit = dict(crit="rel", alpha=0.005) if rng.random() < 0.6 else dict(crit="bh", theta=0.5)
        return dict(kind="box", ngrid=ngrid, pm_n=pm_n, grad=rng.choice(["fd4", "ik"]), bucket=bucket, **crit)
    if kind == "ewald":
        crit = dict(crit="rel", alpha=0.005) if rng.random() < 0.6 else dict(crit="bh", theta=rng.choice([0.5, 0.7]))
        return dict(kind="ewald", ngrid=rng.randint(14, 30), bucket=bucket, **crit)
    if kind == "iso":
        return dict(kind="iso", profile=rng.choice(["plummer", "hernquist"]), n=_logint(rng, 16384, 600000),
                    pm_n=rng.choice([32, 64, 128]), asmth=rng.choice([1.25, 2.5]), bucket=bucket, **crit)
    if kind == "active":
        n = _logint(rng, 16384, 1 << 20)
        return dict(kind="active", profile=rng.choice(["plummer", "hernquist"]), n=n,
                    active=_logint(rng, 64, n // 2), bucket=bucket, **crit)
    if kind == "substep":
        return dict(kind="substep", profile="hernquist", n=_logint(rng, 32768, 900000), tick=rng.choice([4, 8, 16, 32, 64]),
                    bucket=bucket, **crit)
    if kind == "timebins":
        n = _logint(rng, 65536, 900000)
        return dict(kind="timebins", profile="hernquist", n=n, ids=_logint(rng, n // 8, n), bucket=bucket, **crit)
    return dict(kind="round", systems=rng.randint(3, 24), nmin=1 << 12, nmax=_logint(rng, 1 << 14, 1 << 17),
                bucket=bucket, **crit)


# ---------------------------------------------------------------- inputs
def _gen(seed, k=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + k)
    return g


def _directions(n, g):
    d = torch.randn(n, 3, dtype=torch.float64, device=DEV, generator=g)
    return d / torch.linalg.vector_norm(d, dim=1, keepdim=True).clamp_min(1e-300)


def _particles(profile, n, seed, k=0):
    """Positions, masses, |a| of the last step and (two species) softening
    supports of n particles; total mass and scale radius 1."""
    g = _gen(seed, k)
    u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g)
    hs = None
    if profile == "plummer":
        r = 1.0 / torch.sqrt(u.clamp(1e-15, 1.0 - 1e-15) ** (-2.0 / 3.0) - 1.0)
        a = r * (1.0 + r * r) ** -1.5
        mass = torch.full((n,), 1.0 / n, dtype=torch.float32, device=DEV)
    elif profile == "hernquist":
        rs = torch.sqrt(u) * (100.0 / 101.0)
        r = rs / (1.0 - rs)
        a = (101.0 / 100.0) ** 2 / (1.0 + r) ** 2
        mass = torch.full((n,), 1.0 / n, dtype=torch.float32, device=DEV)
    else:  # a fifth of the particles are stars: Plummer sphere of scale 0.1 with a tenth of the mass
        star = torch.rand(n, device=DEV, generator=g) < 0.2
        rs = torch.sqrt(u) * (100.0 / 101.0)
        r = torch.where(star, 0.1 / torch.sqrt(u.clamp(1e-15, 1.0 - 1e-15) ** (-2.0 / 3.0) - 1.0), rs / (1.0 - rs))
        a = 0.9 * (101.0 / 100.0) ** 2 / (1.0 + r) ** 2 + 0.1 * r * (0.01 + r * r) ** -1.5
        mass = torch.where(star, 0.1 / (0.2 * n), 0.9 / (0.8 * n)).to(torch.float32)
        hs = torch.where(star, 0.001, 0.005).to(torch.float32)
    pos = (r[:, None] * _directions(n, g)).contiguous()
    # a floor as the granularity of the particles leaves it at the centre
    return pos, mass, torch.hypot(a, torch.full_like(a, 0.02)).to(torch.float32), hs


def _box(ngrid, seed):
    """Lattice displaced by a Gaussian field with P(k) ~ k^-2 (rms 0.3
    spacings), unit box, and the linear-theory |a| = 4 pi |displacement|."""
    white = torch.randn(ngrid, ngrid, ngrid, dtype=torch.float64, device=DEV, generator=_gen(seed))
    wk = torch.fft.rfftn(white)
    f = torch.fft.fftfreq(ngrid, d=1.0 / ngrid, dtype=torch.float64, device=DEV)
    fz = torch.fft.rfftfreq(ngrid, d=1.0 / ngrid, dtype=torch.float64, device=DEV)
    nx, ny, nz = torch.meshgrid(f, f, fz, indexing="ij")
    n2 = nx * nx + ny * ny + nz * nz
    half = ngrid // 2
    keep = (n2 > 0) & (n2 <= half * half) & (nx.abs() < half) & (ny.abs() < half) & (nz < half)
    amp = torch.where(keep, n2.clamp_min(1.0) ** -1.5, torch.zeros_like(n2))  # sqrt(P) / k^2
    psi = torch.stack([torch.fft.irfftn(1j * c * amp * wk, s=(ngrid,) * 3).reshape(-1) for c in (nx, ny, nz)], dim=1)
    psi *= (0.3 / ngrid) / torch.sqrt((psi * psi).sum(1).mean())
    i = torch.arange(ngrid, dtype=torch.float64, device=DEV) / ngrid
    pos = torch.stack([c.reshape(-1) for c in torch.meshgrid(i, i, i, indexing="ij")], dim=1) + psi
    pos = pos - torch.floor(pos)
    pos = torch.where(pos >= 1.0, torch.zeros_like(pos), pos).contiguous()
    n = ngrid ** 3
    mass = torch.full((n,), 1.0 / n, dtype=torch.float32, device=DEV)
    a = 4.0 * math.pi * torch.linalg.vector_norm(psi, dim=1)
    return pos, mass, torch.hypot(a, torch.full_like(a, 0.005)).to(torch.float32)


def _bins(pos, seed, nbins=8):
    """Power-of-two time bins (0 the longest step): a fraction 2^-b of the
    particles, the densest ones, in bins >= b."""
    r = torch.linalg.vector_norm(pos, dim=1).clamp_min(1e-6)
    dens = torch.log(1.0 / (r * (r + 1.0) ** 3)) + 0.3 * torch.randn(len(r), dtype=torch.float64, device=DEV,
                                                                     generator=_gen(seed, 7))
    rank = torch.empty(len(r), dtype=torch.int64, device=DEV)
    rank[torch.argsort(dens, descending=True, stable=True)] = torch.arange(len(r), device=DEV)
    b = torch.floor(-torch.log2((rank + 1).to(torch.float64) / len(r)))
    return b.clamp(0, nbins - 1).to(torch.int8)


def _softening(case):
    if case["kind"] in ("box", "ewald"):
        return 1.0 / case["ngrid"] / 40.0  # 1/40 of the mean spacing
    return 0.01 if case.get("profile") == "plummer" else 0.005


def _shift(seed):
    """The random root placement a program draws for each build."""
    return tuple(float(x) for x in np.random.RandomState(int(seed) % (1 << 31)).uniform(0.0, 1.0, 3))


def _bparams(case, seed):
    return tpm.BuildParams(G=1.0, h=_softening(case), periodic=case["kind"] in ("box", "ewald"), box=1.0,
                           shift=_shift(seed), leaf_bucket=case["bucket"])


def _fparams(case):
    kw = {}
    if case["kind"] == "box":
        kw = dict(treepm=True, pm_n=case["pm_n"], asmth=1.25, rcut=4.5,
                  pm_grad=tpm.GRAD_IK if case["grad"] == "ik" else tpm.GRAD_FD4)
    elif case["kind"] == "iso":
        kw = dict(treepm=True, pm_n=case["pm_n"], asmth=case["asmth"], rcut=4.5)
    if case["crit"] == "rel":
        return tpm.ForceParams(crit=tpm.CRIT_RELATIVE, alpha=case["alpha"], **kw)
    return tpm.ForceParams(crit=tpm.CRIT_BH, theta=case["theta"], **kw)


_context = None


def _ctx():
    """The program's context: one for all its systems."""
    global _context
    if _context is None:
        _context = tpm.Context(0)
    return _context


class State:
    """What the program holds between calls; gives its resident trees and its plan back when dropped."""

    def __init__(self, **kw):
        self.systems, self.plan = [], None
        self.__dict__.update(kw)

    def __del__(self):
        try:
            if self.plan is not None:
                self.plan.close()
            for s in self.systems:
                s.release()
        except Exception:
            pass


def _outputs(n, device=DEV, pinned=False):
    kw = dict(pin_memory=True) if pinned else dict(device=device)
    return (torch.empty(n, 3, dtype=torch.float32, **kw), torch.empty(n, dtype=torch.float32, **kw),
            torch.empty(n, dtype=torch.int32, **kw))


def _served(case, seed):
    """The systems of a round (profile, particles, ids of the request); sizes spread evenly over the logarithm and
    parts from 1% to 100%, so that every seed has the same work."""
    rng = np.random.RandomState(int(seed) % (1 << 31))
    for k, (n, part) in enumerate(_served_sizes(case)):
        p = "plummer" if rng.randint(2) else "hernquist"
        pos, mass, a_old, _ = _particles(p, n, seed, 11 + k)
        yield p, pos, mass, a_old, torch.randperm(n, device=DEV, generator=_gen(seed, 1000 + k))[:part]


def _served_sizes(case):
    out = []
    for k in range(case["systems"]):
        n = int(case["nmin"] * (case["nmax"] / case["nmin"]) ** ((k + 0.5) / case["systems"]))
        out.append((n, max(1, int((0.01 + 0.99 * ((k * 7) % case["systems"] + 0.5) / case["systems"]) * n))))
    return out


def _request_sizes(total, rng, lo=64, hi=65536):
    """Log-uniform request sizes that add up to total."""
    out, left = [], total
    while left > 0:
        out.append(max(1, min(int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))), left)))
        left -= out[-1]
    return out


def prepare(case, seed):
    kind, ctx = case["kind"], _ctx()
    bp, fp = _bparams(case, seed), _fparams(case)
    rel = case["crit"] == "rel"
    if kind in ("box", "ewald"):
        pos, mass, a_old = _box(case["ngrid"], seed)
        hs = None
    elif kind != "round":
        pos, mass, a_old, hs = _particles(case["profile"], case["n"], seed)
    if kind in ("step", "box", "ewald", "iso"):
        acc, pot, nint = _outputs(len(mass))
        return State(kind=kind, ctx=ctx, pos=pos, mass=mass, hs=hs, a_old=a_old if rel else None, bp=bp, fp=fp,
                     acc=acc, pot=pot, nint=nint)
    if kind == "host":
        acc, pot, nint = _outputs(len(mass), pinned=True)
        pin = lambda x: x.cpu().pin_memory()  # noqa: E731
        return State(kind=kind, ctx=ctx, pos=pin(pos), mass=pin(mass), hs=None, a_old=pin(a_old) if rel else None,
                     bp=bp, fp=fp, acc=acc, pot=pot, nint=nint)
    if kind == "active":
        ids = torch.randperm(case["n"], device=DEV, generator=_gen(seed, 3))[:case["active"]].to(torch.int32)
        acc, pot, nint = _outputs(len(ids))
        s = ctx.build_tree(pos, mass, bp)
        return State(kind=kind, ctx=ctx, systems=[s], ids=ids, a_old=a_old[ids.long()].contiguous() if rel else None,
                     fp=fp, acc=acc, pot=pot, nint=nint)
    if kind == "substep":
        bins = _bins(pos, seed)
        acc, pot, nint = _outputs(len(mass))
        return State(kind=kind, ctx=ctx, pos=pos, mass=mass, bins=bins, amag=a_old, rel=rel, tick=case["tick"],
                     ids=torch.empty(len(mass), dtype=torch.int32, device=DEV),
                     a_old=torch.empty(len(mass), dtype=torch.float32, device=DEV), bp=bp, fp=fp, acc=acc, pot=pot,
                     nint=nint)
    if kind == "timebins":
        # the active sets of substeps of every kind, in key order, cut into requests, until `ids` are drawn
        s = ctx.build_tree(pos, mass, bp)
        perm = torch.from_numpy(s.tree_export()["perm"].astype(np.int64)).to(DEV)
        keyed = _bins(pos, seed)[perm]
        rng = np.random.RandomState(int(seed) % (1 << 31))
        ids, sizes, left, step = [], [], case["ids"], 1
        while left > 0:
            low = 7 - ((step & -step).bit_length() - 1)  # the lowest bin due on this substep
            act = perm[keyed >= max(low, 1)][:left].to(torch.int32)
            ids.append(act)
            sizes += _request_sizes(len(act), rng)
            left -= len(act)
            step = step % 127 + 1
        ids = torch.cat(ids).contiguous()
        systems, off, presorted = [s] * len(sizes), np.concatenate([[0], np.cumsum(sizes)]), True
        aold, keep = a_old[ids.long()].contiguous(), [s]
    else:  # round: one request each on systems of log-uniform size, a random part of the particles
        keep, ids, aold, sizes = [], [], [], []
        for k, (p, pos, mass, a_old, pick) in enumerate(_served(case, seed)):
            keep.append(ctx.build_tree(pos, mass, tpm.BuildParams(h=0.01 if p == "plummer" else 0.005,
                                                                  shift=_shift(seed + k), leaf_bucket=case["bucket"])))
            ids.append(pick.to(torch.int32))
            aold.append(a_old[pick])
            sizes.append(len(pick))
        ids, aold = torch.cat(ids).contiguous(), torch.cat(aold).contiguous()
        systems, off, presorted = keep, np.concatenate([[0], np.cumsum(sizes)]), False
    acc, pot, nint = _outputs(len(ids))
    return State(kind="batch", ctx=ctx, systems=keep, requests=systems, off=off.astype(np.int64), ids=ids,
                 a_old=aold if rel else None, fp=fp, presorted=presorted, plan=ctx.create_plan(len(ids), len(sizes)),
                 acc=acc, pot=pot, nint=nint)


def run(s):
    if s.kind == "batch":
        s.plan.compute_forces_batch(s.requests, s.off, s.fp, s.ids, s.acc, a_old=s.a_old, pot=s.pot, n_int=s.nint,
                                    presorted=s.presorted)
        return {"acc": s.acc, "pot": s.pot, "n_int": s.nint}
    if s.kind == "active":
        s.systems[0].compute_forces(active_ids=s.ids, a_old=s.a_old, fp=s.fp, acc=s.acc, pot=s.pot, n_int=s.nint)
        return {"acc": s.acc, "pot": s.pot, "n_int": s.nint}
    if s.kind == "substep":
        k = tpm.active_set(s.ctx, s.bins, s.tick, 8, s.ids, amag=s.amag, a_old=s.a_old)
        ids, acc, pot, nint = s.ids[:k], s.acc[:k], s.pot[:k], s.nint[:k]
        t = s.ctx.build_tree(s.pos, s.mass, s.bp)
        t.compute_forces(active_ids=ids, a_old=s.a_old[:k] if s.rel else None, fp=s.fp, acc=acc, pot=pot, n_int=nint)
        t.release()
        return {"ids": ids, "acc": acc, "pot": pot, "n_int": nint}
    t = s.ctx.build_tree(s.pos, s.mass, s.bp, hsoft=s.hs)
    if s.fp.treepm:
        t.pm_long_range(s.fp)
    t.compute_forces(a_old=s.a_old, fp=s.fp, acc=s.acc, pot=s.pot, n_int=s.nint)
    t.release()
    return {"acc": s.acc, "pot": s.pot, "n_int": s.nint}


# ---------------------------------------------------------------- work
def _active_count(case):
    kind = case["kind"]
    if kind in ("box", "ewald"):
        return case["ngrid"] ** 3
    if kind == "active":
        return case["active"]
    if kind == "substep":  # bins at and above 7 - log2(tick's trailing zeros) hold 2^-b of the particles
        tz = (case["tick"] & -case["tick"]).bit_length() - 1
        return max(1, case["n"] >> max(7 - tz, 0))
    if kind == "timebins":
        return case["ids"]
    if kind == "round":
        return sum(part for _, part in _served_sizes(case))
    return case["n"]


def work(case):
    """Inputs read once and outputs written once, and 20 flops per interaction
    of the per-particle walk (40 with the short-range factors, 70 with the
    Ewald table); the mesh transforms add 2.5 N log2 N each."""
    kind, act = case["kind"], _active_count(case)
    crit = "rel" if case["crit"] == "rel" else "bh"
    name = {"box": "box", "ewald": "ewald", "iso": "iso", "substep": "dense", "timebins": "dense"}.get(
        kind, case.get("profile", "hernquist"))
    per = INTERACTIONS["%s/%s" % (name, crit)] * (1.0 if crit == "rel" else (0.7 / case["theta"]) ** 3)
    flops = act * per * {"box": 40, "iso": 40, "ewald": 70}.get(kind, 20)
    byts = act * (20 + (4 if crit == "rel" else 0))  # acc, pot, n_int, |a_old|
    if kind in ("active", "timebins", "round"):
        byts += act * (4 + 28)  # ids, and at least the active particles themselves
    else:
        byts += (case["ngrid"] ** 3 if kind in ("box", "ewald") else case["n"]) * (28 + (4 if name == "two" else 0))
    if kind == "substep":
        byts += case["n"] + act * 8
    if kind in ("box", "iso"):
        m = case["pm_n"] if kind == "box" else 2 * case["pm_n"]
        ffts = 5 if case.get("grad") == "ik" else 2
        flops += ffts * 2.5 * m ** 3 * 3 * math.log2(m)
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------- 64 bits
def _spline(r, h):
    """Force factor (over r) and potential of the spline-softened unit mass, support h (Springel 2001)."""
    u = r / h
    s = r.clamp_min(1e-300)
    f1 = (32.0 / 3.0 + u * u * (32.0 * u - 192.0 / 5.0)) / h ** 3
    f2 = (64.0 / 3.0 - 48.0 * u + 192.0 / 5.0 * u * u - 32.0 / 3.0 * u ** 3) / h ** 3 - (1.0 / 15.0) / s ** 3
    p1 = (-14.0 / 5.0 + 16.0 / 3.0 * u ** 2 - 48.0 / 5.0 * u ** 4 + 32.0 / 5.0 * u ** 5) / h
    p2 = (-16.0 / 5.0 + 32.0 / 3.0 * u ** 2 - 16.0 * u ** 3 + 48.0 / 5.0 * u ** 4 - 32.0 / 15.0 * u ** 5) / h + \
        (1.0 / 15.0) / s
    f = torch.where(u < 0.5, f1, torch.where(u < 1.0, f2, 1.0 / s ** 3))
    p = torch.where(u < 0.5, p1, torch.where(u < 1.0, p2, -1.0 / s))
    return f, p


def _direct(pos, mass, hs, ids, h):
    """Direct sum in 64 bits on the particles ids."""
    m = mass.to(torch.float64)
    acc = torch.empty(len(ids), 3, dtype=torch.float64, device=DEV)
    pot = torch.empty(len(ids), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 24) // len(mass))
    for a in range(0, len(ids), step):
        t = ids[a:a + step]
        d = pos[None, :, :] - pos[t][:, None, :]
        r = torch.linalg.vector_norm(d, dim=2)
        sup = h if hs is None else torch.maximum(hs[None, :], hs[t][:, None]).to(torch.float64)
        f, p = _spline(r, sup)
        w = m[None, :].expand_as(r).clone()
        w[torch.arange(len(t), device=DEV), t] = 0.0  # no particle acts on itself
        acc[a:a + step] = torch.einsum("ij,ijk->ik", w * f, d)
        pot[a:a + step] = (w * p).sum(1)
    return acc, pot


def _ewald(pos, mass, h):
    """Periodic forces in 64 bits: the Ewald sum of the unit box split at 10 / box, so that the nearest image
    (erfc(5) = 1.5e-12 at half a box) and |m|^2 <= 290 wave vectors suffice, the nearest image softened."""
    n, a = len(mass), 10.0
    m = mass.to(torch.float64)
    acc = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 24) // n)
    for b in range(0, n, step):
        d = pos[None, :, :] - pos[b:b + step][:, None, :]
        d -= torch.round(d)
        r = torch.linalg.vector_norm(d, dim=2)
        s = r.clamp_min(1e-12)
        g = torch.special.erfc(a * s) + 2.0 * a / math.sqrt(math.pi) * s * torch.exp(-(a * s) ** 2)
        f, _ = _spline(r, h)
        w = m[None, :] * ((g - 1.0) / s ** 3 + f)
        k = torch.arange(len(w), device=DEV)
        w[k, k + b] = 0.0
        acc[b:b + step] = torch.einsum("ij,ijk->ik", w, d)
    q = torch.arange(-17, 18, dtype=torch.float64, device=DEV)
    kv = torch.stack([c.reshape(-1) for c in torch.meshgrid(q, q, q, indexing="ij")], dim=1)
    k2 = (kv * kv).sum(1)
    half = (kv[:, 0] > 0) | ((kv[:, 0] == 0) & ((kv[:, 1] > 0) | ((kv[:, 1] == 0) & (kv[:, 2] > 0))))
    keep = half & (k2 <= 290)
    kv, k2 = 2.0 * math.pi * kv[keep], 4.0 * math.pi ** 2 * k2[keep]
    wk = 2.0 * 4.0 * math.pi * torch.exp(-k2 / (4.0 * a * a)) / k2  # both halves
    for b in range(0, len(k2), 256):
        ph = pos @ kv[b:b + 256].T
        c, s = torch.cos(ph), torch.sin(ph)
        sc, ss = m @ c, m @ s  # source sums: sum_j m_j sin(k (x_j - x_i)) = ss cos - sc sin
        acc += ((ss[None, :] * c - sc[None, :] * s) * wk[None, b:b + 256]) @ kv[b:b + 256]
    return acc


def exact(case, seed):
    """Forces (and, open boundaries, potentials) of the softened direct sum, or of the Ewald sum for a periodic
    box, where they take a few seconds; the counts have no such value."""
    kind, act = case["kind"], _active_count(case)
    if kind in ("timebins", "substep"):
        return None
    if kind in ("box", "ewald"):
        if case["ngrid"] ** 3 > 65536:
            return None
        pos, mass, _ = _box(case["ngrid"], seed)
        sh = torch.tensor(_shift(seed), dtype=torch.float64, device=DEV)
        return {"acc": _ewald((pos + sh) % 1.0, mass, _softening(case)), "pot": None, "n_int": None}
    if kind == "round":
        if sum(n * part for n, part in _served_sizes(case)) > 1.0e10:
            return None
        got = [_direct(pos, mass, None, pick, 0.01 if p == "plummer" else 0.005)
               for p, pos, mass, _, pick in _served(case, seed)]
        return {"acc": torch.cat([a for a, _ in got]), "pot": torch.cat([p for _, p in got]), "n_int": None}
    if act * case["n"] > 1.0e10:
        return None
    pos, mass, _, hs = _particles(case["profile"], case["n"], seed)
    ids = torch.arange(case["n"], device=DEV)
    if kind == "active":
        ids = torch.randperm(case["n"], device=DEV, generator=_gen(seed, 3))[:case["active"]]
    acc, pot = _direct(pos, mass, hs, ids, _softening(case))
    return {"acc": acc, "pot": pot, "n_int": None}
