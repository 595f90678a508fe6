"""The workloads that the framework's speed is measured on: what a user has it do, through its public entry points.

Kinds of pass (every array on the GPU, in the caller's order):

* ``step``     leaf build + the whole step (geometry, corrections, hydro, gravity and both adjoints), the
               headline path: a simulation that hands its particles over anew each step.
* ``gravity``  leaf build + short-range gravity alone: a particle-mesh code that only wants the direct force.
* ``reverse``  gravity and its reverse mode on leaves that are kept: the two heaviest single kernels.
* ``hydro``    geometry, corrections and hydro as single calls on leaves that are kept.
* ``passes``   geometry, corrections, Extras, the Acceleration and Energy passes (limited viscosity) and the
               Courant step as single calls: a host code with its own integrator.
* ``advance``  one two-stage timestep with everything in it (state put back before each pass).
* ``chain``    forward and reverse pass of geometry -> corrections -> hydro on leaves that are kept.
* ``autograd`` leaf build, gravity and geometry under torch autograd, and the gradients of a loss.
* ``batch``    many boxes of uneven size: leaf rebuild + step as one CUDA graph launch.

Particles come from the framework's own seeded generators.  Boxes above side 64 repeat a periodic clustered
box along each axis, every copy jittered on its own: smoothing lengths and clustering are those of the base.
"""
import math

import numpy as np
import torch

from paper_2310_16122_gb300 import api, autograd
from paper_2310_16122_gb300 import workloads as W

SIG_BETA = 3.0
CFL = 0.25
DT_MAX = 1.0
HALOS_PER_64 = 200  # Plummer halos of a side-64 clustered box


def listed():
    return [
        # the smallest whole call: the 2x16^3 lattice box on a fixed chaining mesh, every output
        dict(name="tiny_step", kind="step", layout="lattice", side=16, cells=4, full=True),
        # a PM code's short-range force on an odd number of dark-matter particles, no gas
        dict(name="dm_gravity", kind="gravity", layout="random", n=30011, gas=0.0, max_leaf=128),
        # gradients of |a|^2 + rho in positions and masses, 2x32^3
        dict(name="autograd_32", kind="autograd", layout="clustered", side=32),
        # a batch of independent boxes, sides 12-48, one graph launch per step
        dict(name="batch_24", kind="batch", boxes=24, lo=12, hi=48),
        # the 2x64^3 clustered box, whole step, every output
        dict(name="step_64", kind="step", layout="clustered", side=64, full=True),
        # single calls of the hydro chain, an odd side
        dict(name="hydro_45", kind="hydro", layout="clustered", side=45),
        # Extras, Acceleration and Energy passes as single calls, 2x64^3
        dict(name="passes_64", kind="passes", layout="clustered", side=64),
        # one timestep with gravity and the limited viscosity, 2x64^3
        dict(name="advance_64", kind="advance", layout="clustered", side=64, limited=True, gravity=True),
        # gradients through geometry -> corrections -> hydro, 2x64^3
        dict(name="chain_64", kind="chain", layout="clustered", side=64),
        # gravity and its reverse mode on kept leaves, 2x128^3
        dict(name="reverse_128", kind="reverse", layout="clustered", side=64, tiles=2),
        # the hydro chain as single calls, 2x128^3
        dict(name="hydro_128", kind="hydro", layout="clustered", side=64, tiles=2),
        # the largest box: 2x256^3 particles, the accelerations, rates and gradients of a step
        dict(name="step_256", kind="step", layout="clustered", side=64, tiles=4, full=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "gravity", "reverse", "hydro", "passes", "advance", "chain", "autograd", "batch"])
    c = dict(kind=kind)
    if kind == "batch":
        return dict(c, boxes=rng.randint(3, 24), lo=rng.randint(12, 20), hi=rng.randint(24, 48))
    if kind == "gravity":
        return dict(c, layout="random", n=_log_int(rng, 4000, 2000000), gas=rng.choice([0.0, 0.35, 0.5]),
                    max_leaf=rng.choice([96, 128, 128, 160]))
    top = {"step": 256, "advance": 128, "chain": 128, "autograd": 96}.get(kind, 160)
    side = _log_int(rng, 12, top)
    if kind == "step":
        c["full"] = rng.random() < 0.5
    if kind == "advance":
        c.update(limited=rng.random() < 0.7, gravity=rng.random() < 0.7)
    if side <= 64:
        if kind == "step" and side <= 24 and rng.random() < 0.4:
            return dict(c, layout="lattice", side=side, cells=max(3, side // 4))
        return dict(c, layout="clustered", side=side)
    tiles = -(-side // 64)
    return dict(c, layout="clustered", side=side // tiles, tiles=tiles)


# --------------------------------------------------------------------------- inputs

def _n(case):
    if case["kind"] == "batch":
        return int(sum(2 * s ** 3 for s in _sides(case)))
    if case["layout"] == "random":
        return int(case["n"])
    return 2 * (int(case["side"]) * int(case.get("tiles", 1))) ** 3


def _halos(side):
    return int(round(HALOS_PER_64 * (side / 64.0) ** 3))


def _sides(case):
    """The sides of a batch: the case's, whatever the seed (equal work on every input)."""
    r = np.random.default_rng(1009)
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [int(round(math.exp(r.uniform(lo, hi)))) for _ in range(int(case["boxes"]))]


def _tile(db, tiles, seed):
    """A DeviceBox of tiles^3 copies of the periodic box db, jittered, in a shuffled order."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 17)
    n0, L0 = db.n, db.L
    t3 = tiles ** 3
    n, L = n0 * t3, L0 * tiles
    order = torch.randperm(n, generator=g, device="cuda")
    base, copy = order % n0, order // n0
    for a, (name, div) in enumerate((("x", 1), ("y", tiles), ("z", tiles * tiles))):
        c = getattr(db, name)[base] + ((copy // div) % tiles).float() * L0
        c += 1e-3 * torch.randn(n, generator=g, device="cuda")
        c = torch.where(c >= L, c - L, torch.where(c < 0, c + L, c))
        setattr(db, name, torch.where((c >= 0) & (c < L), c, torch.zeros_like(c)).contiguous())
    for name in ("species", "m", "h"):
        setattr(db, name, getattr(db, name)[base].contiguous())
    gas = (db.species == 0).float()
    db.u = gas * (0.9 + 0.2 * torch.rand(n, generator=g, device="cuda"))
    db.v3 = (gas * 0.05 * torch.randn(3, n, generator=g, device="cuda")).contiguous()
    db.n, db.L = n, float(L)
    return db


def _inputs(case, seed):
    """The particles of a case (a DeviceBox) from the seed alone."""
    if case["layout"] == "lattice":
        box = W.lattice_box(int(case["side"]), 0.2, seed, h=1.0, leaf_mode=0, cells=int(case["cells"]))
    elif case["layout"] == "random":
        n, gas = int(case["n"]), float(case["gas"])
        L = (n / 2.0) ** (1.0 / 3.0)
        h = 1.2 * L / (n * gas) ** (1.0 / 3.0) if gas > 0 else 1.0
        box = W.random_box(n, L, gas, seed, max_leaf=int(case["max_leaf"]), h=h)
    else:
        box = W.clustered_box(int(case["side"]), _halos(int(case["side"])), seed)
    db = api.DeviceBox(box)
    tiles = int(case.get("tiles", 1))
    return _tile(db, tiles, seed) if tiles > 1 else db


def _batch_boxes(case, seed):
    return [W.clustered_box(s, _halos(s), 1000 * int(seed) + b) for b, s in enumerate(_sides(case))]


def _cotangents(n, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 29)
    return torch.randn(3, n, generator=g, device="cuda"), torch.randn(n, generator=g, device="cuda")


# --------------------------------------------------------------------------- the passes

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            ctx = api.Context(0, stream=side)
            db = api.DeviceBatch(_batch_boxes(case, seed))
            lv = api.build_leaves_batch(ctx, db)
            io = api.StepIO(ctx, db, outputs=False)
            graph = api.RebuildStepGraph(ctx, lv, db, io)
        return dict(case=case, ctx=ctx, db=db, lv=lv, io=io, graph=graph)
    db = _inputs(case, seed)
    ctx = api.Context(0)
    s = dict(case=case, ctx=ctx, db=db)
    if kind == "step":
        s["io"] = api.StepIO(ctx, db, outputs=bool(case["full"]))
    elif kind in ("reverse", "hydro", "passes", "chain"):
        s["lv"] = _leaves(ctx, db)
        if kind == "chain":
            s["dvbar"], s["dubar"] = _cotangents(db.n, seed)
    elif kind == "advance":
        s["start"] = [t.clone() for t in (db.x, db.y, db.z, db.v3, db.u)]
        s["ap"] = api.AdvanceParams(cfl=CFL, dt_max=DT_MAX, sig_beta=SIG_BETA, limited=bool(case["limited"]),
                                    gravity=bool(case["gravity"]))
    elif kind == "autograd":
        s["pos"] = torch.stack([db.x, db.y, db.z]).requires_grad_(True)
        s["m"] = db.m.clone().requires_grad_(True)
    return s


def _leaves(ctx, db):
    return api.build_leaves(ctx, db.x, db.y, db.z, db.species, db.h, db.L, db.lp)


def _step_outputs(io):
    out = dict(dv=io.dv, du=io.du, acc=io.acc, gx_grav=io.gx_grav, gm_grav=io.gm_grav, gx_geom=io.gx_geom,
               gm_geom=io.gm_geom, n_singular=io.n_singular)
    if io.full:
        out.update(V=io.V, rho=io.rho, A=io.A, B=io.B, gA=io.gA, gB=io.gB)
    return out


def run(s):
    ctx, db, kind = s["ctx"], s["db"], s["case"]["kind"]
    if kind == "batch":
        s["graph"].launch()
        return _step_outputs(s["io"])
    if kind == "step":
        lv = _leaves(ctx, db)
        api.step(ctx, lv, db, s["io"])
        return dict(_step_outputs(s["io"]), leaves=lv.n_leaves, grav_pairs=lv.n_grav_pairs, hydro_pairs=lv.n_hydro_pairs)
    if kind == "gravity":
        lv = _leaves(ctx, db)
        a, _ = api.grav_short(ctx, lv, db.gp, db.m)
        return dict(a=a, leaves=lv.n_leaves, pairs=lv.n_grav_pairs, images=lv.n_grav_images)
    if kind == "reverse":
        a, _ = api.grav_short(ctx, s["lv"], db.gp, db.m)
        gx, gm = api.grav_short_adjoint(ctx, s["lv"], db.gp, db.m, 2.0 * a)
        return dict(a=a, gx=gx, gm=gm)
    if kind == "hydro":
        lv = s["lv"]
        V, rho, _ = api.geometry(ctx, lv, db.m)
        A, B, gA, gB, ns = api.corrections(ctx, lv, V)
        dv, du, _, _ = api.hydro(ctx, lv, db.hp, db.m, db.v3, db.u, V, rho, A, B, gA, gB)
        return dict(V=V, rho=rho, A=A, B=B, gA=gA, gB=gB, n_singular=ns, dv=dv, du=du)
    if kind == "passes":
        lv = s["lv"]
        V, rho, _ = api.geometry(ctx, lv, db.m)
        A, B, gA, gB, ns = api.corrections(ctx, lv, V)
        rho_r, dvdx, _ = api.extras(ctx, lv, db.m, db.v3, V, A, B, gA, gB)
        args = (db.m, db.v3, db.u, V, rho_r, A, B, gA, gB)
        dv, vsig, _, _ = api.hydro_accel(ctx, lv, db.hp, *args, dvdx=dvdx, sig_beta=SIG_BETA)
        du, _, _ = api.hydro_energy(ctx, lv, db.hp, *args, db.v3, dvdx=dvdx)
        dt = api.timestep(ctx, vsig, CFL, DT_MAX)
        return dict(V=V, rho=rho, rho_r=rho_r, dvdx=dvdx, dv=dv, du=du, dt=dt, n_singular=ns)
    if kind == "advance":
        for t, t0 in zip((db.x, db.y, db.z, db.v3, db.u), s["start"]):
            t.copy_(t0)
        dt = api.advance(ctx, db, s["ap"])
        return dict(x=db.x, y=db.y, z=db.z, v=db.v3, u=db.u, dt=dt)
    if kind == "chain":
        g = api.hydro_chain_adjoint(ctx, s["lv"], db, s["dvbar"], s["dubar"])
        return {k: g[k] for k in ("x", "m", "v", "u", "dv", "du", "n_singular")}
    pos, m = s["pos"], s["m"]
    p = pos.detach()
    lv = api.build_leaves(ctx, p[0], p[1], p[2], db.species, db.h, db.L, db.lp)
    a = autograd.gravity(pos, m, ctx, lv, db.gp)
    V, rho = autograd.geometry(pos, m, ctx, lv)
    gx, gm = torch.autograd.grad((a * a).sum() + rho.sum(), (pos, m))
    return dict(a=a.detach(), V=V.detach(), rho=rho.detach(), gx=gx, gm=gm)


# flop of one in-range ordered pair of each kernel, and 32-bit words read and written per particle
_FLOP = dict(geometry=24, corrections=88, hydro=160, gravity=29, gravity_adjoint=68, geometry_adjoint=31, extras=103,
             accel=216, energy=224, hydro_adjoint=480, corrections_adjoint=535)


def work(case):
    n, kind = _n(case), case["kind"]
    gas = n * (float(case["gas"]) if case.get("layout") == "random" else 0.5) * 58.0  # ordered gas pairs
    grav = n * 2.0 * 4.0 / 3.0 * math.pi * W.R_CUT ** 3                               # ordered gravity pairs
    f = _FLOP
    chain = f["geometry"] + f["corrections"] + f["hydro"]
    if kind in ("step", "batch"):
        words = 10 + 19 + (18 if case.get("full") else 0)
        flops = gas * (chain + f["geometry_adjoint"]) + grav * (f["gravity"] + f["gravity_adjoint"])
    elif kind == "gravity":
        words, flops = 4 + 3, grav * f["gravity"]
    elif kind == "reverse":
        words, flops = 4 + 3 + 4, grav * (f["gravity"] + f["gravity_adjoint"])
    elif kind == "hydro":
        words, flops = 9 + 22, gas * chain
    elif kind == "passes":
        words, flops = 9 + 16, gas * (f["geometry"] + f["corrections"] + f["extras"] + f["accel"] + f["energy"])
    elif kind == "advance":
        per = f["geometry"] + f["corrections"] + (f["extras"] if case["limited"] else 0) + f["accel"] + f["energy"]
        words, flops = 9 + 7, 2 * (gas * per + (grav * f["gravity"] if case["gravity"] else 0))
    elif kind == "chain":
        words = 13 + 12
        flops = gas * (chain + f["hydro_adjoint"] + f["corrections_adjoint"] + f["geometry_adjoint"])
    else:  # autograd
        words = 6 + 9
        flops = grav * (f["gravity"] + f["gravity_adjoint"]) + gas * (f["geometry"] + f["geometry_adjoint"])
    return {"bytes": 4.0 * n * words, "flops": float(flops)}


# --------------------------------------------------------------------------- the same in 64 bits, plain torch

MOST_EXACT = 600000  # particles; above, the pair lists in 64 bits take too long


def _pairs(pos, L, c):
    """All (i, j) with |x_i - x_j| < c_i + c_j (minimum image, i = j included) and x_ij, from a cell list."""
    n = pos.shape[1]
    dev = pos.device
    nc = int(L / (2.0 * float(c.max()) * (1 + 1e-6)))
    brute = nc < 3
    if brute:
        nc = 1
    cell = (pos * (nc / L)).floor().clamp_(max=nc - 1).long()
    cid = (cell[0] * nc + cell[1]) * nc + cell[2]
    order = torch.argsort(cid)
    count = torch.bincount(cid, minlength=nc ** 3)
    first = torch.cumsum(count, 0) - count
    ps, cs, cell = pos[:, order], c[order], cell[:, order]
    out = []
    for k in range(1 if brute else 27):
        off = (0, 0, 0) if brute else (k // 9 - 1, k // 3 % 3 - 1, k % 3 - 1)
        near = [(cell[a] + off[a]) % nc for a in range(3)]
        near = (near[0] * nc + near[1]) * nc + near[2]
        ends = torch.cumsum(count[near], 0)
        lo = 0
        while lo < n:  # about 2e8 candidates at a time
            base = int(ends[lo - 1]) if lo else 0
            hi = max(lo + 1, int(torch.searchsorted(ends, base + 200000000, right=True)))
            nk = count[near[lo:hi]]
            i = torch.repeat_interleave(torch.arange(lo, min(hi, n), device=dev), nk)
            start = torch.cumsum(nk, 0) - nk
            j = first[near[i]] + torch.arange(i.numel(), device=dev) - start[i - lo]
            d = ps[:, i] - ps[:, j]
            d -= L * torch.round(d / L)
            keep = (d * d).sum(0) < (cs[i] + cs[j]) ** 2
            out.append((order[i[keep]], order[j[keep]], d[:, keep]))
            lo = min(hi, n)
    return torch.cat([o[0] for o in out]), torch.cat([o[1] for o in out]), torch.cat([o[2] for o in out], 1)


def _sum(i, v, n):
    return torch.zeros(*v.shape[:-1], n, dtype=v.dtype, device=v.device).index_add(-1, i, v)


class _Gas:
    """The gas chain in 64 bits on one pair list: positions (3, N) and smoothing lengths of the gas particles."""

    def __init__(self, x, h, L, hp, pairs=None):
        self.hp, self.h, self.n = hp, h, x.shape[1]
        self.i, self.j, d = pairs if pairs is not None else _pairs(x, L, h)
        if pairs is not None:  # differentiable separations
            d = x[:, self.i] - x[:, self.j]
            d = d - L * torch.round(d / L).detach()
        self.d = d
        r2 = (d * d).sum(0)
        r = torch.sqrt(r2 + 1e-300)
        hij = 0.5 * (h[self.i] + h[self.j])
        q = r / hij
        t = (1 - 0.5 * q).clamp(min=0)
        norm = 495.0 / (256.0 * math.pi) / hij ** 3
        self.r2, self.r, self.hij = r2, r, hij
        self.Wij = norm * t ** 6 * (1 + 3 * q + 35.0 / 12.0 * q * q)
        self.dWr = norm / hij ** 2 * t ** 5 * (-14.0 / 3.0) * (1 + 2.5 * q)

    def geometry(self, m):
        self.m = m
        s = _sum(self.i, self.Wij, self.n)
        self.V, self.rho = 1 / s, m * s

    def corrections(self):
        i, x, n = self.i, self.d, self.n
        w, vd = self.V[self.j] * self.Wij, self.V[self.j] * self.dWr
        m0 = _sum(i, w, n)
        m1 = _sum(i, w * x, n)                       # (3, n)
        dm0 = _sum(i, vd * x, n)
        rows2, rows3 = {}, {}
        for a in range(3):
            for b in range(a, 3):
                xx = x[a] * x[b]
                rows2[a, b] = (_sum(i, w * xx, n), _sum(i, vd * xx, n))
                for c in range(b, 3):
                    rows3[a, b, c] = _sum(i, vd * xx * x[c], n)
        k2 = lambda a, b: tuple(sorted((a, b)))
        k3 = lambda a, b, c: tuple(sorted((a, b, c)))
        m2 = torch.stack([torch.stack([rows2[k2(a, b)][0] for b in range(3)]) for a in range(3)])
        s2 = torch.stack([torch.stack([rows2[k2(a, b)][1] for b in range(3)]) for a in range(3)])
        s3 = torch.stack([torch.stack([torch.stack([rows3[k3(a, b, c)] for c in range(3)]) for b in range(3)])
                          for a in range(3)])
        eye = torch.eye(3, dtype=x.dtype, device=x.device)
        dm1 = eye[:, :, None] * m0 + s2              # [g, a]
        dm2 = (torch.einsum("ag,bn->gabn", eye, m1) + torch.einsum("bg,an->gabn", eye, m1) + s3)
        Mi = torch.linalg.inv(m2.permute(2, 0, 1)).permute(1, 2, 0)
        B = -torch.einsum("abn,bn->an", Mi, m1)
        A = 1 / (m0 + (B * m1).sum(0))
        dMB = torch.einsum("gabn,bn->gan", dm2, B)
        self.gA = -A * A * (dm0 + 2 * torch.einsum("an,gan->gn", B, dm1) + torch.einsum("an,gan->gn", B, dMB))
        self.gB = -torch.einsum("abn,gbn->gan", Mi, dm1 + dMB)   # [g, a]
        self.A, self.B = A, B

    def _grad(self, p, x):
        """grad W^R of particles p at separations x."""
        one = 1 + (self.B[:, p] * x).sum(0)
        A = self.A[p]
        gBx = (self.gB[:, :, p] * x[None]).sum(1)
        return self.gA[:, p] * (one * self.Wij) + A * self.Wij * (gBx + self.B[:, p]) + A * one * self.dWr * x

    def extras(self, v):
        i, j, n = self.i, self.j, self.n
        wr = self.A[i] * (1 + (self.B[:, i] * self.d).sum(0)) * self.Wij
        g = self._grad(i, self.d)
        dv = self.V[j] * (v[:, j] - v[:, i])
        self.rho_r = _sum(i, self.m[j] * wr, n)
        self.G = torch.stack([torch.stack([_sum(i, dv[a] * g[b], n) for b in range(3)]) for a in range(3)])

    def force(self, v, u, limited):
        """f_ij, v_ij of every pair, with the Monaghan or the limited viscosity."""
        hp, i, j, x = self.hp, self.i, self.j, self.d
        rho = self.rho_r if limited else self.rho
        P = (hp.gamma - 1) * rho * u
        self.c = torch.sqrt(hp.gamma * (hp.gamma - 1) * u)
        vij = v[:, i] - v[:, j]
        if limited:
            si, sj = (self.G[:, :, i] * x[None]).sum(1), (self.G[:, :, j] * x[None]).sum(1)
            ai, aj = (x * si).sum(0), (x * sj).sum(0)
            phi = torch.where(ai * aj > 0, 4 * ai * aj / (ai + aj) ** 2, torch.zeros_like(ai))
            vx = ((vij - 0.5 * phi * (si + sj)) * x).sum(0)
        else:
            vx = (vij * x).sum(0)
        mu = torch.where(vx < 0, self.hij * vx / (self.r2 + hp.eta2 * self.hij ** 2), torch.zeros_like(vx))
        Q = 0.5 * (rho[i] + rho[j]) * (-hp.alpha * 0.5 * (self.c[i] + self.c[j]) * mu + hp.beta * mu * mu)
        return -0.5 * self.V[i] * self.V[j] * (P[i] + P[j] + Q) * (self._grad(i, x) - self._grad(j, -x)), vij

    def hydro(self, v, u):
        f, vij = self.force(v, u, False)
        return _sum(self.i, f, self.n) / self.m, _sum(self.i, -0.5 * (vij * f).sum(0), self.n) / self.m

    def accel(self, v, u, limited):
        f, vij = self.force(v, u, limited)
        w = (vij * self.d).sum(0) / self.r
        vs = self.c[self.i] + self.c[self.j] - SIG_BETA * w.clamp(max=0)
        return _sum(self.i, f, self.n) / self.m, float((vs / self.h[self.i]).max())

    def energy(self, v, u, vstar, limited):
        f, _ = self.force(v, u, limited)
        i, j = self.i, self.j
        dE = -(f * (vstar[:, i] - vstar[:, j])).sum(0)
        du = u[j] - u[i]
        w = 0.5 + 0.5 * torch.sign(dE) * du / (du.abs() + 0.5 * (u[i] + u[j]))
        return _sum(i, w * dE, self.n) / self.m


def _gravity(x, L, m, gp, abar=None):
    """a (3, n), and with a function abar(a) the reverse mode (gx, gm) for that cotangent."""
    n = x.shape[1]
    i, j, d = _pairs(x, L, torch.full((n,), 0.5 * gp.r_cut, dtype=x.dtype, device=x.device))
    off = i != j
    i, j, d = i[off], j[off], -d[:, off]  # x_j - x_i
    s = (d * d).sum(0)
    e2 = float(np.float32(gp.eps)) ** 2
    c = [float(np.float32(v)) for v in gp.poly]
    poly, dpoly = torch.full_like(s, c[5]), torch.full_like(s, 5 * c[5])
    for k in (4, 3, 2, 1, 0):
        poly = poly * s + c[k]
        if k:
            dpoly = dpoly * s + k * c[k]
    g = (s + e2) ** -1.5 - poly
    a = _sum(i, m[j] * g * d, n)
    if abar is None:
        return a
    ab = abar(a)
    dg = -1.5 * (s + e2) ** -2.5 - dpoly
    w = m[i] * ab[:, j] - m[j] * ab[:, i]
    gx = _sum(i, g * w + 2 * dg * (d * w).sum(0) * d, n)
    gm = _sum(i, -g * (ab[:, j] * d).sum(0), n)
    return a, gx, gm


def _full(gas, v, n):
    out = torch.zeros(*v.shape[:-1], n, dtype=v.dtype, device=v.device)
    out[..., gas] = v.detach()
    return out


def _state(db):
    x = torch.stack([db.x, db.y, db.z]).double()
    gas = torch.nonzero(db.species == 0).flatten()
    return x, gas, db.h.double(), db.m.double(), db.v3.double(), db.u.double()


def _geom_grad(G):
    """Gradient of sum rho in the positions and masses."""
    k = (G.m[G.i] + G.m[G.j]) * G.dWr
    return _sum(G.i, k * G.d, G.n), 1 / G.V


def _exact_step(db, full):
    x, gas, h, m, v, u = _state(db)
    n = db.n
    F = lambda t: _full(gas, t, n)
    G = _Gas(x[:, gas], h[gas], db.L, db.hp)
    G.geometry(m[gas])
    G.corrections()
    dv, du = G.hydro(v[:, gas], u[gas])
    gx, gm = _geom_grad(G)
    out = dict(dv=F(dv), du=F(du), gx_geom=F(gx), gm_geom=F(gm), n_singular=None)
    if full:
        out.update(V=F(G.V), rho=F(G.rho), A=F(G.A), B=F(G.B), gA=F(G.gA), gB=F(G.gB.reshape(9, -1)))
    del G
    out["acc"], out["gx_grav"], out["gm_grav"] = _gravity(x, db.L, m, db.gp, lambda a: 2 * a)
    return out


def _exact_advance(db, case):
    x, gas, h, m, v, u = _state(db)
    n, L, limited = db.n, db.L, bool(case["limited"])

    def stage(x, v, u):
        G = _Gas(x[:, gas], h[gas], L, db.hp)
        G.geometry(m[gas])
        G.corrections()
        if limited:
            G.extras(v[:, gas])
        dv, q = G.accel(v[:, gas], u[gas], limited)
        a = _full(gas, dv, n)
        if case["gravity"]:
            a = a + _gravity(x, L, m, db.gp)
        return G, a, q

    G, a, q = stage(x, v, u)
    du = _full(gas, G.energy(v[:, gas], u[gas], v[:, gas], limited), n)
    dt = min(DT_MAX, CFL / q) if q > 0 else DT_MAX
    vp, up = v + 0.5 * dt * a, u + 0.5 * dt * du
    xp = (x + 0.5 * dt * vp) % L
    G, a, _ = stage(xp, vp, up)
    v1 = v + dt * a
    vs = 0.5 * (v + v1)
    u1 = u + dt * _full(gas, G.energy(vp[:, gas], up[gas], vs[:, gas], limited), n)
    x1 = (x + dt * vs) % L
    return dict(x=x1[0], y=x1[1], z=x1[2], v=v1, u=u1, dt=torch.tensor([dt], dtype=torch.float64))


def exact(case, seed):
    kind = case["kind"]
    if _n(case) > MOST_EXACT:
        return None
    if kind == "batch":
        per = [_exact_step(api.DeviceBox(b), False) for b in _batch_boxes(case, seed)]
        return {k: None if per[0][k] is None else torch.cat([p[k] for p in per], -1) for k in per[0]}
    db = _inputs(case, seed)
    x, gas, h, m, v, u = _state(db)
    n = db.n
    F = lambda t: _full(gas, t, n)
    if kind == "step":
        return dict(_exact_step(db, bool(case["full"])), leaves=None, grav_pairs=None, hydro_pairs=None)
    if kind == "gravity":
        return dict(a=_gravity(x, db.L, m, db.gp), leaves=None, pairs=None, images=None)
    if kind == "reverse":
        return dict(zip(("a", "gx", "gm"), _gravity(x, db.L, m, db.gp, lambda a: 2 * a)))
    if kind == "advance":
        return _exact_advance(db, case)
    xg, hg, mg, vg, ug = x[:, gas], h[gas], m[gas], v[:, gas], u[gas]
    if kind == "chain":
        dvbar, dubar = (t.double() for t in _cotangents(n, seed))
        pairs = _pairs(xg, db.L, hg)
        xg, mg, vg, ug = (t.clone().requires_grad_(True) for t in (xg, mg, vg, ug))
        G = _Gas(xg, hg, db.L, db.hp, pairs)
        G.geometry(mg)
        G.corrections()
        dv, du = G.hydro(vg, ug)
        grads = torch.autograd.grad((dvbar[:, gas] * dv).sum() + (dubar[gas] * du).sum(), (xg, mg, vg, ug))
        return dict(zip(("x", "m", "v", "u"), map(F, grads)), dv=F(dv), du=F(du), n_singular=None)
    G = _Gas(xg, hg, db.L, db.hp)
    G.geometry(mg)
    if kind == "autograd":
        gx, gm = _geom_grad(G)
        out = dict(V=F(G.V), rho=F(G.rho))
        gx, gm = F(gx), F(gm)
        del G
        a, gx2, gm2 = _gravity(x, db.L, m, db.gp, lambda a: 2 * a)
        return dict(out, a=a, gx=gx + gx2, gm=gm + gm2)
    G.corrections()
    out = dict(V=F(G.V), rho=F(G.rho), n_singular=None)
    if kind == "hydro":
        dv, du = G.hydro(vg, ug)
        return dict(out, A=F(G.A), B=F(G.B), gA=F(G.gA), gB=F(G.gB.reshape(9, -1)), dv=F(dv), du=F(du))
    G.extras(vg)
    dv, q = G.accel(vg, ug, True)
    du = G.energy(vg, ug, vg, True)
    dt = torch.tensor([min(DT_MAX, CFL / q) if q > 0 else DT_MAX], dtype=torch.float64)
    return dict(out, rho_r=F(G.rho_r), dvdx=F(G.G.reshape(9, -1)), dv=F(dv), du=F(du), dt=dt)
