"""The work users have this library do, as cases that can be timed: steps of
the embedded-boundary advance in both precisions, its flux divergence alone,
ensembles, two-level refinement, the anelastic projection and the warm-start
network, each through the public calls of ``paper_2604_11959_gb300.eb`` (and
``amr.TwoLevel``), at the sizes of this repository's workloads, tests and
benchmark.

Inputs are seeded: terrain from ``inputs``, states built on the GPU with the
formulas of ``inputs.sheltered_state`` (stratified, calm below the terrain
top, wind above, smooth perturbations of 1 %), stored about the reference
profiles and the background wind as the benchmark stores them.  ``exact``
evaluates the flux divergence, the projection and the network in 64 bits with
plain torch operations: cut-cell fractions from clipped triangles and
segments, dense stencils, conjugate gradients, ``conv3d``.  Whole steps have
no such value: weighted state redistribution is a table-driven method of its
own (merging neighbourhoods, limited least-squares slopes), so their outputs
are compared with earlier ones only.
"""
import math

import numpy as np
import torch

from paper_2604_11959_gb300 import amr, eb, inputs, warmstart

F64 = torch.float64
LX = LY = 1.0
LZ = 0.5


def listed():
    return [
        # the smallest workload as configured: a ridge, 10 FP64 steps; launches and latency
        dict(name="step ridge 32x32x16 f64", kind="step", terrain="woa", nx=32, ny=32, nz=16, precision="f64",
             nsteps=10, stages=1),
        # a small odd-sized random terrain (no row starts aligned), one three-stage step, mixed
        dict(name="step grf 45x38x20 rk3", kind="step", terrain="grf", nx=45, ny=38, nz=20, precision="mixed",
             nsteps=1, stages=3),
        # the headline workload: one forward-Euler step of the hill, mixed, schedule tuned as the benchmark does
        dict(name="step hill 256x256x128", kind="step", terrain="gaussian", nx=256, ny=256, nz=128,
             precision="mixed", nsteps=1, stages=1, tune=True),
        # the same hill in FP64, the reference precision
        dict(name="step hill 256x256x128 f64", kind="step", terrain="gaussian", nx=256, ny=256, nz=128,
             precision="f64", nsteps=1, stages=1),
        # the compressible system: pressure gradient and buoyancy in every stage, three stages, untuned
        dict(name="step hill sources rk3", kind="step", terrain="gaussian", nx=256, ny=256, nz=128,
             precision="mixed", nsteps=1, stages=3, sources=True),
        # the largest workload: rough random terrain with tiny cut cells, one three-stage step, tuned
        dict(name="step grf 512x512x256 rk3", kind="step", terrain="grf", nx=512, ny=512, nz=256,
             precision="mixed", nsteps=1, stages=3, tune=True, tiny=16),
        # the flux divergence alone, for users with their own time integrator; sizes no tile divides; FP64 on the
        # ridge, because without the redistribution that follows it a sliver's value is rounding over its volume
        dict(name="flux ridge 250x190x98 f64", kind="flux", terrain="woa", nx=250, ny=190, nz=98, precision="f64"),
        # batched serving: uneven hills (the first of the 64 configured members) advanced 10 steps, tuned
        dict(name="ensemble 12 hills", kind="ensemble", members=12, first=0, nsteps=10, precision="mixed"),
        # one coupled step of two refinement levels, a quarter of the columns refined
        dict(name="two levels 256x256x128", kind="levels", terrain="gaussian", nx=256, ny=256, nz=128, lo=96,
             hi=160, precision="mixed", stages=1),
        # the anelastic projection at its configured size, multigrid preconditioner, to 1e-10
        dict(name="project grf 192x192x96 mg", kind="project", terrain="grf", nx=192, ny=192, nz=96,
             precision="mixed", precond="mg"),
        # the warm-start network on the projection's grid: inference
        dict(name="network 192x192x96", kind="forward", nx=192, ny=192, nz=96),
        # and the gradient of its loss on the training grid
        dict(name="network gradient 96x96x48", kind="gradient", nx=96, ny=96, nz=48),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "flux", "flux", "ensemble", "levels", "project", "forward", "gradient"])
    if kind in ("step", "flux"):
        nx, ny, nz = _log_int(rng, 24, 400), _log_int(rng, 24, 400), _log_int(rng, 12, 160)
        c = dict(kind=kind, terrain="woa" if kind == "flux" else rng.choice(["gaussian", "grf", "grf", "woa"]),
                 nx=nx, ny=ny, nz=nz,
                 precision="f64" if kind == "flux" else rng.choice(["mixed", "mixed", "f64"]))
        if kind == "step":
            c.update(nsteps=rng.choice([1, 1, 2, 5]), stages=rng.choice([1, 3]))
            c["sources"] = rng.random() < 0.25
            c["tune"] = rng.random() < 0.25
        most = 8_000_000 if c["precision"] == "f64" else 100_000_000   # a pass stays below the largest listed one
        while nx * ny * nz * c.get("nsteps", 1) * c.get("stages", 1) > most:
            if c.get("nsteps", 1) > 1:
                c["nsteps"] = 1
            else:
                c["nx"], c["ny"], c["nz"] = nx, ny, nz = max(24, 4 * nx // 5), max(24, 4 * ny // 5), max(12, 4 * nz // 5)
        return c
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randint(2, 10), first=rng.randint(0, 54), nsteps=rng.randint(1, 10),
                    precision="mixed")
    if kind == "levels":
        nx = 2 * _log_int(rng, 48, 140)
        lo = 2 * rng.randint(0, nx // 2 - 1)
        width = 2 * rng.randint(4, max(4, (nx - 50) // 4))
        return dict(kind=kind, terrain=rng.choice(["gaussian", "grf"]), nx=nx, ny=2 * _log_int(rng, 16, 128),
                    nz=2 * _log_int(rng, 8, 64), lo=lo, hi=lo + width, precision="mixed", stages=rng.choice([1, 3]))
    if kind == "project":
        if rng.random() < 0.5:
            m = 16 if rng.random() < 0.5 else 4
            nx, ny, nz = (m * _log_int(rng, a // m, b // m) for a, b in ((32, 176), (32, 176), (16, 96)))
            return dict(kind=kind, terrain="grf", nx=nx, ny=ny, nz=nz, precision="mixed", precond="mg")
        return dict(kind=kind, terrain="grf", nx=_log_int(rng, 20, 56), ny=_log_int(rng, 20, 56),
                    nz=_log_int(rng, 12, 28), precision=rng.choice(["mixed", "f64"]), precond="jacobi")
    top = 160 if kind == "forward" else 96
    return dict(kind=kind, nx=4 * _log_int(rng, 4, top // 4), ny=4 * _log_int(rng, 4, top // 4),
                nz=4 * _log_int(rng, 2, top // 8))


# ---- inputs -----------------------------------------------------------------

def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _workload(case, seed):
    t = case["terrain"]
    return inputs.Workload("case", case["nx"], case["ny"], case["nz"], 1, terrain=t, seed=int(seed) % (1 << 31),
                           hmax=0.1 if t == "woa" else 0.15 if t == "gaussian" else 0.2, tiny=case.get("tiny", 0))


def _fields(w, seed, refs):
    """The sheltered state of the workload, stored about the profiles refs
    (rho0, rho0 theta0, background rho*u, rho*v), FP64 on the GPU."""
    rng = np.random.default_rng([int(seed), w.nx, w.ny, w.nz])
    nz, ny, nx = w.nz, w.ny, w.nx
    x = (torch.arange(nx, dtype=F64, device="cuda") + 0.5) / nx
    y = (torch.arange(ny, dtype=F64, device="cuda") + 0.5) / ny
    zc = (torch.arange(nz, dtype=F64, device="cuda") + 0.5) / nz
    zw = torch.arange(nz + 1, dtype=F64, device="cuda") / nz

    def smooth(z):
        """Six Fourier modes with wavenumbers up to 3."""
        f = torch.zeros(len(z), ny, nx, dtype=F64, device="cuda")
        for _ in range(6):
            kx, ky, kz = (int(v) for v in rng.integers(0, 4, 3))
            px, py, pz = rng.uniform(0, 2 * np.pi, 3)
            a = rng.uniform(-1, 1) / 6
            yx = torch.cos(2 * np.pi * ky * y + py)[:, None] * torch.cos(2 * np.pi * kx * x + px)[None, :]
            f.addcmul_(torch.cos(2 * np.pi * kz * z + pz)[:, None, None], yx[None], value=a)
        return f

    r0n, rt0n = inputs.cell_reference(nz, w.Lz)
    r0, rt0 = _cuda(r0n)[:, None, None], _cuda(rt0n)[:, None, None]
    rw = _cuda(np.concatenate([[r0n[0]], 0.5 * (r0n[:-1] + r0n[1:]), [r0n[-1]]]))[:, None, None]
    dz = w.Lz / nz
    ramp = torch.clamp((zc * w.Lz - (w.hmax + dz)) / (8 * dz), 0.0, 1.0)[:, None, None]
    pert = 1e-2
    U = {"rho": r0 * (1.0 + 0.1 * pert * smooth(zc)), "rhotheta": rt0 * (1.0 + pert * smooth(zc)),
         "rhou": r0 * (ramp + pert * smooth(zc)), "rhov": r0 * (pert * smooth(zc)),
         "rhow": rw * (pert * smooth(zw))}
    U["rhow"][0] = 0.0
    U["rhow"][nz] = 0.0
    for f, r in zip(("rho", "rhotheta", "rhou", "rhov"), refs):
        if r is not None:
            U[f] -= _cuda(r)[:, None, None]
    return U


def _stored(U, precision):
    return {f: t if precision == "f64" else t.float() for f, t in U.items()}


def _geometry(w, precision, refs):
    kw = {k: _cuda(r) for k, r in zip(("ref_rho", "ref_rhotheta", "ref_rhou", "ref_rhov"), refs) if r is not None}
    return eb.Geometry(w.nx, w.ny, w.nz, w.Lx, w.Ly, w.Lz, _cuda(w.heights()), precision=precision, **kw)


def _dt(case, w):
    dt = w.dt()
    return dt / 400.0 if case.get("sources") else dt   # sound travels at about 350 u0


def _network(case, seed):
    """Network inputs of the projection's kind (a right-hand side over its
    RMS, the volume fraction), a smooth target, the mask of the fluid cells
    and He-normal parameters."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng([int(seed), nx, ny, nz])
    h = _cuda(inputs.grf_terrain(nx, ny, int(seed) % (1 << 31), hmax=0.3 * nz)[:ny, :nx])
    k = torch.arange(nz, dtype=F64, device="cuda")[:, None, None]
    alpha = torch.clamp(k + 1 - h, 0.0, 1.0)
    mask = (alpha > 0).to(F64)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rhs = torch.randn(nz, ny, nx, dtype=F64, device="cuda", generator=g)
    rhs *= mask * torch.exp(-((k - h) / (0.2 * nz)) ** 2)   # the divergence sits near the terrain
    rhs /= rhs.square().sum().div(mask.sum()).sqrt()
    ph = rng.uniform(0, 2 * np.pi, 3)
    t = (torch.cos(2 * np.pi * k / nz + ph[0])
         * torch.cos(2 * np.pi * torch.arange(ny, dtype=F64, device="cuda") / ny + ph[1])[:, None]
         * torch.cos(2 * np.pi * torch.arange(nx, dtype=F64, device="cuda") / nx + ph[2]))
    p = warmstart.init_params(int(seed) % (1 << 31))
    return torch.stack([rhs, alpha]).float(), (t * mask).float(), mask.float(), p


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        x, t, m, p = _network(case, seed)
        net = eb.UNet(case["nx"], case["ny"], case["nz"])
        net.set_params(p)
        s = dict(kind=kind, net=net, x=x, t=t, m=m)
        if kind == "forward":
            s["out"] = torch.empty_like(t)
        return s
    if kind == "ensemble":
        geoms, states, dts = [], [], []
        for b in range(case["first"], case["first"] + case["members"]):
            nx, ny, nz, h0, sig = inputs.ensemble_members()[b]
            w = inputs.Workload("member", nx, ny, nz, 1, terrain="gaussian", hmax=h0, sigma=sig)
            refs = w.references("sheltered")
            geoms.append(_geometry(w, case["precision"], refs))
            states.append(_stored(_fields(w, seed + b, refs), case["precision"]))
            dts.append(w.dt())
        ens = eb.Ensemble(geoms)
        for q, U in enumerate(states):
            ens.set_state(q, U)
        ens.tune(dts, reps=2)
        return dict(kind=kind, ens=ens, geoms=geoms, states=states, dts=dts, nsteps=case["nsteps"],
                    out=[g.empty_state() for g in geoms])
    w = _workload(case, seed)
    if kind == "levels":
        refs = w.references("sheltered")
        wc = inputs.Workload("coarse", w.nx // 2, w.ny // 2, w.nz // 2, 1, terrain=w.terrain, hmax=w.hmax)
        crefs = list(inputs.cell_reference(wc.nz, w.Lz)) + list(inputs.background_momentum(
            wc.nz, w.Lz, z_calm=w.hmax + w.Lz / w.nz, ramp=8 * w.Lz / w.nz))
        halo = amr.HALO_EULER if case["stages"] == 1 else amr.HALO_RK3
        lv = amr.TwoLevel(eb, w.nx, w.ny, w.nz, w.Lx, w.Ly, w.Lz, w.heights(), case["lo"], case["hi"], halo,
                          precision=case["precision"], refs_fine=refs, refs_coarse=crefs)
        Uc = _stored(_fields(wc, seed, crefs), case["precision"])
        Uf = lv.fill(Uc, lv.patch.empty_state())
        return dict(kind=kind, lv=lv, Uc=Uc, Uf=Uf, dt=w.dt(), stages=case["stages"])
    if kind == "project":
        refs = inputs.cell_reference(w.nz, w.Lz) + (None, None)   # full momenta
        g = _geometry(w, case["precision"], refs)
        eb.set_preconditioner(g, case["precond"])
        U = _stored(_fields(w, seed, refs), case["precision"])
        U["rho"].zero_()
        return dict(kind=kind, g=g, U=U, P=g.empty_state(), dt=w.dt())
    refs = w.references("sheltered")
    g = _geometry(w, case["precision"], refs)
    U = _stored(_fields(w, seed, refs), case["precision"])
    if case.get("tune"):
        eb.tune(g, U, w.dt(), reps=3)
    if case.get("sources"):
        g.set_sources()
    return dict(kind=kind, g=g, U=U, out=g.empty_state(), dt=_dt(case, w), nsteps=case.get("nsteps"),
                stages=case.get("stages"))


def run(s):
    kind = s["kind"]
    if kind == "step":
        return eb.step(s["g"], s["U"], s["dt"], s["nsteps"], s["stages"], out=s["out"])
    if kind == "flux":
        return eb.flux_div(s["g"], s["U"], out=s["out"])
    if kind == "ensemble":
        for q, U in enumerate(s["states"]):
            s["ens"].set_state(q, U)
        s["ens"].step(s["dts"], s["nsteps"])
        return [s["ens"].get_state(q, out=o) for q, o in enumerate(s["out"])]
    if kind == "levels":
        return s["lv"].step(s["Uc"], s["Uf"], s["dt"], s["stages"])
    if kind == "project":   # in place: on a copy of the provisional momenta
        for f in ("rhou", "rhov", "rhow"):
            s["P"][f].copy_(s["U"][f])
        eb.project(s["g"], s["P"], s["dt"], rtol=1e-10)
        return {f: s["P"][f] for f in ("rhou", "rhov", "rhow")}
    if kind == "forward":
        return s["net"].forward(s["x"], out=s["out"])
    return s["net"].gradient(s["x"], s["t"], s["m"])


def _network_flops(case):
    """Multiply-adds of the network's layers, two operations each."""
    n = case["nx"] * case["ny"] * case["nz"]
    at = [1, 1, 8, 8, 64, 64, 8, 8, 1, 1, 1]
    return sum(2.0 * ci * co * k ** 3 * n / a for (ci, co, k), a in zip(warmstart.LAYERS, at))


def work(case):
    """Every stage reads the state and writes the next one (states outgrow
    the caches); about 300 operations per cell and stage (four advected
    quantities, three faces each).  The projection counts 13 iterations of
    conjugate gradients with one smoothing pass each."""
    kind = case["kind"]
    es = 8 if case.get("precision") == "f64" else 4
    if kind == "ensemble":
        ms = inputs.ensemble_members()[case["first"]:case["first"] + case["members"]]
        n = sum(m[0] * m[1] * m[2] for m in ms)
        return {"bytes": 10.0 * es * n * case["nsteps"], "flops": 300.0 * n * case["nsteps"]}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "step":
        q = case["nsteps"] * case["stages"]
        extra = 5 * es * n * case["nsteps"] * 2 if case["stages"] == 3 else 0   # stages 2, 3 also read the step's start
        return {"bytes": 10.0 * es * n * q + extra, "flops": 300.0 * n * q}
    if kind == "flux":
        return {"bytes": 10.0 * es * n, "flops": 300.0 * n}
    if kind == "levels":
        m = n / 8 + n * (case["hi"] - case["lo"]) / case["nx"]
        return {"bytes": 10.0 * es * m * case["stages"], "flops": 300.0 * m * case["stages"]}
    if kind == "project":
        it = 13 if case["precond"] == "mg" else 4 * max(case["nx"], case["ny"], case["nz"])
        return {"bytes": 6.0 * es * n + it * 100.0 * n, "flops": it * 60.0 * n}
    if kind == "forward":
        return {"bytes": 12.0 * n, "flops": _network_flops(case)}
    return {"bytes": 16.0 * n, "flops": 3.0 * _network_flops(case)}


# ---- 64-bit values ------------------------------------------------------------
# Grids: 0 cells, 1 / 2 / 3 the x / y / z faces' control volumes.  Arrays are
# (levels, ny, nx); lengths in cell units.

def _shift(a, d, s):
    """a at the position s steps along direction d (0 x, 1 y, 2 z): periodic
    in x and y, zero beyond the array in z."""
    if d < 2:
        return torch.roll(a, -s, 2 - d)
    if s == 0:
        return a
    z = torch.zeros_like(a[: abs(s)])
    return torch.cat([a[s:], z]) if s > 0 else torch.cat([z, a[:s]])


def _segment(Ha, Hb, sa, sb, Z):
    """Over the part of a segment with H < Z: integrals of u = Z - H, of s u
    and of u^2 / 2, with s from sa to sb (two-point Gauss, exact for cubics)."""
    ua, ub = Z - Ha, Z - Hb
    t = torch.where(ua != ub, ua / (ua - ub), torch.zeros_like(ua))
    t0 = torch.where((ua <= 0) & (ub > 0), t, torch.zeros_like(ua))
    t1 = torch.where((ua > 0) & (ub <= 0), t, torch.ones_like(ua))
    t1 = torch.where((ua <= 0) & (ub <= 0), t0, t1)
    I = [0.0, 0.0, 0.0]
    for q in (0.5 - math.sqrt(3) / 6, 0.5 + math.sqrt(3) / 6):
        tq = t0 + (t1 - t0) * q
        u, s, wt = ua + tq * (ub - ua), sa + tq * (sb - sa), 0.5 * (t1 - t0) * (sb - sa)
        I = [I[0] + wt * u, I[1] + wt * s * u, I[2] + wt * 0.5 * u * u]
    return I


def _triangle(v, Z):
    """Over the part of a triangle (three (x, y, H)) with H < Z: its area and
    the integrals of x, y and Z - H."""
    H = torch.stack([p[2] for p in v])
    H, order = torch.sort(H, 0)
    x = torch.tensor([p[0] for p in v], dtype=F64, device="cuda")[order]
    y = torch.tensor([p[1] for p in v], dtype=F64, device="cuda")[order]
    (xa, ya), (xb, yb), (xc, yc) = ((p[0], p[1]) for p in v)
    A = 0.5 * abs((xb - xa) * (yc - ya) - (xc - xa) * (yb - ya))
    u = [Z - H[q] for q in range(3)]          # u0 >= u1 >= u2

    def corner(a, b, c):
        """The triangle at vertex a cut off where u vanishes on the edges to b and c."""
        fb = torch.where(u[a] != u[b], u[a] / (u[a] - u[b]), torch.zeros_like(u[a]))
        fc = torch.where(u[a] != u[c], u[a] / (u[a] - u[c]), torch.zeros_like(u[a]))
        ar = A * fb * fc
        mean = lambda w: w[a] + (fb * (w[b] - w[a]) + fc * (w[c] - w[a])) / 3
        return [ar, ar * mean(x), ar * mean(y), ar * u[a] / 3]

    one = torch.ones_like(u[0])
    whole = [A * one, A * one * x.mean(0), A * one * y.mean(0), A * (u[0] + u[1] + u[2]) / 3]
    low, high = corner(0, 1, 2), corner(2, 0, 1)
    out = []
    for q in range(4):
        r = torch.where(u[2] >= 0, whole[q], torch.where(u[1] > 0, whole[q] - high[q], low[q]))
        out.append(torch.where(u[0] <= 0, torch.zeros_like(r), r))
    return out


class _Cut:
    """Volume fractions, low-face fractions and face centroids of the four
    grids above the piecewise-linear terrain (each lattice square split along
    its (0,0)-(1,1) diagonal)."""

    def __init__(self, w, grids):
        h = _cuda(w.heights()) * (w.nz / w.Lz)
        a, b, c, d = h[:-1, :-1], h[:-1, 1:], h[1:, :-1], h[1:, 1:]
        # heights on the 3 x 3 half lattice of every cell, [x half][y half]
        self.H = [[a, 0.5 * (a + c), c], [0.5 * (a + b), 0.5 * (a + d), 0.5 * (c + d)], [b, 0.5 * (b + d), d]]
        self.nz = w.nz
        self.top = min(w.nz, int(float(h.max())) + 2)   # first level that is regular everywhere
        self.alpha, self.beta, self.cent = {}, {}, {}
        for g in grids:
            self._grid(g, w.ny, w.nx)

    def _halves(self, g, d):
        """(cell offset, half indices) the CV of grid g covers along axis d."""
        return [(-1, 1), (0, 0)] if g == d + 1 else [(0, 0), (0, 1)]

    def _at(self, hx, hy, ox, oy):
        return torch.roll(self.H[hx][hy], (-oy, -ox), (0, 1))

    def _area(self, g, Z):
        """Over the footprint of the CVs of grid g, centred: area below Z, its x, y moments, volume below Z."""
        tot = None
        for ox, a in self._halves(g, 0):
            for oy, b in self._halves(g, 1):
                p = lambda i, j: (0.5 * (a + i) + ox - (0.0 if g == 1 else 0.5),
                                  0.5 * (b + j) + oy - (0.0 if g == 2 else 0.5),
                                  self._at(a + i, b + j, ox, oy)[None])
                for tri in ((p(0, 0), p(1, 0), p(1, 1)), (p(0, 0), p(1, 1), p(0, 1))):
                    r = _triangle(tri, Z)
                    tot = r if tot is None else [s + t for s, t in zip(tot, r)]
        return tot

    def _side(self, g, d, Z0, Z1, zc):
        """The low vertical d-face (d 0 or 1): area, transverse and z moments."""
        ox, a = (-1, 1) if g == d + 1 else (0, 0)
        t = 1 - d
        A = S = M = 0.0
        for oy, b in self._halves(g, t):
            ends = []
            for e in (0, 1):
                i, j = (a, b + e) if d == 0 else (b + e, a)
                o = (ox, oy) if d == 0 else (oy, ox)
                ends.append(self._at(i, j, *o)[None])
            s0 = 0.5 * b + oy - (0.0 if g == t + 1 else 0.5)
            hi, lo = _segment(*ends, s0, s0 + 0.5, Z1), _segment(*ends, s0, s0 + 0.5, Z0)
            A = A + hi[0] - lo[0]
            S = S + hi[1] - lo[1]
            M = M + (Z1 - zc) * hi[0] - (Z0 - zc) * lo[0] - (hi[2] - lo[2])
        return A, S, M

    def _grid(self, g, ny, nx):
        K = self.top + 1
        nzg = self.nz + (g == 3)
        k = torch.arange(K, dtype=F64, device="cuda")[:, None, None]
        half = 0.5 if g == 3 else 0.0
        Z0, Z1 = torch.clamp(k - half, min=0.0), torch.clamp(k + 1 - half, max=float(self.nz))
        zc = k if g == 3 else k + 0.5
        lo, hi = self._area(g, Z0), self._area(g, Z1)
        alpha = torch.clamp(hi[3] - lo[3], 0.0, 1.0)
        alpha = torch.where(alpha < 1e-13, torch.zeros_like(alpha), alpha)
        beta, cent = [], []
        for d in range(3):
            if d < 2:
                A, S, M = self._side(g, d, Z0, Z1, zc)
            else:
                A, S, M = lo[0], lo[1], lo[2]
                if g == 3:
                    A = torch.cat([torch.zeros_like(A[:1]), A[1:]])   # below the floor
            A = torch.where(A < 1e-13, torch.zeros_like(A), A)
            pos = A > 0
            ctr = [torch.where(pos, q / torch.where(pos, A, torch.ones_like(A)), torch.zeros_like(A)) for q in (S, M)]
            # a face with open area and a centroid within rounding of its centre is a whole face
            beta.append(A)
            cent.append([torch.where(c.abs() < 1e-12, torch.zeros_like(c), c) for c in ctr])

        def dense(a, fill):
            out = torch.full((nzg, ny, nx), fill, dtype=F64, device="cuda")
            n = min(K, nzg)
            out[:n] = a[:n]
            return out

        self.alpha[g] = dense(alpha, 1.0)
        self.beta[g] = [dense(b, 1.0) for b in beta]
        self.cent[g] = [[dense(c, 0.0) for c in cs] for cs in cent]
        if g == 3:   # the upper half of the highest CV lies above the lid
            self.alpha[g][self.nz] = torch.minimum(self.alpha[g][self.nz], torch.full_like(self.alpha[g][0], 0.5))
            for d in range(2):
                self.beta[g][d][self.nz] = torch.minimum(self.beta[g][d][self.nz],
                                                         torch.full_like(self.alpha[g][0], 0.5))


def _levels(a, n):
    """a with n levels: cut, or zeros added on top."""
    return a[:n] if a.shape[0] >= n else torch.cat([a, torch.zeros_like(a[: n - a.shape[0]])])


def _exact_flux(case, seed):
    w = _workload(case, seed)
    refs = w.references("sheltered")
    U = {f: t.double() for f, t in _stored(_fields(w, seed, refs), case["precision"]).items()}
    for f, r in zip(("rho", "rhotheta", "rhou", "rhov"), refs):
        U[f] = U[f] + _cuda(r)[:, None, None]
    G = _Cut(w, (0, 1, 2, 3))
    nz = w.nz
    delta = (w.Lx / w.nx, w.Ly / w.ny, w.Lz / nz)
    fluid = {g: G.alpha[g] > 0 for g in range(4)}
    mom = {g: torch.where(fluid[g], U[f], torch.zeros_like(U[f])) for g, f in ((1, "rhou"), (2, "rhov"), (3, "rhow"))}
    mom[3][0] = 0.0
    mom[3][nz] = 0.0
    rho = torch.where(fluid[0], U["rho"], torch.zeros_like(U["rho"]))
    out = {}
    for g in range(4):
        nzg = nz + (g == 3)
        S = g - 1
        # advected value: theta, or the momentum over the mean density of the fluid cells beside it
        if g == 0:
            phi = torch.where(fluid[0], U["rhotheta"] / U["rho"], torch.zeros_like(rho))
        else:
            r, c = _levels(rho, nzg), _levels(fluid[0].to(F64), nzg)
            r, c = r + _shift(r, S, -1), c + _shift(c, S, -1)
            phi = torch.where((c > 0) & fluid[g], U[("rhou", "rhov", "rhow")[S]] * c / torch.where(r > 0, r, torch.ones_like(r)),
                              torch.zeros_like(r))
            if g == 3:
                phi[0] = 0.0
                phi[nz] = 0.0
        div_m = div_p = 0.0
        for d in range(3):
            m = _levels(mom[d + 1], nzg)
            if g:
                m = 0.5 * (m + _shift(m, S, -1))   # S == d when the face lies at a cell centre
            f = fluid[g]
            beta = G.beta[g][d]
            on = (beta > 0) & f & _shift(f, d, -1)
            m = torch.where(on, m, torch.zeros_like(m))
            pL, pR, pLL, pRR = _shift(phi, d, -1), phi, _shift(phi, d, -2), _shift(phi, d, 1)
            mid = 0.5 * (pL + pR)
            up = torch.where(m > 0, torch.where(_shift(f, d, -2), (5 * pL + 2 * pR - pLL) / 6, mid),
                             torch.where(_shift(f, d, 1), (5 * pR + 2 * pL - pRR) / 6, mid))
            usable = beta > 0
            if g == 3 and d != 2:
                usable = usable.clone()
                usable[0] = False
                usable[nz] = False
            if g != 3 and d == 2:
                usable = usable.clone()
                usable[0] = False
            ta, tb = (1, 2) if d == 0 else (0, 2) if d == 1 else (0, 1)
            ga, gb = G.cent[g][d]

            def toward(a, ca, cb):
                """a at the neighbours toward the face centroid: along the first, second and both transverse axes."""
                pa, na = _shift(a, ta, 1), _shift(a, ta, -1)
                side = lambda p, n, t, c: torch.where(c >= 0, p, n)
                va = torch.where(ca >= 0, pa, na)
                vb = torch.where(cb >= 0, _shift(a, tb, 1), _shift(a, tb, -1))
                vab = torch.where(ca >= 0, torch.where(cb >= 0, _shift(pa, tb, 1), _shift(pa, tb, -1)),
                                  torch.where(cb >= 0, _shift(na, tb, 1), _shift(na, tb, -1)))
                return va, vb, vab

            ua, ub, uab = toward(usable, ga, gb)
            both = (ga == 0) | (gb == 0) | uab
            wa = torch.where(ua & both, ga.abs(), torch.zeros_like(ga))
            wb = torch.where(ub & both, gb.abs(), torch.zeros_like(gb))

            def centroid(F):
                a, b, ab = toward(F, ga, gb)
                F = (1 - wa) * (1 - wb) * F + wa * (1 - wb) * a + wb * (1 - wa) * b + wa * wb * ab
                F = beta * F
                return (_shift(F, d, 1) - F) / delta[d]

            div_p = div_p + centroid(m * up)
            if g == 0:
                div_m = div_m + centroid(m)
        ok = fluid[g].clone()
        if g == 3:
            ok[0] = False
            ok[nz] = False
        a = torch.where(ok, G.alpha[g], torch.ones_like(G.alpha[g]))
        res = lambda v: torch.where(ok, -v / a, torch.zeros_like(a))
        if g == 0:
            out["rho"] = res(div_m)
        out[("rhotheta", "rhou", "rhov", "rhow")[g]] = res(div_p)
    return {f: out[f] for f in eb.FIELDS}


def _exact_project(case, seed):
    w = _workload(case, seed)
    refs = inputs.cell_reference(w.nz, w.Lz) + (None, None)
    U = {f: t.double() for f, t in _stored(_fields(w, seed, refs), case["precision"]).items()}
    G = _Cut(w, (0,))
    delta = (w.Lx / w.nx, w.Ly / w.ny, w.Lz / w.nz)
    dt = w.dt()
    b = [q.clone() for q in G.beta[0]]
    b[2][0] = 0.0
    m = [U["rhou"], U["rhov"], U["rhow"][: w.nz]]
    high = lambda a, d: _shift(a, d, 1)
    div = lambda f: sum((high(f[d], d) - f[d]) / delta[d] for d in range(3))
    diag = sum((b[d] + high(b[d], d)) / delta[d] ** 2 for d in range(3))
    act = diag > 0
    inv = torch.where(act, 1 / torch.where(act, diag, torch.ones_like(diag)), torch.zeros_like(diag))

    def minus_l(p):
        return -div([b[d] * (p - _shift(p, d, -1)) / delta[d] for d in range(3)])

    rhs = torch.where(act, div([b[d] * m[d] for d in range(3)]) / dt, torch.zeros_like(diag))
    rhs = torch.where(act, rhs - rhs.sum() / act.sum(), torch.zeros_like(rhs))
    r = -rhs
    x, z = torch.zeros_like(r), inv * r
    p, rz = z, (r * z).sum()
    stop = 1e-24 * float(r.square().sum())
    for it in range(20000):
        q = minus_l(p)
        a = rz / (p * q).sum()
        x = x + a * p
        r = r - a * q
        if it % 50 == 49 and float(r.square().sum()) <= stop:
            break
        z = inv * r
        rz, old = (r * z).sum(), rz
        p = z + (rz / old) * p
    new = [torch.where(b[d] > 0, m[d] - dt * (x - _shift(x, d, -1)) / delta[d], m[d]) for d in range(3)]
    return {"rhou": new[0], "rhov": new[1], "rhow": torch.cat([new[2], U["rhow"][w.nz:]])}


def _exact_network(case, seed):
    x, t, m, p = _network(case, seed)
    conv, pool, up = torch.nn.functional.conv3d, torch.nn.functional.avg_pool3d, torch.nn.functional.interpolate
    grad = case["kind"] == "gradient"
    P, o = [], 0
    for ci, co, k in warmstart.LAYERS:   # the weights are used in BF16, the biases in FP32
        n = co * ci * k ** 3
        W = _cuda(p[o:o + n]).bfloat16().double().reshape(co, ci, k, k, k).requires_grad_(grad)
        b = _cuda(p[o + n:o + n + co]).double().requires_grad_(grad)
        P.append((W, b))
        o += n + co

    def layer(l, v):
        return torch.relu(conv(v, *P[l], padding=1))

    with torch.set_grad_enabled(grad):
        v = x.double()[None]
        e1 = layer(1, layer(0, v))
        e2 = layer(3, layer(2, pool(e1, 2)))
        bt = layer(5, layer(4, pool(e2, 2)))
        d2 = layer(7, layer(6, torch.cat([up(bt, scale_factor=2), e2], 1)))
        d1 = layer(9, layer(8, torch.cat([up(d2, scale_factor=2), e1], 1)))
        y = conv(d1, *P[10])[0, 0]
        if not grad:
            return y
        loss = 0.5 * (m.double() * (y - t.double()).square()).sum() / m.double().sum()
        loss.backward()
    return float(loss.detach()), torch.cat([q.grad.reshape(-1) for Wb in P for q in Wb]).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "flux":
        return _exact_flux(case, seed)
    if kind == "project":
        return _exact_project(case, seed)
    if kind in ("forward", "gradient"):
        return _exact_network(case, seed)
    return None
