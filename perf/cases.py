"""Performance cases of the implicit radiation-diffusion path.

Each case is one call, or the short sequence of calls, that a program using
this library makes, through the Python binding `nrd.Context` (which only
marshals the C ABI of include/nrd.h):

  step       one BDF2 time step: predictor, Newton solve, time derivative,
             refinement tags (what `Integrator` and `DynamicAmr` do per step)
  residual   one evaluation of F (one per predicted last Newton iterate)
  linearise  F with the frozen Jacobian and the preconditioner data (one per
             Newton iterate)
  jv         one frozen Jacobian-vector product (one per Krylov iteration)
  vcycle     one preconditioner application (one per Krylov iteration)
  adjoint    one reverse step of the differentiation path: linearise, adjoint
             solve, vector-Jacobian product
  regrid     the device side of a regrid: tags, clustering, transfer of the
             state and its history to another hierarchy

The sizes are those of the tests and the benchmark: single boxes from 32^3 to
256^3, two levels on a base of 64^3 with the Marshak band refined, three
levels of patches with ragged sides, the differentiation hierarchy on 96^3.

`exact` computes the same outputs in 64 bits with dense torch arrays, one per
level over the level's whole index space, in textbook form.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1302_6303_gb300 import nrd
from paper_1302_6303_gb300 import workloads as W

E0 = 1e-5          # cold energy (Sec. 6)
K_COND = 0.01      # conduction constant (Sec. 3.1)
R_IN = 1.0         # incoming flux at x = 0


# ------------------------------------------------------------------ the cases
def _case(kind, n, **kw):
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], levels=1, prec=32, nu1=2, nu2=2, coarse=4,
             smoother="rbgs", tile="32x4x4", dt=5e-4)
    c.update(kw)
    return c


def listed():
    out = []

    def add(name, kind, n, **kw):
        out.append(dict(_case(kind, n, **kw), name=name))

    # the smallest whole call: a small box with the default settings, where
    # launches and the host's share count
    add("step_32", "step", (32, 32, 32))
    # a 2-level step on the refined Marshak band with the schedule and tile
    # the autotuners pick there: the ordinary AMR workload
    add("step_amr2_64", "step", (64, 64, 64), levels=2, nu1=1, nu2=0, coarse=2, tile="8x8x4")
    # the largest single box, the benchmark's default workload
    add("step_256", "step", (256, 256, 256), nu1=3, nu2=3, coarse=6, tile="8x8x8")
    # an odd box: no side a multiple of any tile, default tile
    add("residual_odd", "residual", (125, 91, 77))
    # the linearisation on three levels of patches with ragged sides
    add("linearise_amr3_64", "linearise", (64, 64, 64), levels=3, tile="8x8x4", dt=1e-4)
    # the Krylov loop's operator on the largest box
    add("jv_256", "jv", (256, 256, 256), tile="8x8x8")
    # the Krylov loop's preconditioner on the largest box
    add("vcycle_256", "vcycle", (256, 256, 256), nu1=3, nu2=3, coarse=6, tile="8x8x8")
    # and on three levels of patches, with the schedule picked there
    add("vcycle_amr3_64", "vcycle", (64, 64, 64), levels=3, nu1=1, nu2=0, coarse=2,
        smoother="jacobi", tile="8x8x4", dt=1e-4)
    # the FP64 form of the preconditioner, two levels, default schedule
    add("vcycle_f64_amr2_64", "vcycle", (64, 64, 64), levels=2, prec=64)
    # one reverse step of the differentiation workload
    add("adjoint_96", "adjoint", (96, 96, 96), levels=2, dt=2.5e-4)
    # the device side of a regrid of the 2-level workload
    add("regrid_amr2_64", "regrid", (64, 64, 64), levels=2)
    return out


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sides(lo, hi, g, cube=False):
        s = [max(1, int(round(log_int(lo, hi) / g))) * g for _ in range(3)]
        return (s[0],) * 3 if cube else tuple(s)

    kind = rng.choice(["step", "step", "residual", "linearise", "jv", "jv", "vcycle", "vcycle",
                       "adjoint", "regrid"])
    kw = dict(tile=rng.choice(["32x4x4", "8x8x8", "8x8x4"]))
    levels = rng.choice([1, 1, 2, 2, 3])
    nu = rng.choice([(1, 0, 2), (1, 1, 2), (2, 1, 3), (2, 2, 4), (3, 3, 6)])
    kw.update(nu1=nu[0], nu2=nu[1], coarse=nu[2])
    kw["smoother"] = rng.choice(["rbgs", "rbgs", "rbgs", "jacobi"])
    if kind in ("residual", "linearise", "jv"):
        n = sides(24, 224, rng.choice([1, 1, 2, 8]))
    elif kind == "vcycle":
        n = sides(32, 224, rng.choice([4, 8, 8, 16]))
        kw["prec"] = rng.choice([32, 32, 32, 64])
    else:
        n = sides(32, 160, 8)
        kw["smoother"] = "rbgs"
    if kind == "adjoint":
        n, levels = sides(48, 96, 8, cube=True), 2
    elif kind == "regrid":
        n, levels = sides(32, 80, 8), 2
    elif levels == 2:
        n = tuple(min(x, 96) for x in n)
    elif levels == 3:
        n = sides(24, 64, 8, cube=True)
    kw["dt"] = 1e-4 if levels == 3 else 5e-4
    return _case(kind, n, levels=levels, **kw)


# ------------------------------------------------------------------ the inputs
def _hierarchy(case, other=False):
    """The patches of a case (fixed by its sizes); other: a regrid's target."""
    n = (case["nx"], case["ny"], case["nz"])
    rng = np.random.default_rng(7 if other else 0)
    if case["levels"] == 1:
        return W.uniform(n)
    if case["levels"] == 3:
        return W.config_batching(n[0], seed=0)[0]
    if case["kind"] == "adjoint":
        return W.config_adjoint(n[0], seed=0)[0]
    band = max(2, (3 * n[0]) // 16 if other else n[0] // 8)
    hi = (2 * band - 1, 2 * n[1] - 1, 2 * n[2] - 1)
    return W.Hierarchy(n, [[((0, 0, 0), tuple(x - 1 for x in n))],
                           W.tile_region((0, 0, 0), hi, 16, 32, rng)])


class Layout:
    """Cells of a hierarchy: their places in dense per-level arrays (z, y, x)."""

    def __init__(self, hier):
        self.n = [hier.level_n(l) for l in range(hier.nlevels)]
        self.h = [[1.0 / x for x in n] for n in self.n]
        self.L = hier.nlevels
        self.idx = []
        for l, boxes in enumerate(hier.levels):
            nx, ny, _ = self.n[l]
            part = []
            for lo, hi in boxes:
                i, j, k = (torch.arange(lo[d], hi[d] + 1, device="cuda") for d in range(3))
                part.append((i[None, None, :] + nx * (j[None, :, None] + ny * k[:, None, None]))
                            .reshape(-1))
            self.idx.append(torch.cat(part))
        self.N = sum(x.numel() for x in self.idx)
        self.off = [0]
        for x in self.idx:
            self.off.append(self.off[-1] + x.numel())

    def shape(self, l):
        return tuple(reversed(self.n[l]))

    def centres(self):
        """x, y, z of every cell in the unit cube, in layout order."""
        out = [[], [], []]
        for l, q in enumerate(self.idx):
            nx, ny, _ = self.n[l]
            for d, c in enumerate((q % nx, (q // nx) % ny, q // (nx * ny))):
                out[d].append((c.double() + 0.5) * self.h[l][d])
        return [torch.cat(o) for o in out]

    def masks(self):
        """Per level: cells present, cells covered by the next level."""
        P = [self.dense(torch.ones(self.N, device="cuda", dtype=torch.float64), 0.0)[l] > 0
             for l in range(self.L)]
        C = [P[l + 1][::2, ::2, ::2] if l + 1 < self.L else torch.zeros_like(P[l])
             for l in range(self.L)]
        return P, C

    def dense(self, v, fill):
        out = []
        for l, q in enumerate(self.idx):
            x = torch.full((math.prod(self.n[l]),), fill, dtype=v.dtype, device=v.device)
            out.append(x.index_put((q,), v[self.off[l]:self.off[l + 1]]).reshape(self.shape(l)))
        return out

    def flat(self, levels):
        return torch.cat([x.reshape(-1)[q] for x, q in zip(levels, self.idx)])


def _inputs(case, seed):
    """Material cubes (z in {1, 5, 10}) and a Marshak front in x with its
    history, from the seed."""
    hier = _hierarchy(case)
    lay = Layout(hier)
    rng = np.random.default_rng(seed)
    n = hier.n0
    lo, hi = max(1, min(n) // 16), max(1, min(n) // 6)
    cubes = W.random_cubes(rng, n, 32, lo, hi, (1.0, 5.0, 10.0))
    z = torch.from_numpy(W.material_from_cubes(hier, cubes)).cuda()
    g = torch.Generator(device="cuda").manual_seed(seed)
    x, y, zc = lay.centres()
    front, width = rng.uniform(0.12, 0.35), rng.uniform(0.05, 0.09)
    ph = rng.uniform(0, 2 * math.pi, 2)
    wob = 1 + 0.2 * torch.sin(2 * math.pi * y + ph[0]) * torch.cos(2 * math.pi * zc + ph[1])

    def state(at):
        E = E0 + (1 - E0) * 0.5 * (1 + torch.tanh((at - x) / width)) * wob
        return torch.cat([E, E ** 0.25])

    un = state(front)
    s = dict(hier=hier, lay=lay, z=z, un=un, cubes=cubes)
    if case["kind"] in ("step", "regrid"):
        # the state one step ago and the derivative now: the front moved a little
        s["unm1"] = state(front - 2.0 * case["dt"])
        s["udot"] = (un - s["unm1"]) / case["dt"]
    else:
        noise = 1 + 0.05 * (2 * torch.rand(2 * lay.N, generator=g, device="cuda",
                                           dtype=torch.float64) - 1)
        s["u"] = un * noise
        s["v"] = torch.randn(2 * lay.N, generator=g, device="cuda", dtype=torch.float64)
        if case["kind"] == "adjoint":
            s["v"] *= torch.exp(-((x - 0.4) ** 2 + (y - 0.5) ** 2 + (zc - 0.5) ** 2) / 0.02).repeat(2)
    return s


def _nmg(case):
    m = 1
    while m < 4 and all(case[k] % (1 << m) == 0 for k in ("nx", "ny", "nz")):
        m += 1
    return m


def _context(case, hier, z):
    tx, ty, tz = (int(x) for x in case["tile"].split("x"))
    ctx = nrd.Context(nmg=_nmg(case), nu1=case["nu1"], nu2=case["nu2"],
                      coarse_sweeps=case["coarse"], tile_x=tx, tile_y=ty, tile_z=tz,
                      pc_precision=nrd.PC_F32 if case["prec"] == 32 else nrd.PC_F64,
                      smoother=nrd.SMOOTH_JACOBI if case["smoother"] == "jacobi"
                      else nrd.SMOOTH_RBGS)
    ctx.set_hierarchy_from(hier)
    ctx.set_material(z)
    return ctx


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    st = dict(kind=kind, dt=case["dt"], un=s["un"])
    st["ctx"] = ctx = _context(case, s["hier"], s["z"])
    if kind == "step":
        st.update(unm1=s["unm1"], udot=s["udot"])
    elif kind == "regrid":
        st["vecs"] = torch.stack([s["un"], s["unm1"]])
        dst = _hierarchy(case, other=True)
        st["dst"] = _context(case, dst, torch.from_numpy(
            W.material_from_cubes(dst, s["cubes"])).cuda())
    else:
        st.update(u=s["u"], v=s["v"])
        if kind == "jv":
            ctx.linearise(s["u"], s["un"], 1.0, case["dt"])
        elif kind == "vcycle":
            ctx.precond_setup(s["u"], 1.0, case["dt"])
    return st


def run(st):
    ctx, kind, dt, un = st["ctx"], st["kind"], st["dt"], st["un"]
    if kind == "step":
        u = ctx.predict(un, st["unm1"], st["udot"], dt, dt)
        ctx.step_begin(u, un, st["unm1"], dt, dt)
        udot = ctx.time_derivative(u, un, st["unm1"], dt, dt)
        tags = ctx.tag(u, thr_r=0.1)
        ctx.step_end()
        return dict(u=u, udot=udot, tags=tags)
    if kind == "residual":
        return dict(F=ctx.residual(st["u"], un, 1.0, dt))
    if kind == "linearise":
        return dict(F=ctx.linearise(st["u"], un, 1.0, dt))
    if kind == "jv":
        return dict(Jv=ctx.jv(st["u"], st["v"], 1.0, dt, mode=nrd.JV_FROZEN))
    if kind == "vcycle":
        return dict(y=ctx.precond_apply(st["v"]))
    if kind == "adjoint":
        F = ctx.linearise(st["u"], un, 1.0, dt)
        lam, _ = ctx.adjoint_solve(st["v"], 1.0, dt, rtol=1e-10)
        JTl, dz = ctx.vjp(lam, 1.0, dt)
        return dict(F=F, lam=lam, JTl=JTl, dz=dz)
    # regrid
    tags = ctx.tag(un, thr_r=0.1)
    boxes = ctx.regrid_boxes(tags, tag_bits=4, buffer=1, efficiency=0.7, min_side=16,
                             max_side=32, max_levels=2)
    moved = ctx.transfer_to(st["dst"], st["vecs"])
    found = np.full((512, 6), -1, dtype=np.int64)   # the same shape for every state
    rows = [lo + hi for lev in boxes for lo, hi in lev]
    found[:len(rows)] = rows
    return dict(tags=tags, boxes=found, moved=moved)


def work(case):
    """Bytes and flops per cell of each path from its formulas (inputs read
    once, outputs written once; a division or square root one flop); a step
    with the 3 Newton and 7 Krylov iterations these steps usually take."""
    h = _hierarchy(case)
    N = float(h.ncells)
    pc = (2 * (case["nu1"] + case["nu2"]) * 15 + 40) * 8 / 7
    F, LIN, JV = 103.0, 215.0, 52.0
    kind = case["kind"]
    if kind == "step":
        return dict(bytes=N * (3 * 16 + 4 + 2 * 16 + 1), flops=N * (3 * LIN + F + 7 * (JV + pc)))
    if kind == "residual":
        return dict(bytes=N * 52, flops=N * F)
    if kind == "linearise":
        return dict(bytes=N * (52 + 3 * 6 * 8 + 24 + 24 + 12), flops=N * LIN)
    if kind == "jv":
        return dict(bytes=N * 169, flops=N * JV)
    if kind == "vcycle":
        e = case["prec"] // 8
        return dict(bytes=N * (32 + e * (3 + 6)), flops=N * pc)
    if kind == "adjoint":
        return dict(bytes=N * (3 * 16 + 4 + 3 * 16 + 8), flops=N * (LIN + 25 * (1.3 * JV + pc)))
    M = float(_hierarchy(case, other=True).ncells)
    return dict(bytes=N * (32 + 8 + 1) + M * 32, flops=N * 12 + M * 12)


# --------------------------------------------- the same in 64 bits, densely
def _dim(d):
    return 2 - d


def _lo(x, d):
    return x.narrow(_dim(d), 0, x.shape[_dim(d)] - 1)


def _hi(x, d):
    return x.narrow(_dim(d), 1, x.shape[_dim(d)] - 1)


def _step2(x, d, first=0):
    sl = [slice(None)] * 3
    sl[_dim(d)] = slice(first, None, 2)
    return x[tuple(sl)]


def _pool(x, dims):
    """Mean over pairs along each axis of dims."""
    for d in dims:
        x = 0.5 * (_step2(x, d) + _step2(x, d, 1))
    return x


def _double(x, d, linear):
    """Twice the resolution along one axis: copies, or linear with the edge
    value repeated beyond the domain."""
    m = _dim(d)
    if not linear:
        return x.repeat_interleave(2, dim=m)
    n = x.shape[m]
    lo = torch.cat([x.narrow(m, 0, 1), x.narrow(m, 0, n - 1)], m)
    hi = torch.cat([x.narrow(m, 1, n - 1), x.narrow(m, n - 1, 1)], m)
    y = torch.stack([0.75 * x + 0.25 * lo, 0.75 * x + 0.25 * hi], m + 1)
    return y.flatten(m, m + 1)


def _pad(x, d):
    """x with one zero entry before and after along d."""
    shp = list(x.shape)
    shp[_dim(d)] = 1
    end = torch.zeros(shp, dtype=x.dtype, device=x.device)
    return torch.cat([end, x, end], _dim(d))


class Dense:
    """The method on dense level arrays; boundary: Robin at x = 0."""

    def __init__(self, lay):
        self.lay = lay
        self.P, self.C = lay.masks()
        self.all = [bool(p.all()) for p in self.P]

    def composite(self, X):
        X = list(X)
        for l in range(self.lay.L - 2, -1, -1):
            X[l] = torch.where(self.C[l], _pool(X[l + 1], range(3)), X[l])
        return X

    def sides(self, X, Xc, l, d, material=False):
        """Values on both sides of the interior faces along d, with the
        coarse-fine ghost where one side is missing on the level."""
        a, b = _lo(X[l], d), _hi(X[l], d)
        if self.all[l]:
            return a, b
        up = Xc[l - 1]
        for q in range(3):
            up = _double(up, q, linear=not material and q != d)
        pa, pb = _lo(self.P[l], d), _hi(self.P[l], d)
        ga, gb = _lo(up, d), _hi(up, d)
        if not material:
            ga, gb = b / 3 + 2 * ga / 3, a / 3 + 2 * gb / 3
        return torch.where(pa, a, ga), torch.where(pb, b, gb)

    def match(self, flux):
        """Coarse faces between a covered and an uncovered cell take the mean
        of the four fine fluxes.  flux[l][d]: interior faces."""
        for l in range(self.lay.L - 2, -1, -1):
            for d in range(3):
                fine = _pool(_step2(flux[l + 1][d], d, 1), [q for q in range(3) if q != d])
                cf = _lo(self.C[l], d) != _hi(self.C[l], d)
                flux[l][d] = torch.where(cf, fine, flux[l][d])
        return flux

    def valid(self, l, d):
        return _lo(self.P[l], d) | _hi(self.P[l], d)

    def diffusivities(self, E, T, Z, l, d):
        h = self.lay.h[l][d]
        Ec, Tc = self.composite(E), self.composite(T)
        (Ea, Eb), (Ta, Tb) = self.sides(E, Ec, l, d), self.sides(T, Tc, l, d)
        za, zb = self.sides(Z, Z, l, d, material=True)
        Tf, Ef = 0.5 * (Ta + Tb), 0.5 * (Ea + Eb)
        Dh = 2 * Tf ** 3 / (3 * (za ** 3 + zb ** 3))
        DE = Dh / (1 + Dh * (Eb - Ea).abs() / (h * Ef))
        return DE, K_COND * Tf * Tf * torch.sqrt(Tf), (Eb - Ea) / h, (Tb - Ta) / h

    def residual(self, u, z, b, a0, dt):
        lay = self.lay
        N = lay.N
        E, T, Z = lay.dense(u[:N], 1.0), lay.dense(u[N:], 1.0), lay.dense(z, 1.0)
        fE, fT = [], []
        for l in range(lay.L):
            eE, eT = [], []
            for d in range(3):
                DE, DT, gE, gT = self.diffusivities(E, T, Z, l, d)
                ok = self.valid(l, d)
                eE.append(torch.where(ok, DE * gE, torch.zeros_like(gE)))
                eT.append(torch.where(ok, DT * gT, torch.zeros_like(gT)))
            fE.append(eE)
            fT.append(eT)
        fE, fT = self.match(fE), self.match(fT)
        F = []
        for field, flux in ((0, fE), (1, fT)):
            out = []
            for l in range(lay.L):
                div = 0.0
                for d in range(3):
                    h = lay.h[l][d]
                    f = _pad(flux[l][d], d)
                    if field == 0 and d == 0:
                        # the Robin face x = 0: flux D_b (2 E - 8 R) / (4 D_b + h)
                        E1, T1, Z1 = E[l][..., :1], T[l][..., :1], Z[l][..., :1]
                        Db = T1 ** 3 / (3 * Z1 ** 3)
                        f = torch.cat([Db * (2 * E1 - 8 * R_IN) / (4 * Db + h), f[..., 1:]], -1)
                    div = div + (_hi(f, d) - _lo(f, d)) / h
                c = Z[l] ** 3 / T[l] ** 3 * (T[l] ** 4 - E[l])
                x = E[l] if field == 0 else T[l]
                bb = lay.dense(b[:N] if field == 0 else b[N:], 0.0)[l]
                r = a0 * x - bb - dt * (div + (c if field == 0 else -c))
                out.append(torch.where(self.C[l], torch.zeros_like(r), r))
            F.append(lay.flat(out))
        return torch.cat(F)

    # ---- the preconditioner: FAC over the levels, multigrid on the base box
    def setup(self, u, z, dt, case):
        lay = self.lay
        N = lay.N
        E, T, Z = lay.dense(u[:N], 1.0), lay.dense(u[N:], 1.0), lay.dense(z, 1.0)
        self.case, self.beta = case, dt
        self.coef = [[None] * lay.L, [None] * lay.L]
        self.Db = [None] * lay.L
        for l in range(lay.L - 1, -1, -1):
            both = [[], []]
            for d in range(3):
                DE, DT, _, _ = self.diffusivities(E, T, Z, l, d)
                ok = self.valid(l, d)
                cov = _lo(self.C[l], d) | _hi(self.C[l], d)
                for f, D in enumerate((DE, DT)):
                    D = torch.where(ok, D, torch.zeros_like(D))
                    if l + 1 < lay.L:
                        fine = _pool(_step2(self.coef[f][l + 1][d], d, 1),
                                     [q for q in range(3) if q != d])
                        D = torch.where(cov, fine, D)
                    both[f].append(D)
            for f in range(2):
                self.coef[f][l] = both[f]
            Db = T[l][..., :1] ** 3 / (3 * Z[l][..., :1] ** 3)
            if l + 1 < lay.L:
                Db = torch.where(self.C[l][..., :1], _pool(self.Db[l + 1], (1, 2)), Db)
            self.Db[l] = Db
        # multigrid boxes below the base level: coefficients, D_b, spacings
        self.mg = []
        h, c, Db = lay.h[0], [self.coef[0][0], self.coef[1][0]], self.Db[0]
        self.mg.append((h, c, Db))
        for m in range(1, _nmg(case)):
            h = [2 * x for x in h]
            c = [[_pool(_step2(c[f][d], d, 1), [q for q in range(3) if q != d])
                  for d in range(3)] for f in range(2)]
            Db = _pool(Db, (1, 2))
            self.mg.append((h, c, Db))
        sig = z ** 3 / u[N:] ** 3
        self.sb, self.sbt = sig * dt, sig * dt * u[N:] ** 3
        self.leaf = ~torch.cat([self.C[l].reshape(-1)[q] for l, q in enumerate(lay.idx)])

    def rows(self, f, h, c, Db, there):
        """Diagonal and scaled face coefficients of I - beta div D grad on one
        level; there: cells of the level (None: all)."""
        a = [_pad(self.beta * c[d] / h[d] ** 2, d) for d in range(3)]
        dg = 1.0
        for d in range(3):
            lo, hi = _lo(a[d], d), _hi(a[d], d)
            if there is not None:
                # a missing neighbour is a coarse-fine ghost e / 3
                p = _pad(there.double(), d)
                n = there.shape[_dim(d)]
                lo = lo * (2 / 3 + p.narrow(_dim(d), 0, n) / 3)
                hi = hi * (2 / 3 + p.narrow(_dim(d), 2, n) / 3)
            dg = dg + lo + hi
        if f == 0:
            r = self.beta * 2 * Db / (h[0] * (4 * Db + h[0]))
            dg = torch.cat([dg[..., :1] + r, dg[..., 1:]], -1)
        return dg, a

    @staticmethod
    def off(a, e):
        s = 0.0
        for d in range(3):
            p = _pad(e, d)
            n = e.shape[_dim(d)]
            s = s + _lo(a[d], d) * p.narrow(_dim(d), 0, n) + _hi(a[d], d) * p.narrow(_dim(d), 2, n)
        return s

    def smooth(self, dg, a, e, f, sweeps, red_first, there):
        if self.case["smoother"] == "jacobi":
            for _ in range(sweeps):
                e = e + 6 / 7 * ((f + self.off(a, e)) / dg - e)
                e = e if there is None else torch.where(there, e, torch.zeros_like(e))
            return e
        k, j, i = torch.meshgrid(*[torch.arange(x, device="cuda") for x in e.shape],
                                 indexing="ij")
        odd = (i + j + k) % 2 == 1
        for _ in range(sweeps):
            for colour in ((0, 1) if red_first else (1, 0)):
                at = odd if colour else ~odd
                at = at if there is None else at & there
                e = torch.where(at, (f + self.off(a, e)) / dg, e)
        return e

    def multigrid(self, fld, m, f):
        h, c, Db = self.mg[m]
        dg, a = self.rows(fld, h, c[fld], Db, None)
        e = torch.zeros_like(f)
        if m == len(self.mg) - 1:
            return self.smooth(dg, a, e, f, self.case["coarse"], True, None)
        e = self.smooth(dg, a, e, f, self.case["nu1"], True, None)
        ec = self.multigrid(fld, m + 1, _pool(f - (dg * e - self.off(a, e)), range(3)))
        for d in range(3):
            ec = _double(ec, d, True)
        return self.smooth(dg, a, e + ec, f, self.case["nu2"], False, None)

    def apply_composite(self, fld, X):
        lay = self.lay
        Xc = self.composite(X)
        flux = []
        for l in range(lay.L):
            lev = []
            for d in range(3):
                xa, xb = self.sides(X, Xc, l, d)
                lev.append(self.coef[fld][l][d] * (xb - xa) / lay.h[l][d])
            flux.append(lev)
        flux = self.match(flux)
        out = []
        for l in range(lay.L):
            div = 0.0
            for d in range(3):
                f = _pad(flux[l][d], d)
                if fld == 0 and d == 0:
                    Db, x = self.Db[l], X[l][..., :1]
                    f = torch.cat([2 * Db * x / (4 * Db + lay.h[l][0]), f[..., 1:]], -1)
                div = div + (_hi(f, d) - _lo(f, d)) / lay.h[l][d]
            out.append(X[l] - self.beta * div)
        return out

    def fac(self, fld, w):
        lay = self.lay
        f = lay.dense(torch.where(self.leaf, w, torch.zeros_like(w)), 0.0)
        U = [torch.zeros_like(x) for x in f]

        def resid():
            LU = self.apply_composite(fld, U)
            return self.composite([torch.where(p & ~c, x - y, torch.zeros_like(x))
                                   for x, y, p, c in zip(f, LU, self.P, self.C)])

        def correct(l, e):
            for m in range(l, lay.L):
                if m > l:
                    for d in range(3):
                        e = _double(e, d, True)
                    e = torch.where(self.P[m], e, torch.zeros_like(e))
                U[m] = U[m] + torch.where(self.P[m] & ~self.C[m], e, torch.zeros_like(e))

        def level(l, sweeps, red_first):
            dg, a = self.rows(fld, lay.h[l], self.coef[fld][l], self.Db[l], self.P[l])
            r = resid()[l]
            correct(l, self.smooth(dg, a, torch.zeros_like(r), r, sweeps, red_first, self.P[l]))

        for l in range(lay.L - 1, 0, -1):
            level(l, self.case["nu1"], True)
        correct(0, self.multigrid(fld, 0, resid()[0]))
        for l in range(1, lay.L):
            level(l, self.case["nu2"], False)
        return torch.where(self.leaf, lay.flat(U), torch.zeros_like(w))

    def precondition(self, w, transposed=False):
        N = self.lay.N
        sb, sbt = self.sb, self.sbt
        det = 1 + sb + sbt
        wE, wT = w[:N], w[N:]
        if transposed:
            wE, wT = ((1 + sbt) * wE + sb * wT) / det, (sbt * wE + (1 + sb) * wT) / det
        zE, zT = self.fac(0, wE), self.fac(1, wT)
        if transposed:
            return torch.cat([zE, zT])
        y = torch.cat([((1 + sbt) * zE + sbt * zT) / det, (sb * zE + (1 + sb) * zT) / det])
        return torch.where(self.leaf.repeat(2), y, torch.zeros_like(y))

    def solve(self, A, rhs, tol, its, transposed=False):
        """Flexible GMRES for A x = rhs."""
        V, Z, H = [rhs / rhs.norm()], [], np.zeros((its + 1, its))
        g = np.zeros(its + 1)
        g[0] = float(rhs.norm())
        for j in range(its):
            Z.append(self.precondition(V[j], transposed))
            w = A(Z[j])
            for _ in range(2):
                for i in range(j + 1):
                    q = float(torch.dot(V[i], w))
                    H[i, j] += q
                    w = w - q * V[i]
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
            y, _, _, _ = np.linalg.lstsq(H[:j + 2, :j + 1], g[:j + 2], rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - g[:j + 2]) <= tol * g[0]:
                break
        return sum(c * q for c, q in zip(y, Z))

    def newton(self, u, z, b, a0, dt, case):
        """F(u) = 0 to rounding."""
        self.setup(u, z, dt / a0, case)
        F = self.residual(u, z, b, a0, dt)
        first = last = float(F.norm())
        for _ in range(14):
            J = lambda v: torch.func.jvp(  # noqa: E731
                lambda q: self.residual(q, z, b, a0, dt), (u,), (v,))[1]
            dx = self.solve(J, -F, 1e-3, 12)
            neg = dx < 0
            lam = min(1.0, 0.9 * float((u[neg] / -dx[neg]).min())) if bool(neg.any()) else 1.0
            new = u + lam * dx
            F = self.residual(new, z, b, a0, dt)
            now = float(F.norm())
            if now >= 0.5 * last and last < 1e-9 * first:
                break
            u, last = new, now
            if last <= 1e-14 * first:
                break
            self.setup(u, z, dt / a0, case)
        N = self.lay.N
        return torch.cat([self.lay.flat(self.composite(self.lay.dense(u[f * N:(f + 1) * N], 0.0)))
                          for f in range(2)])


def _transfer(src, dst, u):
    """Conservative linear refinement of one field: same-level cells copied,
    others from the minmod-limited reconstruction of the finest old cell."""
    D = Dense(src)
    X = D.composite(src.dense(u, 0.0))
    slopes = []
    for l in range(src.L):
        lev = []
        for d in range(3):
            step = torch.where(_lo(D.P[l], d) & _hi(D.P[l], d), _hi(X[l], d) - _lo(X[l], d),
                               torch.zeros_like(_lo(X[l], d)))
            p = _pad(step, d)
            a, b = _lo(p, d), _hi(p, d)
            lev.append(torch.where(a * b > 0, torch.sign(a) * torch.minimum(a.abs(), b.abs()),
                                   torch.zeros_like(a)))
        slopes.append(lev)
    out = []
    for l in range(dst.L):
        val = None
        for m in range(min(l, src.L - 1) + 1):
            r = 1 << (l - m)
            v, there = X[m], D.P[m]
            s = slopes[m]
            for d in range(3):
                v = v.repeat_interleave(r, dim=_dim(d))
                there = there.repeat_interleave(r, dim=_dim(d))
                s = [q.repeat_interleave(r, dim=_dim(d)) for q in s]
            if r > 1:
                for d in range(3):
                    at = (torch.arange(v.shape[_dim(d)], device="cuda") % r + 0.5) / r - 0.5
                    shp = [1, 1, 1]
                    shp[_dim(d)] = -1
                    v = v + s[d] * at.reshape(shp)
            val = v if val is None else torch.where(there, v, val)
        out.append(val)
    return dst.flat(out)


def exact(case, seed):
    kind, dt = case["kind"], case["dt"]
    s = _inputs(case, seed)
    lay = s["lay"]
    D = Dense(lay)
    z, un = s["z"].double(), s["un"]
    N = lay.N
    if kind == "step":
        b = 2 * un - 0.5 * s["unm1"]
        u = D.newton(un + 2 * dt * s["udot"] - (un - s["unm1"]), z, b, 1.5, dt, case)
        return dict(u=u, udot=(1.5 * u - 2 * un + 0.5 * s["unm1"]) / dt, tags=None)
    if kind in ("residual", "linearise"):
        return dict(F=D.residual(s["u"], z, un, 1.0, dt))
    if kind == "jv":
        return dict(Jv=torch.func.jvp(lambda q: D.residual(q, z, un, 1.0, dt), (s["u"],),
                                      (s["v"],))[1])
    if kind == "vcycle":
        D.setup(s["u"], z, dt, case)
        return dict(y=D.precondition(s["v"]))
    if kind == "adjoint":
        D.setup(s["u"], z, dt, case)
        u, zz = s["u"].clone().requires_grad_(True), z.clone().requires_grad_(True)
        F = D.residual(u, zz, un, 1.0, dt)
        live = D.leaf.repeat(2)
        back = lambda w, x: torch.autograd.grad(F, x, w, retain_graph=True)[0]  # noqa: E731
        A = lambda w: torch.where(live, back(w, u), torch.zeros_like(w))  # noqa: E731
        g = torch.where(live, s["v"], torch.zeros_like(s["v"]))
        lam = D.solve(A, g, 1e-12, 60, transposed=True)
        lam = torch.where(live, lam, torch.zeros_like(lam))
        dz = torch.where(D.leaf, back(lam, zz), torch.zeros_like(z))
        return dict(F=F.detach(), lam=lam, JTl=A(lam), dz=dz)
    dst = Layout(_hierarchy(case, other=True))
    moved = [torch.cat([_transfer(lay, dst, x[f * N:(f + 1) * N]) for f in range(2)])
             for x in (un, s["unm1"])]
    return dict(tags=None, boxes=None, moved=torch.stack(moved))
