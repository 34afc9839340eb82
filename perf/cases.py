"""The work whose time counts: the calls a simulator makes on this library.

A case is one call (or one whole time step) of the public Python interface on a
seeded synthetic model.  ``listed()`` names the cases that are always measured,
``draw()`` gives others of the same ranges, ``prepare()`` makes what a program
holds before the call, ``run()`` makes the call once, ``work()`` counts what the
call cannot do without, and ``exact()`` evaluates the same definitions plainly
in 64-bit torch tensors, with every derivative from forward-mode dual numbers.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2406_10862_gb300 import fim, ocp, workloads

RB_FT3 = 5.614583         # ft^3 per reservoir barrel
DARCY = 0.001127          # rb cP / (day psi mD ft)
GRAVITY = 1.0 / 144.0     # psi per (lb/ft^3 ft)

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest model anyone runs (the shape of SPE1): one linearisation,
        # all latency
        dict(name="linearize-300", op="linearize", nx=10, ny=10, nz=3, phases=3, undersaturated=0.0,
             face_flux=False),
        # the benchmark's layered black-oil box, with the face fluxes the
        # adjoint and the time stepper ask for
        dict(name="linearize-200k", op="linearize", nx=100, ny=100, nz=20, phases=3, undersaturated=0.0,
             face_flux=True),
        # the large oil-water model (the shape of SPE10 model 2): 2x2 blocks
        dict(name="linearize-oilwater-1122k", op="linearize", nx=60, ny=220, nz=85, phases=2, undersaturated=0.0,
             face_flux=False),
        # an ensemble of 64 uneven models linearised together (history
        # matching and uncertainty runs)
        dict(name="ensemble-64", op="ensemble", models=64, smallest=2e4, largest=4e5, sizes=4, nz=10),
        # the product a caller's own Krylov solver iterates on
        dict(name="spmv-200k", op="spmv", nx=100, ny=100, nz=20, phases=3, undersaturated=0.0, transpose=False),
        # the transposed product (adjoint solvers), oil-water
        dict(name="spmv-transposed-1122k", op="spmv", nx=60, ny=220, nz=85, phases=2, undersaturated=0.0,
             transpose=True),
        # one reverse step of history matching: every gradient of the residual
        dict(name="adjoint-100k", op="adjoint", nx=100, ny=100, nz=10, phases=3, undersaturated=0.4),
        # a whole implicit time step of the smallest model
        dict(name="newton-300", op="newton", nx=10, ny=10, nz=3, phases=3, undersaturated=0.5),
        # a whole implicit time step of the history-matching box: Newton
        # iterations of linearisation, linear solve and update
        dict(name="newton-100k", op="newton", nx=100, ny=100, nz=10, phases=3, undersaturated=0.5),
        # a whole implicit step with rate-controlled wells as unknowns
        dict(name="wells-200k", op="wells", nx=100, ny=100, nz=20, phases=3, undersaturated=0.5),
        # the linearisation in pressure and component amounts
        dict(name="amounts-200k", op="amounts", nx=100, ny=100, nz=20, phases=3, undersaturated=0.0),
        # a whole implicit-pressure explicit-composition step
        dict(name="impec-200k", op="impec", nx=100, ny=100, nz=20, phases=3, undersaturated=0.5),
    ]


def _draw_box(rng, lo, hi):
    """nx, ny, nz of a box of lo..hi cells (log-uniform), flat to deep, odd sizes included."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nz = rng.randint(1, max(1, min(60, int(n / 64))))
    area, ratio = n / nz, math.exp(rng.uniform(math.log(0.4), math.log(2.5)))
    nx = max(4, int(math.sqrt(area * ratio)))
    ny = max(4, int(area / nx))
    return dict(nx=nx, ny=ny, nz=nz)


def draw(rng):
    op = rng.choice(["linearize", "linearize", "ensemble", "spmv", "spmv", "adjoint", "newton", "wells", "amounts",
                     "impec"])
    under = rng.choice([0.0, rng.uniform(0.1, 0.9)])
    phases = rng.choice([3, 3, 2])
    if op == "ensemble":
        return dict(op=op, models=rng.randint(2, 48), smallest=2e4, largest=4e5, sizes=rng.randint(5, 10 ** 6), nz=10)
    if op == "linearize":
        return dict(op=op, phases=phases, undersaturated=under, face_flux=rng.random() < 0.5, **_draw_box(rng, 300, 1.1e6))
    if op == "spmv":
        return dict(op=op, phases=phases, undersaturated=under, transpose=rng.random() < 0.5, **_draw_box(rng, 300, 1.1e6))
    if op in ("adjoint", "amounts"):
        return dict(op=op, phases=phases, undersaturated=under, **_draw_box(rng, 300, 3e5))
    if op == "newton":
        return dict(op=op, phases=3, undersaturated=rng.uniform(0.2, 0.8), **_draw_box(rng, 300, 1e5))
    if op == "wells":
        return dict(op=op, phases=3, undersaturated=rng.uniform(0.2, 0.8), **_draw_box(rng, 1000, 1e5))
    return dict(op=op, phases=3, undersaturated=rng.uniform(0.2, 0.8), **_draw_box(rng, 300, 2e5))


# ---------------------------------------------------------------------- models
def _model(case, seed):
    """A model and a pair of states: layered permeability, wells in every
    layer (five-spot, or two opposite corners of a small box), the deepest
    part of the reservoir undersaturated where the case says so."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, phases = case["nx"], case["ny"], case["nz"], case["phases"]
    n = nx * ny * nz
    lnk = workloads.layered_lnk(rng, nx, ny, nz)
    phi = rng.uniform(0.15, 0.3, n)
    over = dict(dx=50.0, dy=50.0, dz=5.0, swc=0.2) if phases == 2 else {}
    g = workloads.make_grid(nx, ny, nz, lnk, phi, [], nphase=phases, **over)
    inject = 0 if phases == 2 else 2
    if nx >= 12 and ny >= 12:
        corners = [(i, j) for i in (4, nx - 5) for j in (4, ny - 5)]
        centre = (nx // 2 - 1, ny // 2 - 1)
    else:
        corners, centre = [(nx - 1, ny - 1)], (0, 0)
    g.wells = [workloads.Well(kind=0, phase=0, p_bh=3500.0, cells=g.column(i, j)) for i, j in corners]
    g.wells.append(workloads.Well(kind=1, phase=inject, p_bh=5500.0, cells=g.column(*centre)))
    if case["op"] in ("newton", "wells", "impec"):
        return g, _settled_state(g, rng, case["undersaturated"])
    s = workloads.perturbed_state(g, rng, sw0=0.2 if phases == 2 else 0.12)
    if phases == 3 and case["undersaturated"] > 0.0:
        deep = np.arange(n) >= (1.0 - case["undersaturated"]) * n
        rs = rng.uniform(0.3, 0.7, n) * float(np.max(g.tab_Rs))
        for u, flag, f in ((s.u_old, s.flag_old, 1.0), (s.u_new, s.flag_new, rng.uniform(0.97, 1.03, n))):
            u[2, deep] = (rs * f)[deep]
            flag[deep] = 1
    return g, s


def _settled_state(g, rng, undersaturated):
    """The state a time step starts from: pressure growing with depth (and a
    little from cell to cell), a gas cap above undersaturated oil; the step
    is a quarter of a day, as after a change of the wells."""
    n = g.N
    depth = np.arange(n) // (g.nx * g.ny) * g.dz
    u = np.zeros((3, n))
    u[0] = 4800.0 + 0.3 * depth + rng.normal(0.0, 2.0, n)
    u[1] = 0.12 + rng.uniform(0.0, 0.1, n)
    flag = (np.arange(n) >= (1.0 - undersaturated) * n).astype(np.int8)
    rs = (0.7 + rng.uniform(-0.05, 0.05, n)) * 0.3 * 4800.0
    u[2] = np.where(flag == 1, rs, rng.uniform(0.03, 0.1, n))
    return workloads.State(u_new=u.copy(), flag_new=flag.copy(), u_old=u, flag_old=flag, dt=0.25)


def _ensemble(case, seed):
    sizes = random.Random(case["sizes"])
    out = []
    for m in range(case["models"]):
        n = math.exp(sizes.uniform(math.log(case["smallest"]), math.log(case["largest"])))
        nz = case["nz"]
        nx = max(2, int(round(math.sqrt(n / nz))))
        ny = max(2, int(round(n / (nz * nx))))
        rng = np.random.default_rng([seed, m])
        g = workloads.make_grid(nx, ny, nz, rng.normal(math.log(100.0), 1.5, nx * ny * nz),
                                rng.uniform(0.15, 0.3, nx * ny * nz), [])
        g.wells = [workloads.Well(kind=1, phase=2, p_bh=5500.0, cells=g.column(0, 0)),
                   workloads.Well(kind=0, phase=0, p_bh=4000.0, cells=g.column(nx - 1, ny - 1))]
        out.append((g, workloads.perturbed_state(g, rng)))
    return out


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEVICE)


def _states(s, phases):
    flags = (_dev(s.flag_new), _dev(s.flag_old)) if phases == 3 else (None, None)
    return _dev(s.u_new.ravel()), flags[0], _dev(s.u_old.ravel()), flags[1]


def _vector(case, seed, n):
    """The vector a product or a reverse step is applied to."""
    return np.random.default_rng([seed, 17]).normal(size=n)


def _controls(g, rates):
    """Every well on rate control at half of what it gives at its fixed
    pressure (producers their oil rate, the injector its gas rate)."""
    ctrl, limit = [], []
    for w, q in zip(g.wells, rates):
        ctrl.append((1, 1, 0.5 * -float(q[1])) if w.kind == 0 else (1, 2, 0.5 * float(q[2])))
        limit.append(1000.0 if w.kind == 0 else 8000.0)
    return ctrl, limit


# ---------------------------------------------------------------------- passes
def prepare(case, seed):
    op = case["op"]
    if op == "ensemble":
        models = _ensemble(case, seed)
        grids = [ocp.Grid(g) for g, _ in models]
        cells, blocks = sum(g.N for g in grids), sum(g.nnzb for g in grids)
        res, val = grids[0].empty(3 * cells), grids[0].empty(9 * blocks)
        ios, a, b = [], 0, 0
        for grid, (_, s) in zip(grids, models):
            un, fn, uo, fo = _states(s, 3)
            ios.append(dict(u_new=un, flag_new=fn, u_old=uo, flag_old=fo, residual=res[a:a + 3 * grid.N],
                            bsr_val=val[b:b + 9 * grid.nnzb]))
            a, b = a + 3 * grid.N, b + 9 * grid.nnzb
        batch = ocp.Batch(grids)
        batch.set_io(ios)
        return dict(op=op, grids=grids, batch=batch, res=res, val=val)
    g, s = _model(case, seed)
    grid = ocp.Grid(g)
    un, fn, uo, fo = _states(s, case["phases"])
    st = dict(op=op, grid=grid, un=un, fn=fn, uo=uo, fo=fo, dt=s.dt)
    nb, n = grid.nb, grid.N
    if op == "linearize":
        st.update(res=grid.empty(nb * n), val=grid.empty(grid.nnzb * nb * nb),
                  flux=grid.empty(3 * nb * n) if case["face_flux"] else None)
    elif op == "spmv":
        _, val, _ = grid.linearize(un, fn, uo, fo, s.dt)
        st.update(val=val, x=_dev(_vector(case, seed, nb * n)), y=grid.empty(nb * n), transpose=case["transpose"])
    elif op == "adjoint":
        _, val, flux = grid.linearize(un, fn, uo, fo, s.dt, want_face_flux=True)
        st.update(val=val, flux=flux, lam=_dev(_vector(case, seed, nb * n)),
                  out=dict(unew=grid.empty(nb * n), uold=grid.empty(nb * n), lnk=grid.empty(n), phi=grid.empty(n)))
    elif op in ("newton", "wells"):
        st.update(stepper=fim.Stepper(grid))
        if op == "wells":
            ctrl, limit = _controls(g, grid.well_rates(uo, fo).view(grid.nwell, nb).cpu().numpy())
            st.update(ctrl=ocp.well_controls(ctrl, limit, grid.device), p_bh=_dev(np.array([w.p_bh for w in g.wells])))
    elif op == "amounts":
        st.update(pn_new=grid.pn_from_natural(un, fn), pn_old=grid.pn_from_natural(uo, fo), out=None)
    elif op == "impec":
        st.update(pn=grid.pn_from_natural(uo, fo), work=grid.solver_work(), dt=0.1)
    return st


def run(st):
    op = st["op"]
    if op == "ensemble":
        st["batch"].linearize(1.0, graph=True)
        return st["res"], st["val"]
    grid = st["grid"]
    if op == "linearize":
        grid.linearize(st["un"], st["fn"], st["uo"], st["fo"], st["dt"], st["res"], st["val"], st["flux"])
        return st["res"], st["val"], st["flux"]
    if op == "spmv":
        return grid.spmv(st["val"], st["x"], y=st["y"], transpose=st["transpose"])
    if op == "adjoint":
        return grid.adjoint_vjp(st["un"], st["fn"], st["uo"], st["fo"], st["dt"], st["val"], st["flux"], st["lam"],
                                out=st["out"])
    if op == "newton":
        return st["stepper"].step(st["uo"], st["fo"], st["dt"])
    if op == "wells":
        u, flag, p_bh, _ = st["stepper"].step_wells(st["uo"], st["fo"], st["dt"], st["p_bh"], st["ctrl"])
        return u, flag, p_bh
    if op == "amounts":
        st["out"] = grid.linearize_pn(st["pn_new"], st["pn_old"], st["dt"], out=st["out"])
        return {k: st["out"][k] for k in ("residual", "bsr_val", "elim", "flag")}
    pn, dp, _ = fim.impec_step(grid, st["pn"], st["dt"], work=st["work"])
    return pn, dp


# ---------------------------------------------------------------------- work
def _cells(case):
    if case["op"] != "ensemble":
        n, shape = case["nx"] * case["ny"] * case["nz"], [(case["nx"], case["ny"], case["nz"])]
    else:
        sizes, shape = random.Random(case["sizes"]), []
        for _ in range(case["models"]):
            m = math.exp(sizes.uniform(math.log(case["smallest"]), math.log(case["largest"])))
            nx = max(2, int(round(math.sqrt(m / case["nz"]))))
            shape.append((nx, max(2, int(round(m / (case["nz"] * nx)))), case["nz"]))
        n = sum(a * b * c for a, b, c in shape)
    return n, sum(7 * a * b * c - 2 * (b * c + a * c + a * b) for a, b, c in shape)


def work(case):
    """Bytes: each input read once, each output written once (a whole step:
    at least one linearisation and one solve over its Jacobian).  Flops: the
    definitions' own count per cell and per block."""
    op, nb = case["op"], case.get("phases", 3)
    n, blocks = _cells(case)
    matrix, vector = 8 * nb * nb * blocks, 8 * nb * n
    states = 2 * vector + (2 * n if nb == 3 else 0)
    rock = 8 * 4 * n                         # three transmissibilities and a porosity per cell
    lin_flops = (500 if nb == 3 else 300) * n
    if op in ("linearize", "ensemble"):
        flux = 3 * vector if case.get("face_flux") else 0
        return dict(bytes=states + rock + vector + matrix + flux, flops=lin_flops)
    if op == "spmv":
        return dict(bytes=matrix + 2 * vector, flops=2 * nb * nb * blocks)
    if op == "adjoint":
        return dict(bytes=matrix + vector + 3 * vector + 48 * n + states + 8 * n + 2 * vector + 16 * n,
                    flops=2 * nb * nb * blocks + 150 * n)
    if op == "amounts":
        return dict(bytes=2 * 8 * (nb + 1) * n + rock + vector + matrix + 8 * (nb + 1) * n + n,
                    flops=lin_flops + 2 * 20 * blocks)
    if op == "impec":
        # two states, the pressure matrix once, ten iterations of two scalar products
        return dict(bytes=2 * 8 * (nb + 1) * n + rock + 8 * blocks, flops=400 * n + 10 * 4 * blocks)
    # newton, wells: a few linearisations, a few tens of products
    return dict(bytes=states + rock + vector + matrix, flops=4 * lin_flops + 100 * 2 * nb * nb * blocks)


# ---------------------------------------------------------------------- exact
class _Dual:
    """A value per cell or face and its derivatives by k seeds."""

    def __init__(self, v, g):
        self.v, self.g = v, g                 # g: [k, n]

    def __add__(self, o):
        return _Dual(self.v + o.v, self.g + o.g) if isinstance(o, _Dual) else _Dual(self.v + o, self.g)

    def __neg__(self):
        return _Dual(-self.v, -self.g)

    def __sub__(self, o):
        return self + (-o)

    def __mul__(self, o):
        if isinstance(o, _Dual):
            return _Dual(self.v * o.v, self.g * o.v + o.g * self.v)
        return _Dual(self.v * o, self.g * o)

    def __truediv__(self, o):
        if isinstance(o, _Dual):
            q = self.v / o.v
            return _Dual(q, (self.g - q * o.g) / o.v)
        return _Dual(self.v / o, self.g / o)

    __radd__, __rmul__ = __add__, __mul__

    def __rsub__(self, o):
        return -self + o

    def take(self, i, at=0, k=None):
        """The entries i, the seeds moved to the positions at.. of k."""
        g = self.g.new_zeros((k or len(self.g), len(i)))
        g[at:at + len(self.g)] = self.g[:, i]
        return _Dual(self.v[i], g)

    def constant(self):
        return _Dual(self.v, torch.zeros_like(self.g))


def _pick(c, a, b):
    return _Dual(torch.where(c, a.v, b.v), torch.where(c, a.g, b.g))


def _clamped(s):
    """s within [0, 1]; outside, the bound with no derivative."""
    out = _Dual(s.v.clamp(0.0, 1.0), s.g)
    return _Dual(out.v, torch.where((s.v < 0.0) | (s.v > 1.0), torch.zeros_like(s.g), s.g))


def _power(s, n):
    return s * s if n == 2.0 else _Dual(s.v ** n, s.g * (n * s.v ** (n - 1.0)))


class _Fluid:
    """The black-oil closure of one model (tables linear in 1/B, 1/mu, R_s)."""

    def __init__(self, g):
        self.g = g
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEVICE)
        self.p = t(g.tab_p)
        self.cols = dict(bo=1.0 / t(g.tab_Bo), imo=1.0 / t(g.tab_muo), bg=1.0 / t(g.tab_Bg), img=1.0 / t(g.tab_mug),
                         rs=t(g.tab_Rs))

    def piece(self, knots, v):
        return (torch.searchsorted(knots, v.contiguous(), right=True) - 1).clamp(0, len(knots) - 2)

    def column(self, name, p, k):
        y = self.cols[name]
        slope = (y[k + 1] - y[k]) / (self.p[k + 1] - self.p[k])
        return (p - self.p[k]) * slope + y[k]

    def volumes(self, p, x, flag):
        """b_w, b_o, b_g, R_s and the viscosities' reciprocals; x is R_s where flag is 1."""
        g = self.g
        k = self.piece(self.p, p.v)
        q = dict(bw=((p - g.p_ref) * g.cw + 1.0) * g.bw_ref, bo=self.column("bo", p, k), imo=self.column("imo", p, k))
        if g.nphase == 2:
            return q
        q.update(bg=self.column("bg", p, k), img=self.column("img", p, k), rs=self.column("rs", p, k))
        rs = self.cols["rs"]
        kr = self.piece(rs, x.v)
        pb = (x - rs[kr]) * ((self.p[kr + 1] - self.p[kr]) / (rs[kr + 1] - rs[kr])) + self.p[kr]
        under = flag == 1
        q["bo"] = _pick(under, self.column("bo", pb, kr) * ((p - pb) * g.co_under + 1.0), q["bo"])
        q["imo"] = _pick(under, self.column("imo", pb, kr) * ((p - pb) * -g.cmu_under + 1.0), q["imo"])
        q["rs"] = _pick(under, x, q["rs"])
        return q

    def amounts(self, p, sw, x, flag, phi):
        """phi S b of water, oil[, gas]."""
        g, q = self.g, self.volumes(p, x, flag)
        pore = ((p - g.p_ref) * g.cr + 1.0) * phi
        if g.nphase == 2:
            return [pore * sw * q["bw"], pore * (1.0 - sw) * q["bo"]]
        sg = _pick(flag == 1, x.constant() * 0.0, x)
        so = 1.0 - sw - sg
        return [pore * sw * q["bw"], pore * so * q["bo"], pore * (sg * q["bg"] + q["rs"] * so * q["bo"])]

    def cell(self, p, sw, x, flag):
        """Phase pressures, densities, mobilities, R_s and the injection terms."""
        g, q = self.g, self.volumes(p, x, flag)
        three = g.nphase == 3
        wspan = 1.0 - g.swc - g.sorw
        s_w, s_ow = _clamped((sw - g.swc) / wspan), _clamped((1.0 - sw - g.sorw) / wspan)
        krw, kro = _power(s_w, g.nw) * g.krw_max, _power(s_ow, g.now)
        c = dict(q, pw=p - (1.0 - s_w) * (1.0 - s_w) * g.pcow_max, po=p)
        if three:
            sg = _pick(flag == 1, x.constant() * 0.0, x)
            s_g = _clamped((sg - g.sgc) / (1.0 - g.swc - g.sgc - g.sorg))
            s_og = _clamped((1.0 - sg - g.swc - g.sorg) / (1.0 - g.swc - g.sorg))
            krg = _power(s_g, g.ng) * g.krg_max
            kro = (kro + krw) * (_power(s_og, g.nog) + krg) - (krw + krg)
            kro = _pick(kro.v >= 0.0, kro, kro.constant() * 0.0)
            c["pg"] = p + s_g * s_g * g.pcgo_max
        kro = kro * g.kro_cw
        c["rw"], c["lw"] = q["bw"] * g.rho_wsc, krw * q["bw"] * (1.0 / g.muw)
        c["lo"] = kro * q["bo"] * q["imo"]
        c["mob"] = krw * (1.0 / g.muw) + kro * q["imo"]
        if three:
            gas = g.rho_gsc / RB_FT3
            c["ro"], c["rg"] = (q["rs"] * gas + g.rho_osc) * q["bo"], q["bg"] * gas
            c["lg"] = krg * q["bg"] * q["img"]
            c["mob"] = c["mob"] + krg * q["img"]
        else:
            c["ro"] = q["bo"] * g.rho_osc
        return c


class _Mesh:
    """Geometry of one model: faces, transmissibilities, the block pattern."""

    def __init__(self, g):
        self.g, self.n = g, g.N
        nx, ny, nz = g.nx, g.ny, g.nz
        idx = torch.arange(g.N, device=DEVICE)
        i, j, k = idx % nx, (idx // nx) % ny, idx // (nx * ny)
        self.has = torch.stack([k > 0, j > 0, i > 0, idx >= 0, i < nx - 1, j < ny - 1, k < nz - 1])
        self.off = [-nx * ny, -nx, -1, 0, 1, nx, nx * ny]
        count = self.has.sum(0)
        self.start = torch.cumsum(count, 0) - count
        self.slot = self.start + torch.cumsum(self.has.long(), 0) - self.has.long()
        self.blocks = int(count.sum())
        self.phi, kx = _dev(g.phi), torch.exp(_dev(g.lnk))
        self.kx = kx
        self.faces = []
        for d, (h, area, f) in enumerate(((g.dx, g.dy * g.dz, 1.0), (g.dy, g.dx * g.dz, 1.0),
                                          (g.dz, g.dx * g.dy, g.kz_over_kx))):
            a = torch.nonzero(self.has[4 + d]).ravel()
            b = a + self.off[4 + d]
            T = DARCY * area / (0.5 * h / (kx[a] * f) + 0.5 * h / (kx[b] * f))
            self.faces.append((a, b, T, -g.dz if d == 2 else 0.0))
        self.wells = []
        r_o = 0.14 * math.sqrt(g.dx ** 2 + g.dy ** 2)
        for w in g.wells:
            cells = _dev(np.asarray(w.cells, dtype=np.int64))
            geom = DARCY * 2.0 * math.pi * g.dz / (math.log(r_o / w.rw) + w.skin)
            self.wells.append((w, cells, kx[cells] * geom))

    def fluxes(self, cell, seeds):
        """(a, b, T, component fluxes a -> b by the 2 * seeds unknowns of both cells) per direction."""
        names = ["w", "o", "g"][:self.g.nphase]
        for a, b, T, dz in self.faces:
            F, up = [], {}
            for m in names:
                ends = [[cell[q + m].take(i, at, 2 * seeds) for q in "prl"] for i, at in ((a, 0), (b, seeds))]
                dphi = ends[0][0] - ends[1][0] - (ends[0][1] + ends[1][1]) * (0.5 * GRAVITY * dz)
                up[m] = dphi.v >= 0.0
                F.append(_pick(up[m], ends[0][2], ends[1][2]) * dphi * T)
            if self.g.nphase == 3:
                rs = _pick(up["o"], cell["rs"].take(a, 0, 2 * seeds), cell["rs"].take(b, seeds, 2 * seeds))
                F[2] = F[2] + rs * F[1]
            yield a, b, T, F

    def sources(self, cell, p_bh=None):
        """(well, cells, WI, sources into the cells) per well; p_bh: a dual per well in place of its own pressure."""
        nb = self.g.nphase
        for iw, (w, cells, wi) in enumerate(self.wells):
            if p_bh is None:
                drive = w.p_bh - cell["po"].take(cells)
            else:
                drive = p_bh[iw].take(torch.zeros_like(cells)) - cell["po"].take(cells)
            if w.kind == 0:
                on = (drive.v < 0.0).double() * wi
                q = [cell["l" + m].take(cells) * drive * on for m in ["w", "o", "g"][:nb]]
                if nb == 3:
                    q[2] = q[2] + cell["rs"].take(cells) * q[1]
            else:
                on = (drive.v > 0.0).double() * wi
                put = cell["mob"].take(cells) * cell["bw" if w.phase == 0 else "bg"].take(cells) * drive * on
                q = [drive * 0.0 for _ in range(nb)]
                q[0 if w.phase == 0 else 2] = put
            yield w, cells, wi, q


def _unknowns(u, nb, seeds=None, at=0):
    u = u.view(nb, -1)
    out = []
    for v in range(nb):
        g = torch.zeros((seeds or nb, u.shape[1]), dtype=torch.float64, device=u.device)
        g[at + v] = 1.0
        out.append(_Dual(u[v], g))
    return out if nb > 2 else out + [out[0] * 0.0]


def _assemble(mesh, rows, flows, sources, seeds):
    """Residual [N, e] and block values [blocks, e, seeds] from the cells' own
    terms (duals by their own unknowns), the face fluxes and the sources."""
    n, ne = mesh.n, len(rows)
    res = torch.stack([r.v for r in rows], 1)
    val = torch.zeros((mesh.blocks, ne, seeds), dtype=torch.float64, device=res.device)
    diag = torch.stack([r.g.t() for r in rows], 1).clone()          # [N, e, seeds]
    fluxes = torch.zeros((3, ne, n), dtype=torch.float64, device=res.device)
    for d, (a, b, _, F) in enumerate(flows):
        f = torch.stack([q.v for q in F], 1)
        ga = torch.stack([q.g[:seeds].t() for q in F], 1)
        gb = torch.stack([q.g[seeds:].t() for q in F], 1)
        e = len(F)
        res[a, :e] += f
        res[b, :e] -= f
        diag[a, :e] += ga
        diag[b, :e] -= gb
        val[mesh.slot[4 + d][a], :e] = gb
        val[mesh.slot[2 - d][b], :e] = -ga
        fluxes[d][:e, a] = f.t()
    for _, cells, _, q in sources:
        for e, x in enumerate(q):
            res[cells, e] -= x.v
            diag[cells, e] -= x.g[:seeds].t()
    val[mesh.slot[3]] = diag
    return res, val, fluxes


def _linearized(g, u_new, f_new, u_old, f_old, dt, p_bh=None):
    """Residual, Jacobian, fluxes, mesh and sources of the natural-variable equations."""
    nb, mesh, fluid = g.nphase, _Mesh(g), _Fluid(g)
    scale = g.dx * g.dy * g.dz / RB_FT3 / dt
    seeds = nb
    new, old = _unknowns(u_new, nb), _unknowns(u_old, nb)
    cell = fluid.cell(*new, f_new)
    m_new, m_old = fluid.amounts(*new, f_new, mesh.phi), fluid.amounts(*old, f_old, mesh.phi)
    rows = [(a - b.v) * scale for a, b in zip(m_new, m_old)]
    res, val, fluxes = _assemble(mesh, rows, mesh.fluxes(cell, seeds), mesh.sources(cell), seeds)
    return dict(res=res, val=val, fluxes=fluxes, mesh=mesh, cell=cell, m_new=m_new, m_old=m_old, scale=scale)


def _product(mesh, val, x, transpose=False):
    """A x (A^T x) of the block matrix."""
    n, nb = mesh.n, val.shape[1]
    x = x.view(n, nb)
    y = torch.zeros_like(x)
    for t in range(7):
        rows = torch.nonzero(mesh.has[t]).ravel()
        if not len(rows):
            continue
        blk, cols = val[mesh.slot[t][rows]], rows + mesh.off[t]
        if transpose:
            y.index_add_(0, cols, (blk * x[rows][:, :, None]).sum(1))
        else:
            y.index_add_(0, rows, (blk * x[cols][:, None, :]).sum(2))
    return y


def _solved(apply, precondition, b, rounds=6):
    """x with A x = b to the last bits: preconditioned BiCGSTAB, refined."""
    x = torch.zeros_like(b)
    dot = lambda a, c: (a * c).sum()
    best = None
    for _ in range(rounds):
        r = precondition(b - apply(x))
        size = float(r.norm())
        if best is not None and size > 0.1 * best:
            break
        best = size
        if size == 0.0:
            break
        dx, r0, p, v = torch.zeros_like(b), r.clone(), torch.zeros_like(b), torch.zeros_like(b)
        rho = alpha = omega = torch.ones((), dtype=torch.float64, device=b.device)
        for it in range(3000):
            rho1 = dot(r0, r)
            p = r + (rho1 / rho) * (alpha / omega) * (p - omega * v)
            rho = rho1
            v = precondition(apply(p))
            alpha = rho / dot(r0, v)
            s = r - alpha * v
            t = precondition(apply(s))
            omega = dot(t, s) / dot(t, t)
            dx = dx + alpha * p + omega * s
            r = s - omega * t
            if it % 8 == 7 and not float(r.norm()) > 1e-9 * size:
                break
        x = x + dx
    return x


def _padded(mesh, val):
    """The blocks by neighbour type, [7, N, e, v], zero where there is none: fast products."""
    out = val.new_zeros((7, mesh.n) + val.shape[1:])
    nbr = torch.zeros((7, mesh.n), dtype=torch.long, device=val.device)
    for t in range(7):
        rows = torch.nonzero(mesh.has[t]).ravel()
        out[t, rows] = val[mesh.slot[t][rows]]
        nbr[t] = torch.arange(mesh.n, device=val.device)
        nbr[t, rows] += mesh.off[t]
    return out, nbr


def _solve_blocks(mesh, val, b):
    blk, nbr = _padded(mesh, val)
    inverse = torch.linalg.inv(blk[3])
    apply = lambda x: (blk * x[nbr][:, :, None, :]).sum((0, 3))
    return _solved(apply, lambda z: (inverse * z[:, None, :]).sum(2), b)


def _saturated_rs(fluid, p):
    k = fluid.piece(fluid.p, p)
    return fluid.column("rs", _Dual(p, p.new_zeros((1, len(p)))), k).v


def _updated(fluid, u, flag, du):
    """The Newton update: saturations chopped to 0.2, then the phase switch."""
    n = u.shape[1]
    big = du[:, 1].abs()
    big = torch.where(flag == 0, torch.maximum(big, du[:, 2].abs()), big)
    cut = torch.where(big > 0.2, 0.2 / big, torch.ones_like(big))
    p = u[0] - du[:, 0]
    sw = u[1] - du[:, 1] * cut
    x = u[2] - du[:, 2] * torch.where(flag == 0, cut, torch.ones_like(cut))
    rs = _saturated_rs(fluid, p)
    gone, came = (flag == 0) & (x < 0.0), (flag == 1) & (x > rs)
    x = torch.where(gone, rs, torch.where(came, torch.zeros_like(x), x))
    flag = torch.where(gone, torch.ones_like(flag), torch.where(came, torch.zeros_like(flag), flag))
    return torch.stack([p, sw, x]), flag, bool(gone.any() or came.any())


def _stepped(g, u_old, f_old, dt, controls=None, p_bh=None):
    """One implicit step by Newton to the last bits; with controls, the wells'
    pressures are unknowns under surface-rate control."""
    nb, fluid = 3, _Fluid(g)
    u, flag = u_old.view(nb, -1).clone(), f_old.clone()
    last = math.inf
    for _ in range(40):
        if controls is None:
            lin = _linearized(g, u.reshape(-1), flag, u_old, f_old, dt)
            du = _solve_blocks(lin["mesh"], lin["val"], lin["res"])
            moved = du
        else:
            du, dp = _well_correction(g, fluid, u, flag, u_old, f_old, dt, controls, p_bh)
            p_bh = p_bh - dp
            moved = torch.cat([du.reshape(-1), dp])
        u, flag, switched = _updated(fluid, u, flag, du)
        size = float((moved.abs()).max())
        if not switched and (size < 1e-10 or (size < 1e-6 and size > 0.3 * last)):
            break
        last = size
    return u.reshape(-1), flag, p_bh


def _well_correction(g, fluid, u, flag, u_old, f_old, dt, controls, p_bh):
    """The Newton correction of the cells and of the bottom-hole pressures."""
    nb, mesh = 3, _Mesh(g)
    scale = g.dx * g.dy * g.dz / RB_FT3 / dt
    new, old = _unknowns(u.reshape(-1), nb), _unknowns(u_old, nb)
    cell = fluid.cell(*new, flag)
    rows = [(a - b.v) * scale for a, b in
            zip(fluid.amounts(*new, flag, mesh.phi), fluid.amounts(*old, f_old, mesh.phi))]
    # a fourth seed: the well's own pressure
    wide = {k: _Dual(c.v, torch.cat([c.g, torch.zeros_like(c.g[:1])])) for k, c in cell.items()}
    seed = torch.tensor([[0.0], [0.0], [0.0], [1.0]], dtype=torch.float64, device=u.device)
    sources = list(mesh.sources(wide, [_Dual(p_bh[i:i + 1], seed) for i in range(len(p_bh))]))
    res, val, _ = _assemble(mesh, rows, mesh.fluxes(cell, nb), sources, nb)
    B, C, D, R, where = [], [], [], [], []
    for (w, cells, _, q), (_, phase, target) in zip(sources, controls):
        sign = -1.0 if w.kind == 0 else 1.0
        B.append(torch.stack([-x.g[3] for x in q], 1))
        C.append(sign * q[phase].g[:3].t())
        D.append(sign * q[phase].g[3].sum())
        R.append(sign * q[phase].v.sum() - target)
        where.append(cells)
    blk, nbr = _padded(mesh, val)

    def apply(x):
        y = (blk * x[nbr][:, :, None, :]).sum((0, 3))
        for b, c, d, cells in zip(B, C, D, where):
            y[cells] -= b * ((c * x[cells]).sum() / d)
        return y

    own = blk[3].clone()
    for b, c, d, cells in zip(B, C, D, where):
        own[cells] -= b[:, :, None] * c[:, None, :] / d
    inverse = torch.linalg.inv(own)
    rhs = res.clone()
    for b, d, r, cells in zip(B, D, R, where):
        rhs[cells] -= b * (r / d)
    x = _solved(apply, lambda z: (inverse * z[:, None, :]).sum(2), rhs)
    return x, torch.stack([(r - (c * x[cells]).sum()) / d for c, d, r, cells in zip(C, D, R, where)])


def _split(fluid, pn, nb):
    """The phase split of (P, N): natural variables as duals, the flag and V_f."""
    p, nw, no = pn[0], pn[1], pn[2]
    zero = p * 0.0
    if nb == 2:
        q = fluid.volumes(p, zero, None)
        vw, vo = nw / q["bw"], no / q["bo"]
        vf = vw + vo
        return p, vw / vf, zero, None, vf
    ng = pn[3]
    sat = fluid.volumes(p, zero, torch.zeros(len(p.v), dtype=torch.int8, device=p.v.device))
    flag = ((no.v > 0.0) & (ng.v <= sat["rs"].v * no.v)).to(torch.int8)
    rs = ng / no
    q = fluid.volumes(p, _pick(flag == 1, rs, zero), flag)
    vw, vo = nw / q["bw"], no / q["bo"]
    vg = _pick(flag == 1, zero, (ng - q["rs"] * no) / q["bg"])
    vf = vw + vo + vg
    return p, vw / vf, _pick(flag == 1, rs, vg / vf), flag, vf


def _amounts_system(g, pn_new, pn_old, dt):
    """The (P, N) system with N_w eliminated by each cell's volume balance."""
    nb, mesh, fluid = g.nphase, _Mesh(g), _Fluid(g)
    scale = g.dx * g.dy * g.dz / RB_FT3 / dt
    L = nb + 1
    pn = _unknowns(pn_new, L)
    p, sw, x, flag, vf = _split(fluid, pn, nb)
    cell = fluid.cell(p, sw, x, flag)
    old = pn_old.view(L, -1)
    rows = [(pn[e + 1] - old[e + 1]) * scale for e in range(nb)]
    rows.append(((p - g.p_ref) * g.cr + 1.0) * mesh.phi - vf)
    res, val, _ = _assemble(mesh, rows, mesh.fluxes(cell, L), mesh.sources(cell), L)
    a = rows[nb].g                                          # volume row [L, N]
    keep = [0] + list(range(2, L))
    c = a[keep] / a[1]
    c_r = rows[nb].v / a[1]
    red = torch.zeros((mesh.blocks, nb, nb), dtype=torch.float64, device=res.device)
    out = res[:, :nb].clone()
    for t in range(7):
        r = torch.nonzero(mesh.has[t]).ravel()
        if not len(r):
            continue
        s, col = mesh.slot[t][r], r + mesh.off[t]
        full = val[s][:, :nb]
        red[s] = full[:, :, keep] - full[:, :, 1:2] * c[:, col].t()[:, None, :]
        out[r] -= full[:, :, 1] * c_r[col][:, None]
    if flag is None:
        flag = torch.zeros(mesh.n, dtype=torch.int8, device=res.device)
    return out, red, torch.cat([c, c_r[None]]), flag


def _natural_to_amounts(g, u, flag):
    nb, mesh = g.nphase, _Mesh(g)
    m = _Fluid(g).amounts(*_unknowns(u, nb), flag, mesh.phi)
    return torch.cat([u.view(nb, -1)[0]] + [x.v for x in m])


def _impec(g, pn_old, dt):
    """Pressure from the linearised volume balance with old-level coefficients,
    then the explicit update of the amounts."""
    nb, mesh, fluid = g.nphase, _Mesh(g), _Fluid(g)
    L, n = nb + 1, mesh.n
    scale = g.dx * g.dy * g.dz / RB_FT3 / dt
    pn = _unknowns(pn_old, L)
    p, sw, x, flag, vf = _split(fluid, pn, nb)
    cell = {k: c.v for k, c in fluid.cell(p, sw, x, flag).items()}
    pore = ((p - g.p_ref) * g.cr + 1.0) * mesh.phi
    w = vf.g[1:]                                             # dV_f / dN_i
    diag = scale * (pore.g[0] - vf.g[0])
    E0 = scale * (pore.v - vf.v)
    faces = []
    val = torch.zeros((mesh.blocks, 1, 1), dtype=torch.float64, device=E0.device)
    for d, (a, b, T, dz) in enumerate(mesh.faces):
        coef, flow = [], []
        for m in ["w", "o", "g"][:nb]:
            dphi = cell["p" + m][a] - cell["p" + m][b] - (cell["r" + m][a] + cell["r" + m][b]) * (0.5 * GRAVITY * dz)
            up = dphi >= 0.0
            coef.append(T * torch.where(up, cell["l" + m][a], cell["l" + m][b]))
            flow.append(coef[-1] * dphi)
            if m == "o" and nb == 3:
                rs = torch.where(up, cell["rs"][a], cell["rs"][b])
        if nb == 3:
            coef[2], flow[2] = coef[2] + rs * coef[1], flow[2] + rs * flow[1]
        C, K = torch.stack(coef), torch.stack(flow)
        faces.append((a, b, C, K))
        for row, sign, slot in ((a, 1.0, mesh.slot[4 + d][a]), (b, -1.0, mesh.slot[2 - d][b])):
            c = (w[:, row] * C).sum(0)
            E0[row] += sign * (w[:, row] * K).sum(0)
            diag[row] += c
            val[slot, 0, 0] = -c
    wells = []
    for iw, (well, cells, wi) in enumerate(mesh.wells):
        drive = well.p_bh - cell["po"][cells]
        if well.kind == 0:
            on = (drive < 0.0).double() * wi
            c = [on * cell["l" + m][cells] for m in ["w", "o", "g"][:nb]]
            if nb == 3:
                c[2] = c[2] + cell["rs"][cells] * c[1]
        else:
            on = (drive > 0.0).double() * wi
            c = [torch.zeros_like(on) for _ in range(nb)]
            c[0 if well.phase == 0 else 2] = on * cell["mob"][cells] * cell["bw" if well.phase == 0 else "bg"][cells]
        c = torch.stack(c)
        wells.append((cells, c, drive))
        E0[cells] -= (w[:, cells] * c * drive).sum(0)
        diag[cells] += (w[:, cells] * c).sum(0)
    val[mesh.slot[3], 0, 0] = diag
    dp = _solve_blocks(mesh, val, -E0[:, None])[:, 0]
    flow = torch.zeros((nb, n), dtype=torch.float64, device=E0.device)
    for a, b, C, K in faces:
        f = K + C * (dp[a] - dp[b])
        flow[:, a] += f
        flow[:, b] -= f
    for cells, c, drive in wells:
        flow[:, cells] -= c * (drive - dp[cells])
    old = pn_old.view(L, n)
    return torch.cat([old[0] + dp, (old[1:] - flow / scale).reshape(-1)]), dp


def _adjoint(g, s, lam):
    """lambda^T dR/d(u_new, u_old, ln k, phi)."""
    nb = g.nphase
    un, fn, uo, fo = _states(s, nb)
    lin = _linearized(g, un, fn, uo, fo, s.dt)
    mesh, lam = lin["mesh"], lam.view(-1, nb)
    unew = _product(mesh, lin["val"], lam, transpose=True).t().reshape(-1)
    uold = -lin["scale"] * sum(m.g[:nb] * lam[:, e] for e, m in enumerate(lin["m_old"])).reshape(-1)
    phi = lin["scale"] * sum(lam[:, e] * (a.v - b.v) for e, (a, b) in
                             enumerate(zip(lin["m_new"], lin["m_old"]))) / mesh.phi
    lnk = torch.zeros_like(phi)
    for d, (a, b, _, _) in enumerate(mesh.faces):
        t = ((lam[a] - lam[b]).t() * lin["fluxes"][d][:, a]).sum(0)
        ka, kb = mesh.kx[a], mesh.kx[b]
        lnk[a] += kb / (ka + kb) * t
        lnk[b] += ka / (ka + kb) * t
    for _, cells, _, q in mesh.sources(lin["cell"]):
        for e, x in enumerate(q):
            lnk[cells] -= lam[cells, e] * x.v
    return dict(unew=unew, uold=uold, lnk=lnk, phi=phi)


def exact(case, seed):
    op = case["op"]
    if op == "ensemble":
        res, val = [], []
        for g, s in _ensemble(case, seed):
            lin = _linearized(g, *_states(s, 3), s.dt)
            res.append(lin["res"].reshape(-1))
            val.append(lin["val"].reshape(-1))
        return torch.cat(res), torch.cat(val)
    g, s = _model(case, seed)
    nb = case["phases"]
    un, fn, uo, fo = _states(s, nb)
    if op == "linearize":
        lin = _linearized(g, un, fn, uo, fo, s.dt)
        return lin["res"].reshape(-1), lin["val"].reshape(-1), lin["fluxes"].reshape(-1) if case["face_flux"] else None
    if op == "spmv":
        lin = _linearized(g, un, fn, uo, fo, s.dt)
        return _product(lin["mesh"], lin["val"], _dev(_vector(case, seed, nb * g.N)), case["transpose"]).reshape(-1)
    if op == "adjoint":
        return _adjoint(g, s, _dev(_vector(case, seed, nb * g.N)))
    if op == "newton":
        return _stepped(g, uo, fo, s.dt)[:2]
    if op == "wells":
        mesh, cell = _Mesh(g), _Fluid(g).cell(*_unknowns(uo, nb), fo)
        rates = [[float(x.v.sum()) for x in q] for _, _, _, q in mesh.sources(cell)]
        ctrl, _ = _controls(g, rates)
        return _stepped(g, uo, fo, s.dt, ctrl, _dev(np.array([w.p_bh for w in g.wells])))
    if op == "amounts":
        r, v, e, flag = _amounts_system(g, _natural_to_amounts(g, un, fn), _natural_to_amounts(g, uo, fo), s.dt)
        return dict(residual=r.reshape(-1), bsr_val=v.reshape(-1), elim=e.reshape(-1), flag=flag)
    return _impec(g, _natural_to_amounts(g, uo, fo), 0.1)
