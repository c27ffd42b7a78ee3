"""Design iterations of the adjoint lattice Boltzmann solver, as its users run them.

A pass is one evaluation of a design: the design field goes in, the flow (and
temperature) lattice is marched for a fixed number of steps, then its adjoint,
and the objective, the fields and dJ/dgamma come out.  Real solves march the
same steps until a tolerance; a fixed count keeps a pass comparable.

`exact` restates the discrete scheme in 64-bit torch: index gathers for the
streaming, dense moment sums for the collisions, and the boundary rows of each
(node type, normal) group.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_2501_02161_gb300 import inputs as I
from paper_2501_02161_gb300.autograd import SolveOpts, design_to_gamma, lbm_objective
from paper_2501_02161_gb300.serve import Batch
from paper_2501_02161_gb300.solver import Solver

DEV = "cuda" if torch.cuda.is_available() else "cpu"

# the shapes the server mixes: (nx, ny, nz, thermal)
MIX = [(32, 32, 32, True), (64, 64, 64, False), (96, 48, 24, True), (128, 64, 32, False), (192, 96, 48, True)]


def _case(kind, nx, ny, nz, storage, steps, check, model="eq12", tau=0.0, name=None):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "storage": storage, "steps": steps, "check": check,
         "model": model, "tau": tau}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the 2D pipe bend of the level-set optimiser, in double precision
        _case("bend2d", 64, 64, 1, "fp64", 1000, 500, tau=0.6, name="bend2d_64x64_fp64"),
        # the smallest 3D lattice in use (first tries, regression runs): latency only
        _case("bend", 16, 16, 16, "fp32", 1000, 500, tau=0.55, name="bend_16_fp32"),
        # 64-bit reference solves that accuracy is judged by
        _case("bend", 32, 32, 32, "fp64", 300, 150, tau=0.55, name="bend_32_fp64"),
        # the headline workload: 64^3 pipe bend at Re 50
        _case("bend", 64, 64, 64, "fp32", 1000, 500, tau=0.548, name="bend_64_fp32"),
        # a lattice whose sizes divide by nothing, with the linear gamma model
        _case("bend", 97, 61, 43, "fp32", 600, 300, model="linear", tau=0.57, name="bend_97x61x43_fp32"),
        # one iteration of a gradient loop: filter, projection, J, backward to the design variables
        _case("autograd", 96, 48, 24, "fp32", 600, 300, tau=0.566, name="autograd_96x48x24_fp32"),
        # the microchannel heat sink with both lattices and both adjoints
        _case("sink", 128, 64, 32, "fp32", 600, 300, tau=0.59, name="sink_128x64x32_fp32"),
        # the paper's pressure-driven quarter heat sink: symmetry planes and heat generation
        _case("quarter", 192, 48, 24, "fp32", 1000, 500, tau=0.615, name="quarter_192x48x24_fp32"),
        # the largest served shape with 16-bit flow storage
        _case("sink", 192, 96, 48, "fp16", 200, 100, tau=0.638, name="sink_192x96x48_fp16"),
        # five served lattices resident together, advanced by the batch
        _case("batch", 0, 0, 0, "fp32", 400, 200, tau=0.6, name="batch_served_mix_fp32"),
        # a heat sink far beyond the caches
        _case("sink", 320, 160, 80, "fp32", 60, 60, tau=0.734, name="sink_320x160x80_fp32"),
        # a production-size pipe bend
        _case("bend", 256, 256, 256, "fp32", 50, 50, tau=0.692, name="bend_256_fp32"),
    ]


# node updates (all phases) that a drawn pass may cost, about half of the largest listed one
DRAW_UPDATES = 8e8


def draw(rng: random.Random):
    """A lattice of the same families: sizes spread over their logarithm, odd ones
    among them, the number of steps falling with the size."""
    kind = rng.choices(["bend2d", "bend", "sink", "quarter", "autograd"], [2, 5, 3, 3, 1])[0]
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    model = "linear" if rng.random() < 0.25 else "eq12"
    tau = round(rng.uniform(0.56, 0.8), 3)
    if kind == "bend2d":
        nx, ny, nz = log(32, 512), log(32, 512), 1
        storage = rng.choice(["fp64", "fp32"])
    else:
        n = math.exp(rng.uniform(math.log(16 ** 3), math.log(200 ** 3)))   # nodes wanted
        ar = {"bend": (1, 1), "sink": (2, 4), "quarter": (4, 8), "autograd": (2, 4)}[kind]
        if kind == "autograd":
            n = min(n, 3e5)
        sx = (n * ar[0] * ar[1]) ** (1 / 3)
        jig = lambda v: max(12, int(round(v * math.exp(rng.uniform(-0.25, 0.25)))))
        nx, ny, nz = jig(sx), jig(sx / ar[0]), jig(sx / ar[1])
        storage = rng.choices(["fp32", "fp16", "bf16", "fp64"], [5, 2, 2, 1])[0]
        if kind == "autograd":
            storage = "fp32"
        if storage == "fp64":
            nx, ny, nz = min(nx, 48), min(ny, 48), min(nz, 48)
    phases = 2 if kind in ("bend2d", "bend") else 4
    cost = 12 if storage == "fp64" else 1
    steps = int(max(30, min(1000, DRAW_UPDATES / (phases * cost * nx * ny * nz))))
    check = max(1, steps // rng.choice([1, 2, 3]))
    return _case(kind, nx, ny, nz, storage, steps, check, model, tau)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
UMAX, DP_U = 0.05, 0.05


@functools.lru_cache(maxsize=4)
def _geometry(kind, nx, ny, nz, model, tau):
    """The lattice with gamma 1 at every open node; tau is reached through Re
    where the problem is given by Re."""
    gm = I.GAMMA_LINEAR if model == "linear" else I.GAMMA_EQ12
    nu = (tau - 0.5) / 3.0
    if kind == "bend2d":
        return I.pipe_bend_2d(nx, ny, width=max(4, min(nx, ny) // 4), umax=UMAX, tau=tau, gamma_value=1.0,
                              gamma_model=gm)
    if kind == "bend":
        w = max(2, min(nx, ny, nz) // 4)
        return I.pipe_bend_3d(nx, width=w, umax=UMAX, re=UMAX * w / nu, gamma_uniform=1.0, ny=ny, nz=nz,
                              gamma_model=gm)
    if kind in ("sink", "autograd"):
        return I.heat_sink(nx, ny, nz, umax=UMAX, re=UMAX * min(ny - 2, nz - 2) / nu, gamma_uniform=1.0,
                           gamma_model=gm)
    if kind == "quarter":
        lat = I.heat_sink_quarter(nx, ny, nz, re=DP_U * 2 * min(ny - 1, nz - 1) / nu, u_scale=DP_U,
                                  gamma_uniform=1.0)
        lat.gamma_model = gm
        return lat
    raise ValueError(kind)


def _members(case):
    """(geometry key) of every lattice in the case."""
    if case["kind"] == "batch":
        return [("sink" if th else "bend", nx, ny, nz, case["model"], case["tau"]) for nx, ny, nz, th in MIX]
    return [(case["kind"], case["nx"], case["ny"], case["nz"], case["model"], case["tau"])]


def _design(lat, seed):
    """A near-binary random design (blobs of a few cells, three quarters fluid)
    on the fluid nodes, as an optimiser's iterate looks; float64, flat."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    x = torch.randn(1, 1, lat.nz, lat.ny, lat.nx, generator=g, device=DEV, dtype=torch.float32)
    k = (1 if lat.nz == 1 else 5, 5, 5)
    pad = tuple(v // 2 for v in k)
    for _ in range(2):
        x = F.avg_pool3d(x, k, 1, pad, count_include_pad=False)
    x = (x - x.mean()) / x.std()
    d = (0.5 * (1.0 + torch.tanh(3.0 * (x + 0.6745)))).reshape(-1).double()
    fluid = torch.as_tensor((lat.flags & 7) == I.FLUID, device=DEV)
    return torch.where(fluid, d, torch.as_tensor(lat.gamma, device=DEV))


def prepare(case, seed):
    lats = [_geometry(*k) for k in _members(case)]
    st = {"case": dict(case), "lats": lats, "solvers": [], "gamma": []}
    for j, lat in enumerate(lats):
        s = Solver.from_lattice(lat, storage=case["storage"])
        st["solvers"].append(s)
        st["gamma"].append(_design(lat, int(seed) * 16 + j).to(s.rdtype))
    if case["kind"] == "autograd":
        lat = lats[0]
        shape = (lat.nz, lat.ny, lat.nx)
        st["rho"] = st["gamma"][0].reshape(shape)
        st["fixed"] = torch.as_tensor(lat.gamma, dtype=torch.float32, device=DEV).reshape(shape)
        st["mask"] = torch.as_tensor((lat.flags & 7) == I.FLUID, device=DEV).reshape(shape)
    return st


def _outputs(s, J):
    """The objective (in the lattice's precision, as the autograd call gives it),
    the fields and dJ/dgamma."""
    rho, u, T = s.fields()
    out = {"J": torch.tensor(J, dtype=s.rdtype), "rho": rho, "u": u, "sens": s.sensitivity()}
    if T is not None:
        out["T"] = T
    return out


def run(st):
    c = st["case"]
    if c["kind"] == "autograd":
        x = st["rho"].detach().requires_grad_(True)
        gam = design_to_gamma(x, st["mask"], st["fixed"])
        J = lbm_objective(gam.reshape(-1), st["solvers"][0], SolveOpts(0.0, c["steps"], c["check"]))
        (grad,) = torch.autograd.grad(J, x)
        return {"J": J.detach(), "grad": grad}
    if c["kind"] == "batch":
        b = Batch(c["storage"], check_every=c["check"], max_slots=8)
        try:
            for s, g in zip(st["solvers"], st["gamma"]):
                s.set_gamma(g)
                b.admit(s, 0.0, c["steps"], True)
            while b.step():
                pass
            by = {ctx: rep for _, ctx, rep in b.poll()}
        finally:
            b.close()
        return [_outputs(s, by[s._ctx.value].J) for s in st["solvers"]]
    s = st["solvers"][0]
    s.set_gamma(st["gamma"][0])
    fw = s.forward(tol=0.0, max_steps=c["steps"], check_every=c["check"])
    s.adjoint(tol=0.0, max_steps=c["steps"], check_every=c["check"])
    return _outputs(s, fw.J)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# floating-point operations of one node update, from the scheme's formulas:
# moments, equilibrium and relaxation of Q populations and their transposes
FLOPS = {"flow2": 110, "adj2": 130, "flow": 250, "adj": 270, "T": 70, "Tadj": 60}


def work(case):
    """Inputs read once and outputs written once; between steps a lattice that fits
    on the chip need not move, a larger one has to move its populations in and
    out at least once for the whole pass."""
    nb = fl = 0.0
    real = 8 if case["storage"] == "fp64" else 4
    steps = case["steps"]
    for kind, nx, ny, nz, _, _ in _members(case):
        n = nx * ny * nz
        thermal = kind not in ("bend2d", "bend")
        # design, flags and boundary values in; rho, u (T) and dJ/dgamma out
        nb += n * (real + 1 + real * (1 + 3 + 1 + (1 if thermal else 0)))
        if kind == "bend2d":
            fl += n * steps * (FLOPS["flow2"] + FLOPS["adj2"])
        else:
            fl += n * steps * (FLOPS["flow"] + FLOPS["adj"])
            if thermal:
                fl += n * steps * (FLOPS["T"] + FLOPS["Tadj"])
    return {"bytes": nb, "flops": fl}


# ---------------------------------------------------------------------------
# the same passes in 64-bit torch
# ---------------------------------------------------------------------------
AXES = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]


def _dirs(name):
    if name == "D3Q7":
        return [(0, 0, 0)] + AXES, [0.25] + [0.125] * 6
    r = (-1, 0, 1)
    es, ws = [], []
    for x in r:
        for y in r:
            for z in r if name == "D3Q19" else (0,):
                k = abs(x) + abs(y) + abs(z)
                if name == "D3Q19" and k < 3:
                    es.append((x, y, z))
                    ws.append((1 / 3, 1 / 18, 1 / 36)[k])
                elif name == "D2Q9":
                    es.append((x, y, z))
                    ws.append((4 / 9, 1 / 9, 1 / 36)[k])
    return es, ws


class _Stream:
    """Directions of one lattice and the gather that streams them: value i at x
    comes from x + sign e_i, through the periodic seam or mirrored in a
    symmetry plane half a node beyond the face (component reversed)."""

    def __init__(self, name, lat):
        self.e, w = _dirs(name)
        self.Q = len(self.e)
        self.E = torch.tensor(self.e, dtype=torch.float64, device=DEV)          # Q x 3
        self.w = torch.tensor(w, dtype=torch.float64, device=DEV)[:, None]
        self.opp = torch.tensor([self.e.index(tuple(-v for v in e)) for e in self.e], device=DEV)
        self.dims, self.mirror = (lat.nx, lat.ny, lat.nz), lat.mirror
        self.idx = {}

    def source(self, sign):
        nx, ny, nz = self.dims
        n = nx * ny * nz
        ar = torch.arange(n, device=DEV)
        at = [ar % nx, (ar // nx) % ny, ar // (nx * ny)]
        rows = []
        for e in self.e:
            comp, pos = [], []
            for a in range(3):
                c = at[a] + sign * e[a]
                out = (c < 0) | (c >= self.dims[a])
                if self.mirror >> a & 1:
                    comp.append(torch.where(out, -e[a], e[a]))
                    c = torch.where(c < 0, -1 - c, torch.where(c >= self.dims[a], 2 * self.dims[a] - 1 - c, c))
                else:
                    comp.append(torch.full_like(c, e[a]))
                    c = c % self.dims[a]
                pos.append(c)
            table = torch.zeros(27, dtype=torch.int64, device=DEV)
            for j, d in enumerate(self.e):
                table[(d[0] + 1) * 9 + (d[1] + 1) * 3 + d[2] + 1] = j
            j = table[(comp[0] + 1) * 9 + (comp[1] + 1) * 3 + comp[2] + 1]
            rows.append(j * n + pos[0] + nx * (pos[1] + ny * pos[2]))
        return torch.stack(rows)

    def pull(self, f, sign):
        if sign not in self.idx:
            self.idx = {sign: self.source(sign)}     # one at a time: large lattices
        return f.reshape(-1)[self.idx[sign]]


class _Exact:
    def __init__(self, lat, gamma):
        self.lat = lat
        self.N = lat.n
        self.g = gamma.double()
        self.bc = torch.as_tensor(lat.bcval, dtype=torch.float64, device=DEV).reshape(-1, 4)
        fl = torch.as_tensor(lat.flags.astype(np.int64), device=DEV)
        kind, code, heat = fl & 7, fl >> 3 & 7, (fl >> 6 & 1) > 0
        self.wall = (kind == 1).nonzero()[:, 0]
        self.open = (kind != 1).to(torch.float64)
        self.inlet = (kind == 2).nonzero()[:, 0]
        self.groups = []                             # (type, normal, holds T, nodes)
        for k in (2, 3):
            for c in range(6):
                for h in (False, True):
                    nodes = ((kind == k) & (code == c) & (heat == h)).nonzero()[:, 0]
                    if len(nodes):
                        self.groups.append((k, c, k == 2 or h, nodes))
        self.heated = [(c, ((kind == 1) & heat & (code == c)).nonzero()[:, 0]) for c in range(6)]
        U = lat.u_ref if lat.u_ref > 0 else math.sqrt(max(lat.dp, 0.0) / lat.rho0)
        nu = U * lat.l_ref / lat.re if lat.re is not None else (lat.tau - 0.5) / 3.0
        self.om = 1.0 / (0.5 + 3.0 * nu)
        self.kappa = nu / lat.pr if lat.pr else lat.kappa_f
        self.S = _Stream("D2Q9" if lat.stencil == I.D2Q9 else "D3Q19", lat)
        self.n_in = len(self.inlet)
        self.src = lat.w_pin / (3.0 * self.n_in) if self.n_in else 0.0
        self.linear = lat.gamma_model == I.GAMMA_LINEAR
        self.J = 0.0

    def _normal(self, S, c):
        n = torch.tensor(AXES[c], dtype=torch.float64, device=DEV)
        return n, S.E @ n

    # ---- flow -----------------------------------------------------------------
    def flow(self, steps):
        S, r0 = self.S, self.lat.rho0
        fc = torch.zeros(S.Q, self.N, dtype=torch.float64, device=DEV)   # f - w rho0
        for t in range(steps):
            f = S.pull(fc, -1)
            f[:, self.wall] = f[:, self.wall][S.opp]
            for kind, c, _, nodes in self.groups:
                n, d = self._normal(S, c)
                F_ = f[:, nodes]
                tan = d == 0
                if kind == 2:
                    u = self.bc[nodes, :3].T
                else:
                    un = (self.bc[nodes, 0] - r0 - F_[tan].sum(0) - 2 * F_[d < 0].sum(0)) / r0
                    u = n[:, None] * un
                ut = u - n[:, None] * (n @ u)
                Nt = 0.5 * (S.E[tan].T @ F_[tan]) - r0 / 3 * ut
                new = F_[S.opp] + 6 * S.w * r0 * (S.E @ u) - S.E @ Nt
                f[:, nodes] = torch.where((d > 0)[:, None], new, F_)
            drho = f.sum(0)
            u = S.E.T @ f / r0
            a, k = (u, r0 * self.g) if self.linear else (self.g * u, r0)
            ea = S.E @ a
            feq = S.w * (drho + k * (3 * ea + 4.5 * ea * ea - 1.5 * (a * a).sum(0)))
            fc = f + self.om * self.open * (feq - f)
        self.rho, self.u = r0 + drho, u
        if self.n_in:
            self.J += self.lat.w_pin * float(self.rho[self.inlet].sum()) / (3.0 * self.n_in)

    # ---- temperature ------------------------------------------------------------
    def _geq(self, T):
        return self.G.w * T * (1 + 4 * self.g * (self.G.E @ self.u))

    def _outflow(self, c, nodes):
        en = torch.tensor(AXES[c], dtype=torch.float64, device=DEV) @ self.u[:, nodes]
        return en, 0.125 * (1 + 4 * self.g[nodes] * en)

    def temperature(self, steps):
        lat = self.lat
        G = self.G = _Stream("D3Q7", lat)
        self.omT = 1 / (0.5 + 4 * self.kappa * (self.g + (1 - self.g) * lat.k_ratio))

        def collide(g):
            T = g.sum(0)
            Q = lat.beta_max * (1 - self.g) * (1 - T)
            return g + self.open * (self.omT * (self._geq(T) - g) + G.w * Q), T, Q

        gc, _, _ = collide(G.w * torch.full((1, self.N), lat.T0, dtype=torch.float64, device=DEV))
        for t in range(steps):
            g = G.pull(gc, -1)
            g[:, self.wall] = g[:, self.wall][G.opp]
            for c, nodes in self.heated:
                g[c + 1, nodes] += lat.q_flux
            for kind, c, hold, nodes in self.groups:
                K = g[:, nodes].sum(0) - g[c + 1, nodes]
                if hold:
                    g[c + 1, nodes] = self.bc[nodes, 3] - K
                else:
                    _, wa = self._outflow(c, nodes)
                    g[c + 1, nodes] = wa * K / (1 - wa)
            gc, T, Q = collide(g)
        self.gpost, self.gc, self.T = g, gc, T
        self.n_open = float(self.open.sum())
        self.J += lat.w_tmean * float((T * self.open).sum()) / self.n_open
        self.J -= lat.w_qgen * float((Q * self.open).sum())

    def temperature_adjoint(self, steps):
        lat, G = self.lat, self.G
        bg = lat.beta_max * (1 - self.g)
        src = lat.w_tmean / self.n_open + lat.w_qgen * bg
        wa_all = G.w * (1 + 4 * self.g * (G.E @ self.u))
        ga = torch.zeros(7, self.N, dtype=torch.float64, device=DEV)
        ckn = {}
        for t in range(steps):
            s = G.pull(ga, +1)
            new = (1 - self.omT) * s + self.omT * (wa_all * s).sum(0) - bg * (G.w * s).sum(0) - src
            for kind, c, hold, nodes in self.groups:
                cn = new[c + 1, nodes]
                if hold:
                    coef = -1.0
                else:
                    _, wa = self._outflow(c, nodes)
                    coef = wa / (1 - wa)
                    ckn[c] = cn
                new[:, nodes] += coef * cn
                new[c + 1, nodes] = 0.0
            new[:, self.wall] = s[:, self.wall][G.opp]
            ga = new
        # coupling to the flow adjoint and the temperature part of dJ/dgamma
        s = G.pull(ga, +1)
        T, gam = self.T, self.g
        eu = G.E @ self.u
        dom = -4 * self.kappa * (1 - lat.k_ratio) * self.omT ** 2
        self.v = 4 * gam * T * self.omT * (G.E.T @ (G.w * s))
        dgc = -(self.gpost - self._geq(T)) * dom + self.omT * G.w * T * 4 * eu
        self.sT = -(s * dgc).sum(0) + lat.beta_max * (1 - T) * ((G.w * s).sum(0) + lat.w_qgen)
        gs = G.pull(self.gc, -1)
        for kind, c, hold, nodes in self.groups:
            if hold:
                continue
            en, wa = self._outflow(c, nodes)
            K = gs[:, nodes].sum(0) - gs[c + 1, nodes]
            d = ckn[c] * 0.125 * K / (1 - wa) ** 2
            self.v[:, nodes] += 4 * gam[nodes] * d * torch.tensor(AXES[c], dtype=torch.float64, device=DEV)[:, None]
            self.sT[nodes] -= 4 * d * en
        self.v *= self.open / lat.rho0
        self.sT *= self.open
        G.idx = {}

    # ---- flow adjoint -----------------------------------------------------------
    def _adjoint_moments(self, s):
        S = self.S
        ws = S.w * s
        M = S.E.T @ ws
        eu = S.E @ self.u
        Qu = S.E.T @ (ws * eu)                        # sum_m w_m s_m e_m (e_m.u)
        return ws.sum(0), M, Qu

    def adjoint(self, steps):
        S, g, u = self.S, self.g, self.u
        v = getattr(self, "v", None)
        c2, c3 = (9 * g, 3 * g) if self.linear else (9 * g * g, 3 * g * g)
        src = torch.zeros(self.N, dtype=torch.float64, device=DEV)
        src[self.inlet] = self.src
        fa = torch.zeros(S.Q, self.N, dtype=torch.float64, device=DEV)
        for t in range(steps):
            s = S.pull(fa, +1)
            A, M, Qu = self._adjoint_moments(s)
            W = self.om * (3 * g * M + c2 * Qu - c3 * A * u)
            if v is not None:
                W = W + v
            new = (1 - self.om) * s + self.om * A - src + S.E @ W
            for kind, c, _, nodes in self.groups:
                n, d = self._normal(S, c)
                C = new[:, nodes]
                unk = (d > 0)[:, None]
                M_ = S.E.T @ torch.where(unk, C, 0.0)
                P = (6 * S.w * torch.where(unk, C, 0.0)).sum(0) if kind == 3 else 0.0
                down, tan = C + C[S.opp] - 2 * P, C - 0.5 * (S.E @ M_) - P
                new[:, nodes] = torch.where(unk, 0.0, torch.where((d < 0)[:, None], down, tan))
            new[:, self.wall] = s[:, self.wall][S.opp]
            fa = new
        A, M, Qu = self._adjoint_moments(S.pull(fa, +1))
        Mu, uQu, uu = (M * u).sum(0), (Qu * u).sum(0), (u * u).sum(0)
        br = 3 * Mu + 4.5 * uQu - 1.5 * uu * A if self.linear else 3 * Mu + 9 * g * uQu - 3 * g * uu * A
        self.sens = -self.lat.rho0 * self.om * br
        if v is not None:
            self.sens = self.sens + self.sT
        self.sens = self.sens * self.open


def _solve(lat, gamma, steps):
    x = _Exact(lat, gamma)
    x.flow(steps)
    if lat.thermal:
        x.S.idx = {}
        x.temperature(steps)
        x.temperature_adjoint(steps)
    x.adjoint(steps)
    u = x.u.clone()
    out = {"rho": x.rho, "u": u, "sens": x.sens, "J": x.J}
    if lat.thermal:
        out["T"] = x.T
    return out


def _gamma64(x, mask, fixed, radius=2.0, beta=8.0, eta=0.5):
    """Cone filter and smoothed Heaviside of the design variables."""
    r = int(math.floor(radius))
    ax = torch.arange(-r, r + 1, dtype=torch.float64, device=DEV)
    zz, yy, xx = torch.meshgrid(ax, ax, ax, indexing="ij")
    k = torch.clamp(radius - torch.sqrt(xx * xx + yy * yy + zz * zz), min=0.0)
    num, den = torch.zeros_like(x), torch.zeros_like(x)
    xp, one = F.pad(x, (r,) * 6), F.pad(torch.ones_like(x), (r,) * 6)
    nz, ny, nx = x.shape
    for dz in range(2 * r + 1):
        for dy in range(2 * r + 1):
            for dx in range(2 * r + 1):
                w = float(k[dz, dy, dx])
                if w:
                    sl = (slice(dz, dz + nz), slice(dy, dy + ny), slice(dx, dx + nx))
                    num, den = num + w * xp[sl], den + w * one[sl]
    a = math.tanh(beta * eta)
    p = (a + torch.tanh(beta * (num / den - eta))) / (a + math.tanh(beta * (1.0 - eta)))
    return torch.where(mask, p, fixed)


# node updates that exact() takes about 20 seconds for
EXACT_UPDATES = 2.5e9


def exact(case, seed):
    lats = [_geometry(*k) for k in _members(case)]
    phases = sum(lat.n * (4 if lat.thermal else 2) for lat in lats)
    if phases * case["steps"] > EXACT_UPDATES:
        return None
    real = torch.float64 if case["storage"] == "fp64" else torch.float32
    with torch.no_grad():
        outs = []
        for j, lat in enumerate(lats):
            gamma = _design(lat, int(seed) * 16 + j).to(real).double()
            if case["kind"] != "autograd":
                outs.append(_solve(lat, gamma, case["steps"]))
                continue
            shape = (lat.nz, lat.ny, lat.nx)
            mask = torch.as_tensor((lat.flags & 7) == I.FLUID, device=DEV).reshape(shape)
            fixed = torch.as_tensor(lat.gamma, device=DEV).reshape(shape)
            x = gamma.reshape(shape).requires_grad_(True)
            with torch.enable_grad():
                gam = _gamma64(x, mask, fixed)
            got = _solve(lat, gam.detach().reshape(-1), case["steps"])
            (grad,) = torch.autograd.grad(gam, x, got["sens"].reshape(shape))
            return {"J": got["J"], "grad": grad}
    return outs if case["kind"] == "batch" else outs[0]
