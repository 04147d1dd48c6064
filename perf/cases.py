"""What a user of the library has it do, as a list of measurable cases.

Every case is one pass through the public binding (paper_1709_00803_gb300.igks), on the
repository's own synthetic meshes and flows at the sizes of its configurations:

- kind "solve": one steady solve kept on the GPU; a pass restarts it from a host state,
  advances it and reads the state back (a warm start, or one leg of a long run);
- kind "batch": many airfoils of different sizes in one context, the same pass for all;
- kind "serve": a stream of requests through the server until all have finished;
- kind "norms": the residual norms of device arrays without allocation.

exact() restates the method in plain numpy / torch at 64 bits: literal moments of the
Maxwellians, the sweeps level by level with differenced Euler fluxes.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from igks_inputs import fields as F
from igks_inputs import meshgen as G
from paper_1709_00803_gb300 import igks

FP64, FP32, DF64 = igks.PREC_FP64, igks.PREC_MIXED, igks.PREC_DF64


def listed():
    return [
        # the smallest call: norms of one solve's residual, on the caller's stream
        dict(name="norms", kind="norms", cells=60160),
        # the laminar plate, the smallest configuration: launches and latency count
        dict(name="laminar_plate_fp64", kind="solve", mesh="quads", nx=64, ny=32, precision=FP64, limiter=0,
             scheme=0, order=0, iters=20),
        # the turbulent plate in each sweep precision: 351 thin sweep levels
        dict(name="turbulent_plate_fp64", kind="solve", mesh="plate", cells=20480, precision=FP64, limiter=0,
             scheme=0, order=0, iters=10),
        dict(name="turbulent_plate_fp32", kind="solve", mesh="plate", cells=20480, precision=FP32, limiter=0,
             scheme=0, order=0, iters=20),
        dict(name="turbulent_plate_df64", kind="solve", mesh="plate", cells=20480, precision=DF64, limiter=0,
             scheme=0, order=0, iters=10),
        # an odd-sized hybrid plate with the smooth limiter
        dict(name="plate_venkat_fp32", kind="solve", mesh="plate", cells=5003, precision=FP32, limiter=2,
             scheme=0, order=0, iters=20),
        # the airfoil workload: SA, Barth-Jespersen limiter
        dict(name="naca0012_fp32", kind="solve", mesh="naca", cells=60160, precision=FP32, limiter=1,
             scheme=0, order=0, iters=10),
        # general polygons in a random numbering: stencils larger than a sweep record
        dict(name="polygons_df64", kind="solve", mesh="refined", n=24, precision=DF64, limiter=0, scheme=0,
             order=0, iters=20),
        # the cavity: explicit scheme, and the multicolour numbering's few wide levels
        dict(name="cavity_explicit", kind="solve", mesh="cavity", n=100, precision=FP64, limiter=0, scheme=1,
             order=0, iters=20),
        dict(name="cavity_multicolour_fp32", kind="solve", mesh="cavity", n=100, precision=FP32, limiter=0,
             scheme=0, order=1, iters=20),
        # the headline: a batch of seeded airfoils of 8k-80k cells, groups of solves on streams
        dict(name="airfoil_batch_fp32", kind="batch", solves=16, cells_lo=8000, cells_hi=80000, batch_seed=4,
             precision=FP32, groups=8, iters=10),
        # serving: plates and sections of 2k-12k cells, all submitted at once
        dict(name="serving", kind="serve", requests=8, cells_lo=2000, cells_hi=12000, stream_seed=5,
             precision=FP32, iters=200),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["norms", "quads", "plate", "plate", "naca", "naca", "refined", "cavity", "batch", "serve"])
    prec = rng.choice([FP64, FP32, FP32, DF64])
    if kind == "norms":
        return dict(kind="norms", cells=size(500, igks.NOALLOC_MAX_CELLS))
    if kind == "batch":
        return dict(kind="batch", solves=rng.randint(3, 10), cells_lo=size(2000, 8000), cells_hi=size(9000, 60000),
                    batch_seed=rng.randint(10, 10000), precision=prec, groups=rng.choice([1, 2, 4, 8]),
                    iters=rng.randint(4, 10))
    if kind == "serve":
        return dict(kind="serve", requests=rng.randint(2, 6), cells_lo=size(2000, 4000), cells_hi=size(5000, 12000),
                    stream_seed=rng.randint(10, 10000), precision=prec, iters=rng.randint(40, 120))
    c = dict(kind="solve", mesh=kind, precision=prec, limiter=0, scheme=0, order=0, iters=rng.randint(5, 20))
    if kind == "quads":
        return dict(c, nx=size(24, 160), ny=size(12, 90), limiter=rng.choice([0, 1, 2]))
    if kind == "plate":
        return dict(c, cells=size(1000, 60000), limiter=rng.choice([0, 0, 2]), scheme=rng.choice([0, 0, 0, 1]))
    if kind == "naca":
        return dict(c, cells=size(4000, 70000), limiter=rng.choice([1, 1, 2]))
    if kind == "refined":
        return dict(c, n=size(12, 60))
    return dict(c, n=size(20, 160), scheme=rng.choice([0, 1]), order=rng.choice([0, 1]))


# ---- meshes and flows ---------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _plate(cells):
    return G.turbulent_plate() if cells == 20480 else G.plate_scaled(cells, 1)


@functools.lru_cache(maxsize=64)
def _naca(m, p, t, cells, seed):
    return G.naca_scaled(m, p, t, cells, seed)


@functools.lru_cache(maxsize=64)
def _simple(mesh, a, b, order):
    if mesh == "quads":
        return G.flat_plate_quads(a, b, 1.1)
    if mesh == "refined":
        return G.refined_cavity(a, permute_seed=11)
    m = G.cavity(a)
    return m.renumbered(igks.order_cells(m, igks.ORDER_MULTICOLOR)[0]) if order else m


def _solve_of(case):
    """Mesh and flow of a "solve" case."""
    kind = case["mesh"]
    if kind == "plate":
        mesh, flow = _plate(case["cells"]), F.turbulent_plate_flow()
    elif kind == "naca":
        mesh, flow = _naca(0.0, 0.0, 0.12, case["cells"], 3), F.naca_flow()
    elif kind == "quads":
        mesh, flow = _simple(kind, case["nx"], case["ny"], 0), F.laminar_plate_flow()
    else:
        mesh, flow = _simple(kind, case["n"], 0, case["order"]), F.cavity_flow()
    flow.limiter, flow.scheme = case["limiter"], case["scheme"]
    return mesh, flow


def _solves_of(case):
    """Meshes and flows of every solve of a "batch" or "serve" case."""
    if case["kind"] == "batch":
        out = []
        for s in G.naca_batch_specs(case["solves"], case["batch_seed"], case["cells_lo"], case["cells_hi"]):
            out.append((_naca(s["m"], s["p"], s["t"], s["cells"], s["mesh_seed"]),
                        F.naca_flow(s["mach"], s["reynolds"], s["aoa"])))
        return out
    if case["kind"] == "serve":
        out = []
        for s in G.serving_specs(case["requests"], case["stream_seed"], case["cells_lo"], case["cells_hi"]):
            if s["kind"] == "plate":
                flow = F.turbulent_plate_flow()
                flow.mach, flow.reynolds = s["mach"], s["reynolds"]
                mesh = _plate(s["cells"])
            else:
                flow = F.naca_flow(s["mach"], s["reynolds"], s["aoa"])
                mesh = _naca(s["m"], s["p"], s["t"], s["cells"], s["mesh_seed"])
            flow.eq40_target = 3e-8
            out.append((mesh, flow))
        return out
    return [_solve_of(case)]


def _starts(case, solves, seed):
    """The starting states: a smooth seeded perturbation of each free stream."""
    return [F.perturbed_state(m, f, seed=1000 * seed + k, amp=0.02) for k, (m, f) in enumerate(solves)]


def _pinned(a):
    t = torch.empty(a.shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    t.numpy()[...] = a
    return t.numpy()


def _norm_arrays(case, seed):
    g = np.random.default_rng(seed)
    n = case["cells"]
    area = 10.0 ** g.uniform(-9.0, -2.0, n)
    return g.standard_normal(n) * area * 10.0 ** g.uniform(-4.0, 0.0, n), area


# ---- one pass -----------------------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "norms":
        m, a = _norm_arrays(case, seed)
        return dict(case=case, m=torch.from_numpy(m).cuda(), area=torch.from_numpy(a).cuda(),
                    out=torch.zeros(2, dtype=torch.float64, device="cuda"))
    solves = _solves_of(case)
    W0 = _starts(case, solves, seed)
    if case["kind"] == "serve":
        srv = igks.Server(precision=case["precision"], max_iters=case["iters"])
        return dict(case=case, server=srv, solves=solves, W0=W0)
    ctx = igks.Context(precision=case["precision"], groups=case.get("groups", 1))
    for m, f in solves:
        ctx.set_flow(ctx.mesh_upload(m), f)
    for k in range(len(solves)):
        ctx.init_freestream(k)
    W0 = _pinned(np.concatenate(W0, axis=1))
    return dict(case=case, ctx=ctx, solves=solves, W0=W0, W=_pinned(np.zeros_like(W0)))


NAMES = ("rho", "rho_u", "rho_v", "rho_e", "nu")


def run(state):
    case = state["case"]
    if case["kind"] == "norms":
        igks.residual_norms_noalloc(state["m"].data_ptr(), state["area"].data_ptr(), case["cells"],
                                    state["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return dict(norms=state["out"])
    if case["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(m, f, W0=W) for (m, f), W in zip(state["solves"], state["W0"])]
        done = {}
        while len(done) < len(ids):
            srv.step()
            for r in srv.poll():
                done[r["id"]] = r
        res = [done[i] for i in ids]
        return dict(W=[srv.take_fields(i) for i in ids], iters=[r["iters"] for r in res],
                    state=[r["state"] for r in res], forces=np.array([r["forces"] for r in res]))
    ctx, W = state["ctx"], state["W"]
    for k, (_, f) in enumerate(state["solves"]):
        ctx.set_scalars(k, dict(iter=0, cfl=f.cfl_init, res_inf_prev=0.0, res_l2_first=0.0, state=0))
    ctx.set_fields_all(state["W0"])
    _, st = ctx.iterate(case["iters"])
    ctx.get_fields_all(W)
    out = {n: W[k] for k, n in enumerate(NAMES)}
    for n in ("res_l2_rho", "res_inf", "eq40_ratio", "cfl", "dt"):
        out[n] = np.array([s[n] for s in st])
    out["iters"] = np.array([s["iters"] for s in st])
    out["state"] = np.array([s["state"] for s in st])
    return out


def work(case):
    """Per iteration: a cell's state in and out with its area, centre and wall distance, a
    face's length, normal, midpoint and two cells, the flux's 2000 flops a face and about
    400 flops a cell; once a pass: the states from and to the host."""
    if case["kind"] == "norms":
        return dict(bytes=16 * case["cells"] + 16, flops=4 * case["cells"])
    solves = _solves_of(case)
    nc, nf = sum(m.n_cells for m, _ in solves), sum(m.n_faces for m, _ in solves)
    return dict(bytes=case["iters"] * (112 * nc + 48 * nf) + 80 * nc, flops=case["iters"] * (400 * nc + 2000 * nf))


# ---- the method in plain numpy, 64 bits -----------------------------------------------------

K = 3
GAM = (K + 4.0) / (K + 2.0)
CB1, CB2, SIG, KAP = 0.1355, 0.622, 2.0 / 3.0, 0.41
CW1 = CB1 / KAP ** 2 + (1.0 + CB2) / SIG
CW2, CW3, CV1, CV2, CV3 = 0.3, 2.0, 7.1, 0.7, 0.9


def _pressure(W):
    return (GAM - 1.0) * (W[3] - 0.5 * (W[1] ** 2 + W[2] ** 2) / W[0])


def _sutherland(f, lam):
    tr = GAM * f.mach ** 2 / 2.0 / lam
    s = f.s_suth / f.t_ref
    return tr * np.sqrt(tr) * (1.0 + s) / (tr + s) / f.reynolds


def _mu(f, W):
    mu = _sutherland(f, W[0] / (2.0 * _pressure(W)))
    if not f.sa_on:
        return mu, np.zeros_like(mu)
    chi = np.maximum(W[4], 0.0) * W[0] / mu
    return mu, W[0] * np.maximum(W[4], 0.0) * chi ** 3 / (chi ** 3 + CV1 ** 3)


class _Max:
    """A Maxwellian in the face frame and its moments <u^i>, <u^i>_{u>=0}, <u^i>_{u<0}, <v^i>, <xi^2i>."""

    def __init__(self, W):
        self.r, self.U, self.V = W[0], W[1] / W[0], W[2] / W[0]
        self.h = 2.0 / (K + 2) * (W[3] / W[0] - 0.5 * (self.U ** 2 + self.V ** 2))
        self.lam = 0.5 / self.h
        one = np.ones_like(self.r)
        x = np.sqrt(self.lam) * self.U
        e = 0.5 * np.exp(-x * x) / np.sqrt(math.pi * self.lam)
        erfc = torch.special.erfc
        p0, n0 = (0.5 * erfc(torch.from_numpy(np.ascontiguousarray(s * x))).numpy() for s in (-1.0, 1.0))
        self.full = self._table(self.U, one, self.U)
        self.pos = self._table(self.U, p0, self.U * p0 + e)
        self.neg = self._table(self.U, n0, self.U * n0 - e)
        self.v = self._table(self.V, one, self.V)
        self.x = [one, K * self.h, K * (K + 2) * self.h ** 2]

    def _table(self, U, m0, m1):
        m = [m0, m1]
        for k in range(6):
            m.append(U * m[k + 1] + (k + 1) * self.h * m[k])
        return m

    def solve(self, b):
        """a with <a psi psi> = b"""
        E2 = self.U ** 2 + self.V ** 2 + (K + 2) * self.h
        R2, R3, R4 = b[1] - self.U * b[0], b[2] - self.V * b[0], 2.0 * b[3] - E2 * b[0]
        a3 = 4.0 * self.lam ** 2 / (K + 2) * (R4 - 2.0 * self.U * R2 - 2.0 * self.V * R3)
        a2, a1 = 2.0 * self.lam * R3 - self.V * a3, 2.0 * self.lam * R2 - self.U * a3
        return [b[0] - self.U * a1 - self.V * a2 - 0.5 * a3 * E2, a1, a2, a3]

    def mom(self, a, i, j, u):
        """<u^i v^j (a . psi) psi> with the u-table u; a = None: <u^i v^j psi>"""
        terms = [(1.0, 0, 0, 0)] if a is None else [
            (a[0], 0, 0, 0), (a[1], 1, 0, 0), (a[2], 0, 1, 0),
            (0.5 * a[3], 2, 0, 0), (0.5 * a[3], 0, 2, 0), (0.5 * a[3], 0, 0, 1)]
        psi = [[(1.0, 0, 0, 0)], [(1.0, 1, 0, 0)], [(1.0, 0, 1, 0)],
               [(0.5, 2, 0, 0), (0.5, 0, 2, 0), (0.5, 0, 0, 1)]]
        return [sum(c * w * u[i + p + q] * self.v[j + r + s] * self.x[k + l]
                    for c, p, r, k in terms for w, q, s, l in ps) for ps in psi]


def _add(*vs):
    return [sum(x) for x in zip(*vs)]


def _face_flux(f, WL, WR, sLn, sLt, sRn, sRt, cL, cR, dL, dR, mut, dt):
    """Time-integrated flux of every face in its own frame (Eq. 4-14 with the Prandtl fix)."""
    sides = []
    for W, sn, st, pos in ((WL, sLn, sLt, True), (WR, sRn, sRt, False)):
        g = _Max(W)
        an, at = g.solve([s / g.r for s in sn]), g.solve([s / g.r for s in st])
        A = g.solve([-m for m in _add(g.mom(an, 1, 0, g.full), g.mom(at, 0, 1, g.full))])
        sides.append((g, an, at, A, g.pos if pos else g.neg))
    W0 = _add(*[[g.r * m for m in g.mom(None, 0, 0, u)] for g, _, _, _, u in sides])
    g0 = _Max(W0)
    bl = g0.solve([(W0[k] - cL[k]) / dL / g0.r for k in range(4)])
    br = g0.solve([(cR[k] - W0[k]) / dR / g0.r for k in range(4)])
    bt = g0.solve([0.5 * (sLt[k] + sRt[k]) / g0.r for k in range(4)])
    eq = [_add(g0.mom(bl, i + 1, 0, g0.pos), g0.mom(br, i + 1, 0, g0.neg), g0.mom(bt, i, 1, g0.full)) for i in (0, 1)]
    B = g0.solve([-m for m in eq[0]])
    pL, pR = (s[0].r * s[0].h for s in sides)
    tau = (_sutherland(f, g0.lam) + mut) / (g0.r * g0.h) + f.c_num * np.abs(pL - pR) / (pL + pR) * dt
    ome = -np.expm1(-dt / tau)
    e = 1.0 - ome
    q = [dt - tau * ome, 2 * tau ** 2 * ome - tau * dt * (1 + e), 0.5 * dt ** 2 - tau * dt + tau ** 2 * ome,
         tau * ome, -2 * tau ** 2 * ome + tau * dt * e, -tau ** 2 * ome]

    def integral(i):   # int int u^i psi f over the time step
        t = [q[0] * g0.r * a + q[1] * g0.r * b + q[2] * g0.r * c for a, b, c in
             zip(g0.mom(None, i, 0, g0.full), eq[i], g0.mom(B, i, 0, g0.full))]
        for g, an, at, A, u in sides:
            n = _add(g.mom(an, i + 1, 0, u), g.mom(at, i, 1, u))
            t = [x + g.r * (q[3] * a + q[4] * b + q[5] * c)
                 for x, a, b, c in zip(t, g.mom(None, i, 0, u), n, g.mom(A, i, 0, u))]
        return t
    Ws, Fn = integral(0), integral(1)
    U, V, e0 = g0.U, g0.V, g0.U ** 2 + g0.V ** 2
    heat = (Fn[3] - U * Fn[1] - V * Fn[2] + 0.5 * e0 * Fn[0]      # int int (u - U) |c - (U, V)|^2 / 2 f;
            - U * (Ws[3] - U * Fn[0] - V * Ws[2] + 0.5 * e0 * Ws[0]))   # <u f> is the mass flux
    Fn[3] = Fn[3] + (1.0 / f.prandtl - 1.0) * heat
    return Fn


class _Numpy:
    """One steady solve, cell and face arrays as numpy vectors."""

    def __init__(self, m, flow, W):
        self.f, self.W, self.m = flow, W.copy(), m
        x, y, n = m.xy[:, 0], m.xy[:, 1], m.n_cells
        cp, cn = m.cell_ptr.astype(np.int64), m.cell_nodes
        own = np.repeat(np.arange(n), np.diff(cp))
        nxt = np.arange(cn.size) + 1
        nxt[cp[1:] - 1] = cp[:-1]
        cr = x[cn] * y[cn[nxt]] - x[cn[nxt]] * y[cn]
        s = lambda v: np.bincount(own, v, n)
        self.area = 0.5 * s(cr)
        self.cx = s((x[cn] + x[cn[nxt]]) * cr) / (6 * self.area)
        self.cy = s((y[cn] + y[cn[nxt]]) * cr) / (6 * self.area)
        self.own, self.vx, self.vy = own, x[cn] - self.cx[own], y[cn] - self.cy[own]
        a, b = m.face_nodes.T
        dx, dy = x[b] - x[a], y[b] - y[a]
        self.S = np.sqrt(dx * dx + dy * dy)
        self.nx, self.ny = dy / self.S, -dx / self.S
        self.mx, self.my = 0.5 * (x[a] + x[b]), 0.5 * (y[a] + y[b])
        self.L, self.R, self.bc = m.face_cells[:, 0], m.face_cells[:, 1], m.face_bc
        L, R, nx, ny = self.L, self.R, self.nx, self.ny
        self.dL = (self.mx - self.cx[L]) * nx + (self.my - self.cy[L]) * ny
        inn = R >= 0
        self.inn, self.ox = inn, np.where(inn, self.cx[R], self.cx[L] + 2 * self.dL * nx)
        self.oy = np.where(inn, self.cy[R], self.cy[L] + 2 * self.dL * ny)
        self.dR = (self.ox - self.mx) * nx + (self.oy - self.my) * ny
        self.dn = np.abs((self.ox - self.cx[L]) * nx + (self.oy - self.cy[L]) * ny)
        self.wall = np.full(n, 1e300)
        for f in np.nonzero((self.bc == 3) | (self.bc == 5))[0] if flow.sa_on else ():
            ex, ey = dx[f], dy[f]
            t = np.clip(((self.cx - x[a[f]]) * ex + (self.cy - y[a[f]]) * ey) / (ex * ex + ey * ey), 0.0, 1.0)
            self.wall = np.minimum(self.wall, np.hypot(x[a[f]] + t * ex - self.cx, y[a[f]] + t * ey - self.cy))
        p = 1.0 / (GAM * flow.mach ** 2)
        al = math.radians(flow.aoa_deg)
        self.inf = np.array([1.0, math.cos(al), math.sin(al), p / (GAM - 1) + 0.5,
                             flow.nut_ratio_inf / flow.reynolds if flow.sa_on else 0.0])
        self.levels = [self._levels(d) for d in (0, 1)] if flow.scheme == 0 else None
        self.it, self.cfl, self.prev, self.eq40, self.state = 0, flow.cfl_init, 0.0, 0.0, 0

    def _levels(self, back):
        """Sweep levels: (cells, entries' position in the level, neighbour, face, side)."""
        n, L, R = self.m.n_cells, self.L, self.R
        keep = self.inn | (back & np.isin(self.bc, (2, 3, 5)))
        f = np.nonzero(keep)[0]
        lo, hi = np.where(self.inn[f], np.minimum(L[f], R[f]), L[f]), np.where(self.inn[f], np.maximum(L[f], R[f]), -1)
        cell, nb = (np.where(hi >= 0, lo, L[f]), hi) if back else (hi, lo)
        by = np.argsort(cell, kind="stable")
        cell, nb, f = cell[by], nb[by], f[by]
        ptr = np.concatenate([[0], np.cumsum(np.bincount(cell, minlength=n))])
        lev, pl, nl = [0] * n, ptr.tolist(), nb.tolist()
        for i in range(n - 1, -1, -1) if back else range(n):
            lev[i] = max((lev[j] + 1 for j in nl[pl[i]:pl[i + 1]] if j >= 0), default=0)
        lev = np.array(lev)
        out = []
        order = np.argsort(lev, kind="stable")
        for c in np.split(order, np.cumsum(np.bincount(lev))[:-1]):
            cnt = ptr[c + 1] - ptr[c]
            pos = np.repeat(np.arange(c.size), cnt)
            e = np.repeat(ptr[c], cnt) + np.arange(cnt.sum()) - np.repeat(np.cumsum(cnt) - cnt, cnt)
            out.append((c, pos, nb[e], f[e], np.where(L[f[e]] == c[pos], 0, 1)))
        return out

    def _ghost(self):
        Wi, nx, ny = self.W[:, self.L], self.nx, self.ny
        g = np.repeat(self.inf[:, None], self.L.size, 1)
        b = self.bc == 3
        g[:, b] = Wi[:, b] * np.array([1.0, -1, -1, 1, -1])[:, None]
        b = self.bc == 2
        mn = Wi[1] * nx + Wi[2] * ny
        g[:, b] = np.stack([Wi[0], Wi[1] - 2 * mn * nx, Wi[2] - 2 * mn * ny, Wi[3], Wi[4]])[:, b]
        r, u, v = Wi[0], Wi[1] / Wi[0], Wi[2] / Wi[0]
        b = self.bc == 5
        uw = -self.inf[1] * ny + self.inf[2] * nx
        ug, vg = -2 * uw * ny - u, 2 * uw * nx - v
        g[:, b] = np.stack([r, r * ug, r * vg, Wi[3] + 0.5 * r * (ug ** 2 + vg ** 2 - u ** 2 - v ** 2), -Wi[4]])[:, b]
        b = self.bc == 4
        c, ei = np.sqrt(GAM * _pressure(Wi) / r), Wi[3] - 0.5 * r * (u ** 2 + v ** 2)
        un, uo = u * nx + v * ny, self.inf[1] * nx + self.inf[2] * ny
        ub = 0.5 * (un + uo) + (c - 1.0 / self.f.mach) / (GAM - 1)
        bx, by = u + (ub - un) * nx, v + (ub - un) * ny
        g[:, b] = np.stack([r, r * bx, r * by, ei + 0.5 * r * (bx ** 2 + by ** 2), Wi[4]])[:, b]
        return np.where(self.inn, self.W[:, self.R], g)

    def _gather(self, left, right):
        n = self.m.n_cells
        return np.bincount(self.L, left, n) + np.bincount(self.R[self.inn], right[self.inn], n)

    def _rot(self, g):
        return [g[0], g[1] * self.nx + g[2] * self.ny, -g[1] * self.ny + g[2] * self.nx, g[3]]

    def step(self):
        f, W, L, R, inn, nx, ny, S, n = (self.f, self.W, self.L, self.R, self.inn, self.nx, self.ny, self.S,
                                         self.m.n_cells)
        G_ = self._ghost()
        WLc = W[:, L]
        muL, mtL = _mu(f, WLc)
        muR, mtR = _mu(f, G_)
        # spectral radius and time steps
        u = [0.5 * (WLc[k] / WLc[0] + G_[k] / G_[0]) for k in (1, 2)]
        lam = np.abs(u[0] * nx + u[1] * ny) + 0.5 * sum(np.sqrt(GAM * _pressure(q) / q[0]) for q in (WLc, G_))
        if f.visc_sr:
            lam = lam + 2 * GAM * (muL + mtL + muR + mtR) / ((WLc[0] + G_[0]) * f.prandtl * self.dn)
        Lam = self._gather(0.5 * lam * S, 0.5 * lam * S)
        self.dt = dt = float(np.min(f.cfl_exp * self.area / Lam))
        # least-squares gradients over both cells of every face, limiter
        dx, dy = self.ox - self.cx[L], self.oy - self.cy[L]
        A = [self._gather(q, q) for q in (dx * dx, dx * dy, dy * dy)]
        det = A[0] * A[2] - A[1] ** 2
        gx, gy, phi = np.empty((4, n)), np.empty((4, n)), np.ones((4, n))
        for v in range(4):
            dw = G_[v] - WLc[v]
            r0, r1 = self._gather(dx * dw, dx * dw), self._gather(dy * dw, dy * dw)
            gx[v], gy[v] = (A[2] * r0 - A[1] * r1) / det, (A[0] * r1 - A[1] * r0) / det
            if f.limiter:
                hi, lo = W[v].copy(), W[v].copy()
                for op, z in ((np.maximum, hi), (np.minimum, lo)):
                    op.at(z, L, G_[v])
                    op.at(z, R[inn], WLc[v][inn])
                d = gx[v][self.own] * self.vx + gy[v][self.own] * self.vy
                ex = np.where(d > 0, hi[self.own], lo[self.own]) - W[v][self.own]
                with np.errstate(all="ignore"):
                    if f.limiter == 1:
                        r = np.where(d != 0, np.minimum(1.0, ex / d), 1.0)
                    else:
                        e2 = ((f.venkat_k * np.sqrt(self.area)) ** 3)[self.own]
                        r = np.where(d != 0, ((ex ** 2 + e2) * d + 2 * d * d * ex)
                                     / (d * (ex ** 2 + 2 * d * d + d * ex + e2)), 1.0)
                np.minimum.at(phi[v], self.own, r)
        om = np.abs((gx[2] - W[2] / W[0] * gx[0]) / W[0] - (gy[1] - W[1] / W[0] * gy[0]) / W[0])
        # face states and slopes
        px, py = phi * gx, phi * gy
        side = []
        for c, q in ((L, WLc), (np.where(inn, R, L), G_)):
            ox, oy = self.mx - self.cx[c], self.my - self.cy[c]
            fx, fy = px[:, c], py[:, c]
            side.append([self._rot(q[:4] + fx * ox + fy * oy), self._rot(fx * nx + fy * ny),
                         self._rot(fy * nx - fx * ny)])
        (wl, ln, lt), (wr, rn, rt) = side
        mir, st = np.isin(self.bc, (2, 3, 5)), np.where(self.bc == 2, 1.0, -1.0)
        ut = wl[2] / wl[0]
        utg = np.where(self.bc == 5, 2 * (self.inf[2] * nx - self.inf[1] * ny), 0.0) + st * ut
        ghost = [wl[0], -wl[1], wl[0] * utg, wl[3] + 0.5 * wl[0] * (utg ** 2 - ut ** 2)]
        gc = self._rot(G_)
        pick = lambda i, m_, o: np.where(inn, i, np.where(mir, m_, o))
        wr = [pick(a, b, c) for a, b, c in zip(wr, ghost, gc)]
        rn = [pick(a, b, 0.0) for a, b in zip(rn, (-ln[0], ln[1], -st * ln[2], -ln[3]))]
        rt = [pick(a, b, 0.0) for a, b in zip(rt, (lt[0], -lt[1], st * lt[2], lt[3]))]
        Fn = _face_flux(f, wl, wr, ln, lt, rn, rt, self._rot(WLc), gc, self.dL, self.dR, 0.5 * (mtL + mtR), dt)
        Fg = [Fn[0] * S, (Fn[1] * nx - Fn[2] * ny) * S, (Fn[1] * ny + Fn[2] * nx) * S, Fn[3] * S]
        M = np.zeros((5, n))
        for v in range(4):
            M[v] = -self._gather(Fg[v], -Fg[v]) / dt
        # Spalart-Allmaras
        sa, sad = None, None
        if f.sa_on:
            vi, vj = ((q[1] * nx + q[2] * ny) / q[0] for q in (WLc, G_))
            gn = (G_[4] - WLc[4]) / self.dn
            kap = ((muL / WLc[0] + muR / G_[0]) + (1 + CB2) * (WLc[4] + G_[4])) / (2 * SIG)
            inv = np.maximum(vi, 0) * WLc[4] + np.minimum(vj, 0) * G_[4]
            M[4] = self._gather((-inv + kap * gn - CB2 / SIG * WLc[4] * gn) * S,
                                (inv - kap * gn + CB2 / SIG * G_[4] * gn) * S)
            kd = kap / self.dn
            sa = (S * (np.minimum(vj, 0) - kd), S * (np.minimum(-vi, 0) - kd))
            mu, nut = _mu(f, W)[0], W[4]
            chi = nut * W[0] / mu
            fv1 = chi ** 3 / (chi ** 3 + CV1 ** 3)
            k2 = nut / (KAP * self.wall) ** 2
            sb = (1 - chi / (1 + chi * fv1)) * k2
            with np.errstate(all="ignore"):
                St = np.where(sb >= -CV2 * om, om + sb,
                              om + om * (CV2 ** 2 * om + CV3 * sb) / ((CV3 - 2 * CV2) * om - sb))
                r = np.where(k2 < 10 * St, k2 / St, 10.0)
            g = r + CW2 * (r ** 6 - r)
            fw = g * ((1 + CW3 ** 6) / (g ** 6 + CW3 ** 6)) ** (1.0 / 6.0)
            M[4] += self.area * (CB1 * St * nut - CW1 * fw * (nut / self.wall) ** 2)
            sad = self._gather(S * (np.maximum(vi, 0) + kd), S * (np.maximum(-vj, 0) + kd))
            sad = sad + 2 * self.area * CW1 * fw * nut / self.wall ** 2
        # norms and CFL (Eq. 25)
        self.l2, self.inf_norm = float(np.sqrt(np.mean((M[0] / self.area) ** 2))), float(np.max(np.abs(M[0])))
        self.cfl = f.cfl_init if self.it == 0 else min(max(self.cfl * self.prev / self.inf_norm, f.cfl_min), f.cfl_max)
        self.prev = self.inf_norm
        if f.scheme == 1:
            dW = dt * M / self.area
        else:
            dW = self._sweeps(M, lam, Lam, sa, sad, G_)
        self.eq40 = float(np.max(np.sqrt(np.sum(dW[:4] ** 2, 0)) / np.sqrt(np.sum(W[:4] ** 2, 0))))
        self.W = W + dW
        self.W[4] = np.maximum(self.W[4], 0.0)
        self.it += 1

    def _sweeps(self, M, lam, Lam, sa, sad, G_):
        W, n = self.W, self.m.n_cells
        D, Ds = Lam / self.cfl + Lam, (Lam / self.cfl + sad) if sa else None
        dW = [np.zeros((5, n)), np.zeros((5, n))]
        for back in (0, 1):
            for c, pos, j, f, side in self.levels[back]:
                nx, ny, h = self.nx[f], self.ny[f], 0.5 * self.S[f]
                Wj, dj = W[:, j], dW[back][:, j]
                if back and (j < 0).any():
                    gh = j < 0
                    own = dW[0][:, c[pos]]
                    mn = 2 * (own[1] * nx + own[2] * ny)
                    sym = np.stack([own[0], own[1] - mn * nx, own[2] - mn * ny, own[3], own[4]])
                    wal = own * np.array([1.0, -1, -1, 1, -1])[:, None]
                    Wj = np.where(gh, G_[:, f], Wj)
                    dj = np.where(gh, np.where(self.bc[f] == 2, sym, wal), dj)
                sg = np.where(side == 0, h, -h)
                q, p0 = Wj + dj, _pressure(Wj)
                p1 = _pressure(q)
                v0, v1 = (Wj[1] * nx + Wj[2] * ny) / Wj[0], (q[1] * nx + q[2] * ny) / q[0]
                dF = [dj[1] * nx + dj[2] * ny, q[1] * v1 - Wj[1] * v0 + (p1 - p0) * nx,
                      q[2] * v1 - Wj[2] * v0 + (p1 - p0) * ny, (q[3] + p1) * v1 - (Wj[3] + p0) * v0]
                base = M[:, c] if not back else np.zeros((5, c.size))
                for v in range(4):
                    s = np.bincount(pos, sg * dF[v] - h * lam[f] * dj[v], c.size)
                    dW[back][v, c] = (base[v] - s) / D[c] if not back else dW[0][v, c] - s / D[c]
                if sa:
                    s = np.bincount(pos, np.where(side == 0, sa[0][f], sa[1][f]) * dj[4], c.size)
                    dW[back][4, c] = (base[4] - s) / Ds[c] if not back else dW[0][4, c] - s / Ds[c]
        return dW[1]


def exact(case, seed):
    if case["kind"] == "norms":
        m, a = _norm_arrays(case, seed)
        return dict(norms=np.array([np.max(np.abs(m)), math.sqrt(math.fsum((m / a) ** 2) / m.size)]))
    if case["kind"] != "solve":
        return None
    mesh, flow = _solve_of(case)
    if case["iters"] * (mesh.n_cells + 12000) > 1.1e6:   # about 15 s
        return None
    s = _Numpy(mesh, flow, _starts(case, [(mesh, flow)], seed)[0])
    for _ in range(case["iters"]):
        s.step()
    out = {n: s.W[k] for k, n in enumerate(NAMES)}
    one = lambda v: np.array([v], dtype=np.float64)
    return dict(out, res_l2_rho=one(s.l2), res_inf=one(s.inf_norm), eq40_ratio=one(s.eq40), cfl=one(s.cfl),
                dt=one(s.dt), iters=None, state=None)
