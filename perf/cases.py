"""The work that a user of this framework has it do, as measurable cases.

One pass of a case is one complete use of the public interface: the initial fields (or a saved
state) go in from host memory, the time steps run, and the result comes back to host memory.

The listed cases are the repository's own configurations at their own sizes (the Sod tube, the
Couette channel, the shock-interface, the 8192 x 8192 shear layer, a batch of uneven grids, a
stream of mixed requests), and beside them the sizes and options in between: odd and ragged grids,
each limiter, walls, dy != dx, both precisions, checkpoint and analysis output.

Results of the float32 mode are kept as float32, which is what the mode resolves; velocities come
as one array of both components (one of them is zero by symmetry in several flows).

`exact` advances the same inputs in float64 with dense transformation matrices and the limiter of
Sec. III in plain torch; it shares only the input recipes with the framework.
"""
import math

import numpy as np
import torch

from paper_1305_4736_gb300 import lbm, serving
from paper_1305_4736_gb300 import workloads as wl


def listed():
    return [
        # the smallest solves, where latency and launches count: the Sod tube at its stated length
        # in each precision, and the thermal Couette channel (walls, four columns wide)
        _solve("sod_f64", "riemann", 200, 4, 0, 2000),
        _solve("sod_f32", "riemann", 200, 4, 1, 2000),
        _solve("couette_f64", "couette", 4, 200, 0, 1000),
        # ordinary solves on odd sizes: a channel with the Lax-Wendroff scheme (a validation run
        # against the analytic profile), and a periodic shear layer with dy != dx
        _solve("channel_f64", "couette", 161, 97, 0, 500, limiter=1),
        _solve("shear_mid_f64", "shear", 1023, 517, 0, 100, dy=0.8),
        # the shock-interface at its full size; its non-equilibrium moments are read in float64
        _solve("shock_f64", "shock", 4096, 1024, 0, 20, delta=True, pinned=True),
        _solve("shock_f32", "shock", 4096, 1024, 1, 100, pinned=True),
        # the largest grid, in each precision, with its conserved totals
        _solve("shear_f64", "shear", 8192, 8192, 0, 10, totals=True, pinned=True),
        _solve("shear_f32", "shear", 8192, 8192, 1, 100, totals=True, pinned=True),
        # an ensemble of uneven grids stepped together
        {"name": "batch_f32", "kind": "batch", "count": 24, "nx_max": 2048, "ny_max": 1024, "precision": 1,
         "steps": 100, "sizes": 1305},
        # continuous batching of mixed requests (sizes, flows, precisions), all waiting at the start
        {"name": "serving_mixed", "kind": "serving", "count": 48, "nx_max": 2048, "ny_max": 512, "steps": 100,
         "sizes": 1305},
        # a run resumed from a checkpoint for some steps, analysed (Delta, Delta*, totals) and saved
        {"name": "resume_f64", "kind": "resume", "nx": 2048, "ny": 512, "precision": 0, "steps": 20},
    ]


def _solve(name, flow, nx, ny, precision, steps, limiter=0, dy=1.0, delta=False, totals=False, pinned=False):
    c = {"kind": "solve", "flow": flow, "nx": nx, "ny": ny, "precision": precision, "steps": steps,
         "limiter": limiter, "dy": dy, "delta": delta, "totals": totals, "pinned": pinned}
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 7 + ["batch", "serving", "resume"])
    precision = rng.randrange(2)
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 32), "nx_max": _log_int(rng, 256, 2048),
                "ny_max": _log_int(rng, 64, 1024), "precision": precision, "steps": rng.randint(10, 40),
                "sizes": rng.randrange(1 << 30)}
    if kind == "serving":
        return {"kind": "serving", "count": rng.randint(8, 40), "nx_max": _log_int(rng, 256, 2048),
                "ny_max": _log_int(rng, 32, 512), "steps": rng.randint(20, 100), "sizes": rng.randrange(1 << 30)}
    if kind == "resume":
        return {"kind": "resume", "nx": _log_int(rng, 64, 2048), "ny": _log_int(rng, 16, 1024),
                "precision": 0, "steps": rng.randint(1, 30)}
    flow = rng.choice(["riemann", "couette", "shock", "shear"])
    if flow == "riemann":
        nx, ny = _log_int(rng, 33, 4096), _log_int(rng, 1, 64)
    elif flow == "couette":
        nx, ny = _log_int(rng, 4, 1024), _log_int(rng, 16, 1024)
    else:
        nx, ny = _log_int(rng, 64, 4096), _log_int(rng, 16, 2048)
    cells = nx * ny
    steps = max(4, min(1000, int((1e9 if precision else 2e8) / cells)))
    limiter = rng.choice([0, 0, 0, 1, 2]) if flow in ("couette", "shear") else 0
    dy = rng.choice([1.0, 1.0, 0.8, 1.25]) if flow == "shear" else 1.0
    return _solve(None, flow, nx, ny, precision, steps, limiter, dy, delta=precision == 0 and rng.random() < 0.3,
                  totals=rng.random() < 0.3, pinned=cells >= 1 << 20)


# ------------------------------------------------------------------------------------ inputs
def _problem(c, seed):
    """The flow of a solve: grid, rates, boundaries and initial fields (input recipes only)."""
    rng = np.random.default_rng(seed)
    nx, ny, flow = c["nx"], c["ny"], c["flow"]
    if flow == "riemann":
        # the Sod states, varied by a few per cent from seed to seed
        v = rng.uniform(0.95, 1.05, 4)
        p = wl.riemann(nx, ny, (v[0], 0.0, 0.0, v[1]), (0.125 * v[2], 0.0, 0.0, 0.8 * v[3]), name="sod")
        p.s = wl.rates(min(5e3, 0.5 / p.dt))
    elif flow == "couette":
        p = wl.couette(float(rng.uniform(0.5, 2.0)), nx=nx, ny=ny, u0=float(rng.uniform(0.05, 0.3)))
        s5 = min(1e3, 0.5 / p.dt / max(1.0, p.Pr))          # every s dt <= 0.5 on coarse channels too
        p.s = wl.rates(s5, p.Pr * s5, s5)
        p.ux = p.ux + 1e-3 * np.sin(2 * math.pi * (np.arange(ny)[:, None] + 0.5) / ny + rng.uniform(0, 6))
    elif flow == "shock":
        p = wl.shock_interface(nx, ny, seed=int(seed))
        p.dt = min(p.dt, 0.3125 * p.dx / 6.0)               # the Courant number of the full size at most
        p.s = wl.rates(0.5 / p.dt)
    else:
        p = wl.shear_layer(nx, seed=int(seed), ny=ny)
        if c["dy"] != 1.0:
            p.dy = c["dy"] * p.dx
    p.limiter = c["limiter"]
    return p


def _batch_problems(c, seed):
    sizes = np.random.default_rng(c["sizes"])
    out = []
    for k in range(c["count"]):
        nx = int(round(math.exp(sizes.uniform(math.log(c["nx_max"] / 4), math.log(c["nx_max"])))))
        ny = int(round(math.exp(sizes.uniform(math.log(c["ny_max"] / 4), math.log(c["ny_max"])))))
        out.append(wl.shear_layer(nx, seed=int(seed) + k, ny=ny))
    return out


def _requests(c, seed):
    """Mixed requests: the sizes of the case, states and rates varied by the seed."""
    reqs = wl.serving_requests(c["count"], seed=c["sizes"], max_nx=c["nx_max"], max_ny=c["ny_max"], steps=c["steps"])
    rng = np.random.default_rng(seed)
    for r in reqs:
        r["problem"].rho = r["problem"].rho * rng.uniform(0.98, 1.02)
        r["problem"].T = r["problem"].T * rng.uniform(0.99, 1.01)
    return reqs


def _resume_problem(c, seed):
    return _problem({"flow": "shear", "nx": c["nx"], "ny": c["ny"], "limiter": 0, "dy": 1.0}, seed)


def _host(shape, pinned):
    return torch.empty(shape, dtype=torch.float64, pin_memory=pinned)


def _solver(p, precision):
    return lbm.Solver.from_problem(p, precision=precision)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        p = _problem(case, seed)
        shape = (p.ny, p.nx)
        fields = []
        for a in p.fields():
            t = _host(shape, case["pinned"])
            t.numpy()[...] = a
            fields.append(t.numpy())
        st = {"case": case, "solver": _solver(p, case["precision"]), "fields": fields,
              "out": _host((4,) + shape, case["pinned"])}
        if case["precision"]:
            st["out32"] = torch.empty((4,) + shape, dtype=torch.float32)
        if case["delta"]:
            st["delta"] = _host((16,) + shape, case["pinned"])
        return st
    if kind == "batch":
        probs = _batch_problems(case, seed)
        n = sum(p.cells for p in probs)
        out = _host((4, n), True)
        solvers, fields, views, at = [], [], [], 0
        for p in probs:
            solvers.append(_solver(p, case["precision"]))
            ts = [_host((p.ny, p.nx), True) for _ in range(4)]
            for t, a in zip(ts, p.fields()):
                t.numpy()[...] = a
            fields.append([t.numpy() for t in ts])
            views.append([out[k, at:at + p.cells].numpy().reshape(p.ny, p.nx) for k in range(4)])
            at += p.cells
        st = {"case": case, "solvers": solvers, "batch": _batch_of(solvers, fields), "fields": fields, "views": views,
              "out": out}
        if case["precision"]:
            st["out32"] = torch.empty((4, n), dtype=torch.float32)
        return st
    if kind == "serving":
        return {"case": case, "requests": _requests(case, seed),
                "engine": serving.Engine(serving.GpuBackend(), chunk=100, realtime=False)}
    p = _resume_problem(case, seed)
    shape = (p.ny, p.nx)
    f = _host((16,) + shape, True)
    f.copy_(_Flow(p).equilibrium_fields())
    return {"case": case, "solver": _solver(p, case["precision"]), "f": f.numpy(), "out": _host((4,) + shape, True),
            "delta": _host((16,) + shape, True), "dstar": _host((16,) + shape, True), "f_out": _host((16,) + shape, True)}


def _batch_of(solvers, fields):
    """A batch needs initialised members."""
    for s, f in zip(solvers, fields):
        s.init(*f)
    return lbm.Batch(solvers)


# -------------------------------------------------------------------------------------- a pass
def _moments(h, rho, u, v, T, delta=None):
    rc = lbm.lbm_moments(h, rho, u, v, T, delta)
    if rc != lbm.LBM_OK:
        raise lbm.LbmError(rc, "lbm_moments")


def _named(out):
    return {"rho": out[0], "velocity": out[1:3], "T": out[3]}


def _result(st):
    """rho, velocity, T of the pass: float64, or float32 in the float32 mode."""
    if "out32" in st:
        st["out32"].copy_(st["out"])
        return _named(st["out32"])
    return _named(st["out"])


def run(st):
    c = st["case"]
    if c["kind"] == "solve":
        s = st["solver"]
        s.init(*st["fields"])
        s.step(c["steps"])
        totals = s.totals() if c["totals"] else None
        o = st["out"].numpy()
        d = st.get("delta")
        _moments(s.h, o[0], o[1], o[2], o[3], d.numpy() if d is not None else None)
        r = _result(st)
        if totals is not None:
            r["totals"] = totals.astype(np.float32) if c["precision"] else totals
        if d is not None:
            r["delta"] = d
        return r
    if c["kind"] == "batch":
        for s, f in zip(st["solvers"], st["fields"]):
            s.init(*f)
        st["batch"].step(c["steps"])
        for s, v in zip(st["solvers"], st["views"]):
            _moments(s.h, *v)
        return _result(st)
    if c["kind"] == "serving":
        results, _ = st["engine"].run(st["requests"])
        r = {}
        for prec, name, dtype in ((0, "f64", torch.float64), (1, "f32", torch.float32)):
            m = [x.moments for x in results if x.precision == prec]
            if m:
                out = torch.cat([torch.stack([torch.from_numpy(a).reshape(-1) for a in x]) for x in m], dim=1)
                r[name] = _named(out.to(dtype))
        return r
    s = st["solver"]
    s_f, o = st["f_out"].numpy(), st["out"].numpy()
    lbm.lbm_set_state(s.h, st["f"])
    s.step(c["steps"])
    _moments(s.h, o[0], o[1], o[2], o[3], st["delta"].numpy())
    lbm.lbm_moments_central(s.h, st["dstar"].numpy())
    totals = s.totals()
    lbm.lbm_get_state(s.h, s_f)
    return dict(_named(st["out"]), delta=st["delta"], delta_star=st["dstar"], totals=totals, f=st["f_out"])


# ---------------------------------------------------------------------------------------- work
def _cost(cells, precision, steps, host_planes):
    """A step reads and writes 16 populations of a cell; its arithmetic is 335 operations, about 130
    of them multiply-adds.  Host planes (float64) cross once, and the state once more for each end."""
    state = 16 * (4 if precision else 8)
    return {"bytes": cells * (2.0 * state * steps + 2.0 * state + 16.0 * host_planes), "flops": cells * 465.0 * steps}


def work(case):
    kind = case["kind"]
    if kind == "solve":
        return _cost(case["nx"] * case["ny"], case["precision"], case["steps"], 8 + (16 if case["delta"] else 0))
    if kind == "resume":
        return _cost(case["nx"] * case["ny"], case["precision"], case["steps"], 16 + 4 + 32 + 16)
    if kind == "batch":
        parts = [(p.cells, case["precision"]) for p in _batch_problems(case, 0)]
    else:
        parts = [(r["problem"].cells, r["precision"]) for r in _requests(case, 0)]
    costs = [_cost(n, prec, case["steps"], 8) for n, prec in parts]
    return {k: sum(w[k] for w in costs) for k in ("bytes", "flops")}


# --------------------------------------------------------------------------------------- exact
class _Flow:
    """One flow in float64 with dense 16 x 16 transformations, in plain torch."""

    def __init__(self, p):
        self.p = p
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        r2 = math.sqrt(2.0)
        axis, diag = [(1, 0), (0, 1), (-1, 0), (0, -1)], [(1, 1), (-1, 1), (-1, -1), (1, -1)]
        v = np.array([(a * x, a * y) for a, d in ((1.0, axis), (6.0, axis), (r2, diag), (3.0 / r2, diag)) for x, y in d])
        self.vx, self.vy = v[:, 0], v[:, 1]
        self.M = self._rows(self.vx, self.vy)
        self.Mi = np.linalg.inv(self.M)
        self.b = 2.0 / (p.gamma - 1.0)

    @staticmethod
    def _rows(vx, vy):
        v2 = vx * vx + vy * vy
        eta2 = np.where(np.arange(16) < 4, 6.25, 0.0)
        w, d = v2 + eta2, vx * vx - vy * vy
        return np.array([vx ** 0, vx, vy, w, v2, d, vx * vy, vx * w, vy * w, vx * v2, vy * v2, vx * d, vy * d, v2 * w,
                         vx * vy * w, d * w])

    def t(self, a):
        return torch.as_tensor(a, dtype=torch.float64, device=self.dev)

    def mul(self, A, f):
        return (self.t(A) @ f.reshape(16, -1)).reshape(f.shape)

    def feq_hat(self, rho, ux, uy, T):
        b, P = self.b, rho * T
        jx, jy = rho * ux, rho * uy
        J2, d = jx * ux + jy * uy, jx * ux - jy * uy
        e, k = b * P + J2, (b + 4.0) * P + J2
        return torch.stack([rho, jx, jy, e, 2 * P + J2, d, jx * uy, (e + 2 * P) * ux, (e + 2 * P) * uy,
                            (4 * P + J2) * ux, (4 * P + J2) * uy, (2 * P + d) * ux, (d - 2 * P) * uy,
                            (2 * (b + 2) * P * P + (6 + b) * P * J2 + J2 * J2) / rho, k * ux * uy, k * d / rho])

    def macro(self, f):
        """rho, u, v, T of populations."""
        rho, jx, jy, e = (torch.einsum("q,qyx->yx", self.t(self.M[k]), f) for k in range(4))
        ux, uy = jx / rho, jy / rho
        return rho, ux, uy, (e - jx * ux - jy * uy) / (self.b * rho)

    def equilibrium_fields(self):
        return self.mul(self.Mi, self.feq_hat(*(self.t(a) for a in self.p.fields())))

    def ghosts(self, f):
        """f with two ghost layers along each edge (the corners hold ones: no stencil reads them)."""
        _, ny, nx = f.shape
        g = torch.ones((16, ny + 4, nx + 4), dtype=f.dtype, device=f.device)
        g[:, 2:-2, 2:-2] = f
        for edge, (kind, rho, u, v, T) in enumerate(self.p.bc):
            n, hi = (nx if edge < 2 else ny), edge % 2 == 1
            for layer in (1, 2):
                at = n + 1 + layer if hi else 2 - layer           # index of the ghost layer in g
                inner = f if edge < 2 else f.transpose(1, 2)
                if kind == wl.BC_PERIODIC:
                    col = inner[:, :, (n - 1 + layer if hi else -layer) % n]
                elif kind == wl.BC_ZERO_GRADIENT:
                    col = inner[:, :, n - 1 if hi else 0]
                elif kind == wl.BC_EQUILIBRIUM:
                    one = torch.ones_like(inner[0, :, :1])
                    col = self.mul(self.Mi, self.feq_hat(*(one * x for x in (rho, u, v, T))))[:, :, 0]
                else:
                    m = min(max(n - layer if hi else layer - 1, 0), n - 1)
                    fm = inner[:, :, m:m + 1]
                    rm, um, vm, Tm = self.macro(fm)
                    fg = fm + self.mul(self.Mi, self.feq_hat(rm, 2 * u - um, 2 * v - vm, 2 * T - Tm)
                                       - self.feq_hat(rm, um, vm, Tm))
                    col = fg[:, :, 0]
                if edge < 2:
                    g[:, 2:-2, at] = col
                else:
                    g[:, at, 2:-2] = col
        return g

    def slope(self, a, b):
        if self.p.limiter == wl.LIMITER_UPWIND:
            return torch.zeros_like(a)
        if self.p.limiter == wl.LIMITER_LW:
            return b
        m = torch.minimum(torch.minimum(2 * a.abs(), 2 * b.abs()), 0.5 * (a + b).abs())
        return torch.where(a * b > 0, m * torch.sign(a), torch.zeros_like(a))

    def step(self, f):
        p = self.p
        dx, dy = p.dx, (p.dx if p.dy is None else p.dy)
        _, ny, nx = f.shape
        g = self.ghosts(f)
        _, ux, uy, _ = self.macro(g[:, 1:-1, 1:-1])
        c = slice(1, -1)
        xx, xy = (ux[c, 2:] - ux[c, :-2]) / (2 * dx), (ux[2:, c] - ux[:-2, c]) / (2 * dy)
        yx, yy = (uy[c, 2:] - uy[c, :-2]) / (2 * dx), (uy[2:, c] - uy[:-2, c]) / (2 * dy)
        rho, u, v, T = self.macro(f)
        D = self.mul(self.M, f) - self.feq_hat(rho, u, v, T)
        s = np.array(p.s, dtype=np.float64)
        if s[7] != s[4]:
            k, P, div, shr = (s[7] / s[4] - 1.0) / s[7], rho * T, xx + yy, yx + xy
            D[7] += k * P * (u * (4 * xx - 4 / self.b * div) + 2 * v * shr)
            D[8] += k * P * (2 * u * shr + v * (4 * yy - 4 / self.b * div))
        D[:4] = 0.0
        out = f - self.mul(self.Mi * (p.dt * s)[None, :], D)
        del D
        for q in range(16):
            for vel, h, ax in ((self.vx[q], dx, 1), (self.vy[q], dy, 0)):
                if vel == 0.0:
                    continue
                sg, cr = (1 if vel > 0 else -1), abs(vel) * p.dt / h
                n = nx if ax else ny

                def at(k):
                    i = slice(2 + k * sg, 2 + k * sg + n)
                    return g[q, 2:-2, i] if ax else g[q, i, 2:-2]

                d0, d1, d2 = at(-1) - at(-2), at(0) - at(-1), at(1) - at(0)
                out[q] -= cr * (d1 + 0.5 * (1.0 - cr) * (self.slope(d1, d2) - self.slope(d0, d1)))
        return out

    def advance(self, f, n):
        for _ in range(n):
            f = self.step(f)
        return f

    def delta(self, f):
        return self.mul(self.M, f) - self.feq_hat(*self.macro(f))

    def delta_star(self, f):
        rho, u, v, T = self.macro(f)
        fn = self.mul(self.Mi, self.delta(f))
        out = torch.zeros_like(f)
        for q in range(16):
            wx, wy = self.vx[q] - u, self.vy[q] - v
            w2, d = wx * wx + wy * wy, wx * wx - wy * wy
            we = w2 + (6.25 if q < 4 else 0.0)
            rows = (torch.ones_like(wx), wx, wy, we, w2, d, wx * wy, wx * we, wy * we, wx * w2, wy * w2, wx * d, wy * d,
                    w2 * we, wx * wy * we, d * we)
            for k, r in enumerate(rows):
                out[k] += fn[q] * r
        return out

    def totals(self, f):
        dy = self.p.dx if self.p.dy is None else self.p.dy
        return (self.t(self.M[:4]) @ f.reshape(16, -1).sum(dim=1)) * (self.p.dx * dy)


def _exact_named(m):
    return {"rho": m[0].cpu(), "velocity": torch.stack(list(m[1:3])).cpu(), "T": m[3].cpu()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if case["nx"] * case["ny"] * case["steps"] > 2e9:
            return None                       # minutes of plain torch
        F = _Flow(_problem(case, seed))
        f = F.advance(F.equilibrium_fields(), case["steps"])
        r = _exact_named(F.macro(f))
        if case["totals"]:
            r["totals"] = F.totals(f).cpu()
        if case["delta"]:
            r["delta"] = F.delta(f).cpu()
        return r
    if kind == "resume":
        F = _Flow(_resume_problem(case, seed))
        f = F.advance(F.equilibrium_fields(), case["steps"])
        return dict(_exact_named(F.macro(f)), delta=F.delta(f).cpu(), delta_star=F.delta_star(f).cpu(),
                    totals=F.totals(f).cpu(), f=f.cpu())
    if kind == "batch":
        parts = [(case["precision"], p) for p in _batch_problems(case, seed)]
        if sum(p.cells for _, p in parts) * case["steps"] > 2e9:
            return None
    else:
        parts = [(r["precision"], r["problem"]) for r in sorted(_requests(case, seed), key=lambda r: r["id"])]
    out = {0: [], 1: []}
    for prec, p in parts:
        F = _Flow(p)
        m = F.macro(F.advance(F.equilibrium_fields(), case["steps"]))
        out[prec].append(torch.stack([a.reshape(-1) for a in m]).cpu())
    if kind == "batch":
        return _exact_named(torch.cat(out[case["precision"]], dim=1))
    return {name: _exact_named(torch.cat(out[k], dim=1)) for k, name in ((0, "f64"), (1, "f32")) if out[k]}
