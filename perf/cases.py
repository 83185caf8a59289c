"""Workloads by which this framework's speed and accuracy are followed.

A case is one pass of what a user's program does: advance one simulation, or
a batch of them, by some time steps through the public API and read the
results back to the host.  The cases span the range the framework is used
over: 80 x 40 to 4096 x 1024 lattices, FP64, FP32 and FP16 storage, one
instance and batches of 10 to 512, the three collision models, walls and
periodic boxes, lattices that are and are not whole numbers of tiles.

Results are returned in the precision the run computes in: float64 for FP64
runs; float32 for FP32 runs; for FP16 storage float32 positions and densities
(FP64 and near-unity quantities) and float16 velocities.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2212_14153_gb300 import fpd, tumbling
from paper_2212_14153_gb300 import workloads as wl

PRECISION = {"f64": wl.PRECISION_F64, "f32": wl.PRECISION_F32, "f16": wl.PRECISION_F16}
ELEM = {"f64": 8, "f32": 4, "f16": 2}
MAGIC, LL, BGK = 0, 1, 2
ENDLESS = 1 << 40  # steps requested of a batch instance that is advanced as long as the program runs


# ------------------------------------------------------------------- cases
def _one(name, nx, ny, precision, steps, n_beads=0, n_fibers=0, a=2.0, xi=1.0, re=5.0, K=0.33, nu=-1.0,
         collision=MAGIC, tuning="default", read="fields"):
    c = dict(kind="one", nx=nx, ny=ny, precision=precision, steps=steps, n_beads=n_beads, n_fibers=n_fibers,
             a=a, xi=xi, re=re, K=K, nu=nu, collision=collision, tuning=tuning, read=read)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a stiff 8-bead fiber on a small lattice in FP64: the reference-quality run
        # that reduced precisions are judged against, and the smoke test's lattice
        _one("small_f64", 80, 40, "f64", 128, 8, 1, a=2.0, re=1.0, K=3.3),
        # a program that looks at the fiber after every single step (steering,
        # plotting): the smallest call there is, one step and one bead read
        _one("follow_f32", 100, 200, "f32", 1, 10, 1, a=2.0, xi=0.5, re=1.0, K=3.3, read="beads"),
        # one flexible 20-bead fiber at Re = 10: a production run of one instance,
        # whose state fits in L2
        _one("medium_f32", 1024, 256, "f32", 512, 20, 1, a=4.0, re=10.0, K=3.3e-5, tuning="auto"),
        # three fibers on a lattice of no whole tiles, BGK collision
        _one("ragged_f32", 333, 171, "f32", 256, 9, 3, a=2.5, xi=0.625, re=4.0, K=0.05, collision=BGK),
        # the headline lattice, two 20-bead fibers, in each storage precision
        _one("large_f32", 4096, 1024, "f32", 256, 20, 2, a=4.0, tuning="auto"),
        _one("large_f16", 4096, 1024, "f16", 256, 20, 2, a=4.0, tuning="auto"),
        _one("large_f64", 4096, 1024, "f64", 24, 20, 2, a=4.0, tuning="auto"),
        # start-up Couette flow without fibers at constant Lallemand-Luo rates
        _one("couette_ll_f32", 1000, 500, "f32", 256, nu=0.1, collision=LL),
        # the driven-particle benchmark: one bead in a doubly periodic box
        dict(name="driven_f32", kind="driven", a=8.0, r_eta=100.0, r_xi=0.0625, Re_p=1.0, precision="f32", steps=256),
        # a tumbling-period sweep: ten instances, looked at every 200 steps
        dict(name="tumbling_f32", kind="batch", family="tumbling", n=10, layout=1, precision="f32", steps=200,
             read="beads"),
        # the paper's parameter sweep: many instances of uneven size at once
        dict(name="sweep512_f32", kind="batch", family="sweep", n=512, layout=4, precision="f32", steps=192,
             read="beads"),
        # a batch in FP16 storage whose flow fields are kept
        dict(name="sweep48_f16", kind="batch", family="sweep", n=48, layout=5, precision="f16", steps=128,
             read="fields"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choices(["fiber", "flow", "driven", "batch"], [5, 1, 1, 3])[0]
    precision = rng.choices(["f64", "f32", "f16"], [1, 3, 1])[0]
    # steps so that a pass makes about 100 million to a billion cell updates, FP64 fewer
    most = 1.0e8 if precision == "f64" else 1.0e9
    if kind in ("fiber", "flow"):
        ny = int(_log(rng, 32, 1024))
        nx = max(32, min(4096, int(ny * _log(rng, 1.0, 8.0))))
        steps = max(1, min(int(_log(rng, 1, 512)), int(most / (nx * ny))))
        tuning = rng.choice(["default", "auto"])
        read = rng.choice(["fields", "beads"])
        if kind == "flow":
            return _one(None, nx, ny, precision, steps, nu=_log(rng, 0.02, 0.3),
                        collision=rng.choice([MAGIC, LL, BGK]), tuning=tuning)
        a = rng.uniform(2.0, 4.0)
        n_fibers = rng.randint(1, 3)
        length = rng.uniform(0.2, 0.8) * min(ny, nx / n_fibers)
        n_beads = max(3, min(30, round(length / (2 * a))))
        return _one(None, nx, ny, precision, steps, n_beads, n_fibers, a=a, xi=a / 4.0, re=_log(rng, 1.0, 10.0),
                    K=_log(rng, 3.3e-3, 3.3), collision=rng.choice([MAGIC, MAGIC, BGK, LL]), tuning=tuning, read=read)
    if kind == "driven":
        return dict(kind="driven", a=rng.uniform(3.0, 12.0), r_eta=_log(rng, 1.0, 200.0),
                    r_xi=rng.choice([0.03, 0.0625, 0.125]), Re_p=_log(rng, 0.1, 3.0), precision=precision,
                    steps=int(_log(rng, 16, 512)))
    n = int(_log(rng, 4, 256))
    return dict(kind="batch", family=rng.choice(["tumbling", "sweep"]), n=n, layout=rng.randint(10, 1 << 20),
                precision=precision, steps=max(1, min(int(_log(rng, 16, 256)), int(most / (5e4 * n)))),
                read="fields" if n <= 60 and rng.random() < 0.5 else "beads")


# ------------------------------------------------------------------ inputs
def _fiber_config(case, seed):
    """One lattice with its fibers side by side, each near its centre and at a
    seeded angle, as the workloads module lays them out."""
    rng = np.random.default_rng(seed)
    nx, ny, nf, N, a = case["nx"], case["ny"], case["n_fibers"], case["n_beads"], case["a"]
    U = float(rng.uniform(0.008, 0.012))
    nu = case["nu"]
    if nu <= 0:
        # from Re, within the range of viscosities a run is set up with
        nu = min(0.6, max(0.02, 2.0 * U / ny * (2.0 * a * N) ** 2 / case["re"]))
    cen = [[(f + 0.5) * nx / nf + float(rng.uniform(-1, 1)), ny / 2.0 + float(rng.uniform(-1, 1))] for f in range(nf)]
    th = [float(rng.uniform(math.radians(30), math.radians(60))) for _ in range(nf)]
    base = wl.couette_only(nx, ny, u=U, nu=nu, init_couette=1 if nf else 0, precision=PRECISION[case["precision"]])
    return dict(base, re=case["re"], xi=case["xi"], a=a, n_beads=N, n_fibers=nf, stiffness_K=case["K"],
                centres=cen or [[0.0, 0.0]], theta0=th or [0.0], collision=case["collision"])


def _driven_config(case, seed):
    from paper_2212_14153_gb300 import studies
    rng = np.random.default_rng(seed)
    cfg = studies.driven_case(case["a"], case["r_eta"], case["r_xi"], case["Re_p"] * float(rng.uniform(0.9, 1.1)))
    L = cfg["nx"]
    cfg["centres"] = [[L / 2.0 + float(rng.uniform(-1, 1)), L / 2.0 + float(rng.uniform(-1, 1))]]
    return dict(cfg, precision=PRECISION[case["precision"]])


def _batch_configs(case, seed):
    """Lattices and bead counts from the case's layout, angles and stiffnesses
    from the seed."""
    lay, rng = np.random.default_rng(case["layout"]), np.random.default_rng(seed)
    out = []
    for _ in range(case["n"]):
        if case["family"] == "sweep":
            cfg = wl.sweep_instance(lay)
        else:
            cfg, _ = tumbling.tumbling_case(3.3, 0.2, float(lay.uniform(0.25, 3.0)), N=10, a=2.0)
        cfg["theta0"] = [float(rng.uniform(math.radians(30), math.radians(60)))]
        cfg["stiffness_K"] = float(10.0 ** rng.uniform(math.log10(3.3e-3), math.log10(3.3)))
        out.append(dict(cfg, precision=PRECISION[case["precision"]]))
    return out


def _configs(case, seed):
    if case["kind"] == "batch":
        return _batch_configs(case, seed)
    return [_driven_config(case, seed) if case["kind"] == "driven" else _fiber_config(case, seed)]


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True)


def _types(precision):
    """Result types: positions and densities, velocities."""
    if precision == "f64":
        return torch.float64, torch.float64
    return torch.float32, torch.float32 if precision == "f32" else torch.float16


def prepare(case, seed):
    cfgs = _configs(case, seed)
    if case["kind"] == "batch":
        cells = sum(c["nx"] * c["ny"] for c in cfgs)
        pool = 18 * ELEM[case["precision"]] * (cells + 64 * sum(c["ny"] for c in cfgs)) + 4096 * len(cfgs)
        b = fpd.Batch(PRECISION[case["precision"]], len(cfgs), pool, sum(c["n_beads"] for c in cfgs))
        return dict(case=case, batch=b, slots=[b.add(c, ENDLESS) for c in cfgs])
    cfg = cfgs[0]
    sim = fpd.Simulation(cfg, tuning="auto" if case.get("tuning") == "auto" else None)
    st = dict(case=case, sim=sim)
    if case.get("read") != "beads" or not sim.nb:
        # page-locked host buffers for the fields, and arrays to keep them in
        st["host"] = _pinned((3, cfg["ny"], cfg["nx"]))
        rt, ut = _types(case["precision"])
        st["keep"] = dict(u=torch.empty((2, cfg["ny"], cfg["nx"]), dtype=ut),
                          rho=torch.empty((cfg["ny"], cfg["nx"]), dtype=rt))
    return st


# --------------------------------------------------------------------- run
def _beads(R, V, precision):
    rt, ut = _types(precision)
    return dict(R=torch.from_numpy(R).to(rt), V=torch.from_numpy(V).to(ut))


def run(state):
    case = state["case"]
    precision = case["precision"]
    if case["kind"] == "batch":
        return _run_batch(case, state["batch"], state["slots"])
    sim, out = state["sim"], {}
    sim.step(case["steps"])
    if sim.nb:
        R, V, _, _ = sim.beads()
        out.update(_beads(R, V, precision))
    if "host" in state:
        h, keep = state["host"], state["keep"]
        sim.fields(out=(h[0].numpy(), h[1].numpy(), h[2].numpy()))
        if precision == "f64":
            out.update(u=h[:2], rho=h[2])
        else:
            keep["u"].copy_(h[:2])
            keep["rho"].copy_(h[2])
            out.update(keep)
    return out


def _run_batch(case, b, slots):
    left = case["steps"]
    while left > 0:
        left -= b.run(left)
    beads = [b.beads(s) for s in slots]
    out = _beads(np.concatenate([x[0] for x in beads]), np.concatenate([x[1] for x in beads]), case["precision"])
    if case["read"] == "fields":
        rt, ut = _types(case["precision"])
        f = [b.fields(s) for s in slots]
        out["u"] = torch.cat([torch.from_numpy(x).reshape(-1).to(ut) for ux, uy, _ in f for x in (ux, uy)])
        out["rho"] = torch.cat([torch.from_numpy(r).reshape(-1).to(rt) for _, _, r in f])
    return out


# -------------------------------------------------------------------- work
def work(case):
    """Per step each of the nine populations of a cell is read once and
    written once; about 120 operations a cell.  Fields read back are three
    doubles a cell."""
    cfgs = _configs(case, 0)
    cells = sum(c["nx"] * c["ny"] for c in cfgs)
    fields = 0 if case.get("read") == "beads" and cfgs[0]["n_beads"] else 24 * cells
    return {"bytes": case["steps"] * cells * 18 * ELEM[case["precision"]] + fields, "flops": case["steps"] * cells * 120}


# ------------------------------------------------- the method in 64 bits
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _moments(dev):
    """Lallemand-Luo moment matrix (rho, e, eps, jx, qx, jy, qy, pxx, pxy)."""
    c = [(x, y, x * x + y * y) for x, y in zip(CX, CY)]
    rows = [[1.0] * 9, [3.0 * s - 4 for _, _, s in c], [4 - 10.5 * s + 4.5 * s * s for _, _, s in c],
            [float(x) for x, _, _ in c], [x * (3.0 * s - 5) for x, _, s in c],
            [float(y) for _, y, _ in c], [y * (3.0 * s - 5) for _, y, s in c],
            [float(x * x - y * y) for x, y, _ in c], [float(x * y) for x, y, _ in c]]
    return torch.tensor(rows, dtype=torch.float64, device=dev)


class _Reference:
    """The time step of the method (one instance) in plain 64-bit torch."""

    def __init__(self, cfg, dev):
        self.c, self.dev = cfg, dev
        nx, ny = cfg["nx"], cfg["ny"]
        kw = dict(dtype=torch.float64, device=dev)
        self.l0 = 2.0 * cfg["a"]
        gd = (cfg["u_top"] - cfg["u_bottom"]) / ny
        lc = cfg["n_beads"] * self.l0
        self.nu = cfg["nu_f"] if cfg["nu_f"] > 0 else abs(gd) * lc * lc / cfg["re"]
        self.ks = cfg["k_s"] if cfg["k_s"] >= 0 else 0.25 * math.pi * cfg["a"] ** 2 * self.l0 ** 2
        self.kb = cfg["stiffness_K"] * self.nu * abs(gd) * lc * lc / 2 if cfg["stiffness_K"] > 0 else cfg["k_b"]
        self.kev = cfg["k_ev"] if cfg["k_ev"] >= 0 else self.ks / self.l0 ** 2
        self.per_y = bool(cfg.get("periodic_y", 0))
        self.M = _moments(dev)
        self.Mi = torch.linalg.inv(self.M.cpu()).to(dev)
        self.cx = torch.tensor(CX, **kw)[:, None]
        self.cy = torch.tensor(CY, **kw)[:, None]
        self.w = torch.tensor(W, **kw)[:, None]
        y = torch.arange(ny, **kw) + 0.5
        ux = (cfg["u_bottom"] + gd * y if cfg["init_couette"] else 0 * y)[:, None].expand(ny, nx).reshape(-1)
        self.g = self._eq(0 * ux, 1 + 0 * ux, ux, 0 * ux)  # pulled populations less their rest values
        self.nb = cfg["n_beads"] * cfg["n_fibers"]
        self.V = torch.zeros((self.nb, 2), **kw)
        self.F = self.phi = None
        if self.nb:
            i = torch.arange(cfg["n_beads"], **kw) - (cfg["n_beads"] - 1) / 2.0
            R = [[cx + float(o) * self.l0 * math.cos(t), cy + float(o) * self.l0 * math.sin(t)]
                 for (cx, cy), t in zip(cfg["centres"], cfg["theta0"]) for o in i]
            self.R = torch.tensor(R, **kw)

    def _eq(self, drho, rho, ux, uy):
        cu = self.cx * ux + self.cy * uy
        return self.w * (drho + rho * (3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy)))

    def _profiles(self):
        """Cells near each bead (flat index, profile phi; zero outside the
        cutoff and the walls) and S = sum phi."""
        c, nx, ny = self.c, self.c["nx"], self.c["ny"]
        rc = c["a"] + c["phi_cut"] * c["xi"]
        h = math.ceil(rc) + 2

        def axis(r, n, periodic):
            if periodic and 2 * h + 1 >= n:
                i = torch.arange(n, device=self.dev)[None].expand(len(r), n)
            else:
                i = torch.floor(r).long()[:, None] + torch.arange(-h, h + 1, device=self.dev)
            d = i + 0.5 - r[:, None]
            if periodic:
                return i % n, d - n * torch.floor(d / n + 0.5), torch.ones_like(i, dtype=torch.bool)
            return i.clamp(0, n - 1), d, (i >= 0) & (i < n)

        ix, dx, _ = axis(self.R[:, 0], nx, True)
        iy, dy, ok = axis(self.R[:, 1], ny, self.per_y)
        r2 = dx[:, None, :] ** 2 + dy[:, :, None] ** 2
        phi = 0.5 * (torch.tanh((c["a"] - r2.sqrt()) / c["xi"]) + 1.0)
        phi = torch.where((r2 < rc * rc) & ok[:, :, None], phi, torch.zeros_like(phi))
        idx = iy[:, :, None] * nx + ix[:, None, :]
        self.idx, self.phi = idx.reshape(self.nb, -1), phi.reshape(self.nb, -1)
        self.S = self.phi.sum(1)

    def _forces(self):
        c, N, R = self.c, self.c["n_beads"], self.R
        F = torch.zeros_like(R)
        for f in range(c["n_fibers"]):
            r = R[f * N:(f + 1) * N]
            if N > 1:
                d = r[1:] - r[:-1]
                L = d.norm(dim=1, keepdim=True)
                t = d / L
                pad = torch.zeros((1, 2), dtype=R.dtype, device=self.dev)
                nb = torch.cat([t[1:], pad]) + torch.cat([pad, t[:-1]])  # tangents beside each segment
                bend = self.kb * (nb - (nb * t).sum(1, keepdim=True) * t) / L
                pull = self.ks / self.l0 ** 2 * (L - self.l0) * t - bend
                F[f * N:f * N + N - 1] += pull
                F[f * N + 1:f * N + N] -= pull
        if self.kev:
            d = R[:, None] - R[None]
            nx, ny = c["nx"], c["ny"]
            dx = d[..., 0] - nx * torch.round(d[..., 0] / nx)
            dy = d[..., 1] - ny * torch.round(d[..., 1] / ny) if self.per_y else d[..., 1]
            r = (dx * dx + dy * dy).sqrt()
            k = torch.arange(self.nb, device=self.dev)
            bonded = (k[:, None] // N == k[None] // N) & ((k[:, None] - k[None]).abs() < 2)
            m = torch.where((r < self.l0) & (r > 0) & ~bonded, self.kev * (self.l0 - r) / r.clamp(min=1e-300), 0 * r)
            F += torch.stack([(m * dx).sum(1), (m * dy).sum(1)], 1)
        return F + torch.tensor([c.get("bead_fx", 0.0), c.get("bead_fy", 0.0)], dtype=R.dtype, device=self.dev)

    def _velocity(self):
        drho = self.g.sum(0)
        rho = 1 + drho
        Fx, Fy = self.F if self.F is not None else (self.c["gx"], self.c["gy"])
        return drho, rho, ((self.cx * self.g).sum(0) + 0.5 * Fx) / rho, ((self.cy * self.g).sum(0) + 0.5 * Fy) / rho

    def step(self):
        c, nx, ny = self.c, self.c["nx"], self.c["ny"]
        if self.nb:
            if self.phi is not None:  # Eq. 5 with the force that drove the last collision
                _, _, ux, uy = self._velocity()
                self.V = torch.stack([(self.phi * ux[self.idx]).sum(1), (self.phi * uy[self.idx]).sum(1)], 1) / self.S[:, None]
                self.R = self.R + self.V
            self._profiles()
            G = self._forces() / self.S[:, None]
            Phi, Fx, Fy = (torch.zeros(nx * ny, dtype=torch.float64, device=self.dev) for _ in range(3))
            flat = self.idx.reshape(-1)
            Phi.index_add_(0, flat, self.phi.reshape(-1))
            Fx.index_add_(0, flat, (self.phi * G[:, :1]).reshape(-1))
            Fy.index_add_(0, flat, (self.phi * G[:, 1:]).reshape(-1))
            self.F = (Fx + c["gx"], Fy + c["gy"])
            nu = self.nu * (1 + (c["visc_ratio"] - 1) * Phi)
        else:
            zero = torch.zeros(nx * ny, dtype=torch.float64, device=self.dev)
            self.F, nu = (zero + c["gx"], zero + c["gy"]), zero + self.nu
        drho, rho, ux, uy = self._velocity()
        Fx, Fy = self.F
        s_nu = 1 / (3 * nu + 0.5)
        if c["collision"] == LL:
            s_e, s_eps, s_q = c["s_e"], c["s_eps"], c["s_q"]
        else:
            s_e = s_eps = s_nu
            s_q = s_nu if c["collision"] == BGK else 1 / (0.5 + 0.1875 / (1 / s_nu - 0.5))
        cu, cF = self.cx * ux + self.cy * uy, self.cx * Fx + self.cy * Fy
        src = self.w * (3 * (cF - (ux * Fx + uy * Fy)) + 9 * cu * cF)
        m, ms = self.M @ (self.g - self._eq(drho, rho, ux, uy)), self.M @ src
        for row, s in enumerate((0.0, s_e, s_eps, 0.0, s_q, 0.0, s_q, s_nu, s_nu)):
            # momentum at rate 0: the source brings all of F less the half that u holds
            ms[row] = (1 - 0.5 * s) * ms[row] - s * m[row]
        g = (self.g + self.Mi @ ms).reshape(9, ny, nx)
        new = torch.empty_like(g)
        for k in range(9):
            p = torch.roll(g[k], (CY[k], CX[k]), (0, 1))
            if not self.per_y and CY[k]:
                row, u = (0, c["u_bottom"]) if CY[k] > 0 else (ny - 1, c["u_top"])
                p[row] = g[OPP[k]][row] + 6 * W[k] * CX[k] * u
            new[k] = p
        self.g = new.reshape(9, -1)

    def result(self, fields):
        out = {}
        _, rho, ux, uy = self._velocity()
        if self.nb:
            out.update(R=self.R.cpu(), V=self.V.cpu())
        if fields:
            shape = (self.c["ny"], self.c["nx"])
            out.update(u=torch.stack([ux.reshape(shape), uy.reshape(shape)]).cpu(), rho=rho.reshape(shape).cpu())
        return out


def exact(case, seed):
    """What run returns for a new state, computed step by step in plain
    64-bit torch; None for batches too long to follow one by one."""
    cfgs = _configs(case, seed)
    cells = sum(c["nx"] * c["ny"] for c in cfgs)
    if len(cfgs) * case["steps"] > 8000 or cells * case["steps"] > 1.2e9:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    fields = case.get("read") != "beads" or not cfgs[0]["n_beads"]
    got = []
    for cfg in cfgs:
        ref = _Reference(cfg, dev)
        for _ in range(case["steps"]):
            ref.step()
        got.append(ref.result(fields))
    if case["kind"] != "batch":
        return got[0]
    out = {k: torch.cat([g[k] for g in got]) for k in ("R", "V")}
    if fields:
        out["u"] = torch.cat([x.reshape(-1) for g in got for x in g["u"]])
        out["rho"] = torch.cat([g["rho"].reshape(-1) for g in got])
    return out
