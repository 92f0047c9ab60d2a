"""What a user of this library has it do, as measurable cases.

A pass takes a lattice (or a batch of them, or a channel with obstacles)
through one interval between two readings of its state: `step(n)`, then the
fields rho, phi, u on the device and the statistics, and where the run is
about them the contact angle or the meniscus.  The state goes on from pass to
pass, as in a run.  FP32 lattices keep their snapshots in FP32, FP64 ones in
FP64.

`exact` is the method in plain torch and FP64, node by node through gather
tables (pull-streaming with bounce-back, wetting ghosts, Appendix A
equilibria, BGK or MRT): none of the library's code.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch

import paper_0812_1282_gb300 as lbf

A = KAPPA = 0.04
EX = (0, 1, -1, 0, 0, 1, -1, -1, 1)
EY = (0, 0, 0, 1, -1, 1, -1, 1, -1)
OPP = (0, 2, 1, 4, 3, 6, 5, 8, 7)


# ------------------------------------------------------------------- cases
def listed():
    return [
        # The spurious-current stripe of Sec. IV.A, the smallest lattice anyone
        # steps (20000 times): latency of one step.
        dict(name="stripe_28x15_fp64", kind="lattice", nx=28, ny=15, precision="fp64",
             collision="bgk", init="stripe", walls=True, tau_a=10.0, tau_b=10.0, theta=90.0,
             steps=500),
        # The 100 x 50 parity drop: a short run from a given phi, read once.
        dict(name="drop_100x50_bgk_fp64", kind="lattice", nx=100, ny=50, precision="fp64",
             collision="bgk", init="drop", walls=True, tau_a=1.0, tau_b=1.0, theta=90.0,
             angle=True, steps=500),
        # The contact-angle sweep, its readings every 500 steps, in the library's
        # default precision.
        dict(name="sweep_200x100_mrt_fp64", kind="lattice", nx=200, ny=100, precision="fp64",
             collision="mrt", init="drop", walls=True, tau_a=1.5, tau_b=0.6, theta=60.0,
             angle=True, steps=500),
        # The same in FP32 with compact g storage, as whoever wants the speed has it.
        dict(name="sweep_200x100_mrt_compact", kind="lattice", nx=200, ny=100, precision="fp32",
             compact=True, collision="mrt", init="drop", walls=True, tau_a=1.5, tau_b=0.6,
             theta=120.0, angle=True, steps=500),
        # The quasi-static ramp (300 x 100, Gamma 0.5, tau 3 / 0.7): the wetting
        # gradient changes, then a stretch of steps; FP32, full storage.
        dict(name="ramp_300x100_mrt_fp32", kind="ramp", nx=300, ny=100, precision="fp32",
             collision="mrt", init="drop", walls=True, gamma_mob=0.5, tau_a=3.0, tau_b=0.7,
             theta=60.0, angle=True, steps=1000),
        # Capillary filling (Sec. VI), the front read every 500 steps.
        dict(name="capillary_1000x120_fp32", kind="channel", nx=1000, ny=120, res_len=200,
             ch_w=40, precision="fp32", collision="mrt", tau_a=1.5, tau_b=0.6, theta=60.0,
             front=True, tune=2, steps=500),
        # A smaller channel of ragged size in FP64.
        dict(name="channel_401x77_fp64", kind="channel", nx=401, ny=77, res_len=101, ch_w=25,
             precision="fp64", collision="mrt", tau_a=1.5, tau_b=0.6, theta=60.0, tune=2,
             steps=200),
        # 256 sessile drops of uneven sizes in one batch: the many-run job.
        dict(name="batch_256_drops_compact", kind="batch", n=256, lo=64, hi=512, sizes=2026,
             precision="fp32", compact=True, collision="mrt", tune=2, steps=256),
        # A few smaller drops in full storage with the schedule a batch starts with.
        dict(name="batch_40_drops_fp32", kind="batch", n=40, lo=48, hi=200, sizes=7,
             precision="fp32", collision="mrt", tune=0, steps=256),
        # A periodic spinodal lattice of odd sizes, BGK, full FP32 storage.
        dict(name="spinodal_3001x2047_bgk_fp32", kind="lattice", nx=3001, ny=2047,
             precision="fp32", collision="bgk", init="random", walls=False, tau_a=1.5, tau_b=0.6,
             theta=90.0, tune=1, steps=100),
        # The spinodal lattice in FP64.
        dict(name="spinodal_2048_mrt_fp64", kind="lattice", nx=2048, ny=2048, precision="fp64",
             collision="mrt", init="random", walls=True, tau_a=1.5, tau_b=0.6, theta=90.0,
             tune=1, steps=50),
        # The headline lattice: 8192^2, FP32, compact g, statistics every 100 steps.
        dict(name="spinodal_8192_mrt_compact", kind="lattice", nx=8192, ny=8192,
             precision="fp32", compact=True, collision="mrt", init="random", walls=True,
             tau_a=1.5, tau_b=0.6, theta=90.0, tune=1, steps=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("lattice", "lattice", "lattice", "lattice", "channel", "batch", "batch",
                       "ramp"))
    coll = rng.choice(("bgk", "mrt"))
    storage = rng.choice(("fp64", "fp32", "compact"))
    base = dict(kind=kind, precision="fp64" if storage == "fp64" else "fp32", collision=coll,
                compact=storage == "compact")
    # steps between two readings, fewer where the lattice is large or FP64
    def steps(nodes):
        most = {"fp64": 2e8, "fp32": 3e9, "compact": 5e9}[storage] / nodes
        return int(max(3, min(rng.choice((100, 250, 500)), most)))
    taus = rng.choice(((1.0, 1.0), (1.5, 0.6), (0.8, 0.6), (3.0, 0.7)))
    base.update(tau_a=taus[0], tau_b=taus[1])
    if kind == "batch":
        n = _log(rng, 4, 256)
        lo = rng.randint(24, 96)
        hi = min(512, lo + _log(rng, 8, 420))
        if storage == "fp64":
            n = min(n, 64)
        return dict(base, n=n, lo=lo, hi=hi, sizes=rng.randint(1, 1 << 20), collision="mrt",
                    tune=rng.choice((0, 2)), steps=steps(n * ((lo + hi) / 2) ** 2))
    if kind == "channel":
        if storage == "compact":  # obstacles need the full storage
            storage = "fp32"
            base["compact"] = False
        nx, ny = _log(rng, 120, 2000), rng.randint(48, 200)
        n = steps(nx * ny)
        # a front to read: not before it has bent, and not in a short channel
        # that fills up
        return dict(base, nx=nx, ny=ny, res_len=rng.randint(nx // 6, nx // 3),
                    ch_w=rng.randint(ny // 4, ny // 2), collision="mrt", tau_a=1.5, tau_b=0.6,
                    theta=rng.uniform(50.0, 80.0), front=n >= 400 and nx >= 700, tune=2, steps=n)
    if kind == "ramp":
        nx = _log(rng, 80, 600)
        ny = max(24, nx // 3 + rng.randint(-7, 7))
        return dict(base, nx=nx, ny=ny, init="drop", walls=True, gamma_mob=0.5, angle=True,
                    theta=rng.uniform(50.0, 85.0), steps=steps(nx * ny))
    top = 2600 if storage == "fp64" else 8192
    nx, ny = _log(rng, 24, top), _log(rng, 15, top)
    if rng.random() < 0.5:
        ny = max(15, min(top, nx // 2 + rng.randint(0, 3)))
    init = rng.choice(("drop", "random"))
    walls = init == "drop" or rng.random() < 0.5
    return dict(base, nx=nx, ny=ny, init=init, walls=walls,
                theta=rng.uniform(60.0, 120.0) if init == "drop" else 90.0,
                tune=1 if nx * ny > 500000 else 0, steps=steps(nx * ny))


def work(case):
    """Per node update: the populations read and written once (9 f + 9 g, or
    9 f + 4 numbers with compact g); the flops of Steps 1-4 in their plainest
    form.  A channel updates its fluid nodes only."""
    nodes = sum(nx * ny for nx, ny in _sizes(case))
    if case["kind"] == "channel":
        nodes -= (case["nx"] - case["res_len"]) * (case["ny"] - case["ch_w"])
    per = 288 if case["precision"] == "fp64" else (104 if case.get("compact") else 144)
    return {"bytes": float(nodes) * per * case["steps"], "flops": float(nodes) * 250 * case["steps"]}


# -------------------------------------------------------- inputs from a seed
def _sizes(case):
    if case["kind"] != "batch":
        return [(case["nx"], case["ny"])]
    r = random.Random(case["sizes"])
    return [(r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"]))
            for _ in range(case["n"])]


def _domains(case, seed):
    """Per domain: size, parameters and initial state."""
    rng = random.Random(seed * 1000003 + 17)
    out = []
    for nx, ny in _sizes(case):
        d = dict(nx=nx, ny=ny, walls=case.get("walls", True), theta=case.get("theta", 90.0),
                 tau_a=case.get("tau_a", 1.5), tau_b=case.get("tau_b", 0.6),
                 gamma=case.get("gamma_mob", 0.1), init=case.get("init", "drop"))
        if case["kind"] == "batch":
            ratio = rng.choice((1, 3, 10))
            d.update(theta=rng.uniform(30.0, 150.0), tau_b=0.6, tau_a=0.5 + 0.1 * ratio)
        # drops that clear the side and the top
        R = 0.3 * min(nx, ny) if case["kind"] == "batch" else 0.2 * min(nx, 2 * ny)
        d.update(R=R * rng.uniform(0.9, 1.1), cx=nx / 2 + rng.uniform(-1.0, 1.0), seed=rng.randrange(1 << 40),
                 xa=nx / 4 + rng.uniform(-0.4, 0.4), xb=3 * nx / 4 + rng.uniform(-0.4, 0.4),
                 tilt=rng.uniform(0.02, 0.05), theta=d["theta"] + rng.uniform(-1.0, 1.0))
        d["h"] = lbf.lb_wetting_h(d["theta"], A, KAPPA) if d["init"] == "drop" else 0.0
        out.append(d)
    return out


def _stripe_phi(d):
    """A stripe of alpha across the channel with slightly bent edges."""
    ell = math.sqrt(2 * KAPPA / A)
    x = np.arange(d["nx"])[None, :]
    bend = d["tilt"] * (np.arange(d["ny"])[:, None] - d["ny"] / 2)
    return np.where(x < d["nx"] / 2, np.tanh((x - d["xa"] - bend) / ell),
                    -np.tanh((x - d["xb"] - bend) / ell))


class State:
    pass


def prepare(case, seed):
    doms = _domains(case, seed)
    s = State()
    s.case, s.doms = case, doms
    fp32 = case["precision"] == "fp32"

    def par(d):
        return lbf.params(a=A, kappa=KAPPA, gamma_mob=d["gamma"], tau_alpha=d["tau_a"],
                          tau_beta=d["tau_b"], collision=case["collision"],
                          h_bottom=0.0 if case["kind"] == "channel" else d["h"],
                          precision=case["precision"], walls=d["walls"],
                          step2_relax_momentum=_relax(case),
                          compact_g=bool(case.get("compact")))

    if case["kind"] == "batch":
        s.sim = lbf.Batch([par(d) for d in doms], [d["nx"] for d in doms],
                          [d["ny"] for d in doms])
    else:
        s.sim = lbf.Lattice(par(doms[0]), doms[0]["nx"], doms[0]["ny"])
    if case["kind"] == "channel":
        s.sim.init_channel(case["res_len"], case["ch_w"], doms[0]["h"], 0.0)
    else:
        _init(s)
    if case.get("tune"):
        s.sim.autotune(reps=case["tune"])
    n = sum(d["nx"] * d["ny"] for d in doms)
    s.out = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(4)]
    s.keep = torch.float32 if fp32 else torch.float64
    s.stats = lbf.Stats()
    s.ramp = 0
    return s


def _relax(case):
    """The momentum-relaxing reading of Step 2, stable at every angle; the
    spinodal lattices have neutral walls and take the literal one."""
    return case["collision"] == "mrt" and case.get("init") != "random"


def _init(s):
    for k, d in enumerate(s.doms):
        if d["init"] == "random":
            s.sim.init_random(0.1, d["seed"], dom=k)
        elif d["init"] == "stripe":
            s.sim.init_phi(_stripe_phi(d), dom=k)
        else:
            s.sim.init_drop(d["R"], d["cx"], -0.5, dom=k)


def _ramp_h(d, k):
    """The wetting gradient after k changes: up to its end value and back."""
    t = (k % 400) / 200.0
    return d["h"] * (1.0 + 0.2 * (t if t <= 1.0 else 2.0 - t))


# --------------------------------------------------------------- one pass
def run(s):
    case, sim = s.case, s.sim
    if case["kind"] == "ramp":
        s.ramp += 1
        sim.set_wetting(_ramp_h(s.doms[0], s.ramp), 0.0)
    sim.step(case["steps"])
    at, mass, max_u, bad = 0, 0.0, 0.0, 0
    for k, d in enumerate(s.doms):
        p = [ctypes.c_void_p(t.data_ptr() + 8 * at) for t in s.out]
        rc = lbf.lib().lb_moments(sim.h, k, 1, *p, ctypes.byref(s.stats))
        if rc != lbf.LB_OK:
            raise lbf.LBError(rc, lbf.lib().lb_last_error().decode())
        mass += s.stats.mass
        max_u = max(max_u, s.stats.max_u)
        bad += s.stats.nonfinite
        at += d["nx"] * d["ny"]
    shape = (-1,) if case["kind"] == "batch" else (s.doms[0]["ny"], s.doms[0]["nx"])
    out = {n: t.to(s.keep).view(shape) for n, t in zip(("rho", "phi", "ux", "uy"), s.out)}
    out.update(mass=mass, max_u=max_u, nonfinite=bad)
    if case.get("angle"):
        out["theta"], out["R"] = sim.contact_angle()[:2]
    if case.get("front"):
        y0 = (case["ny"] - case["ch_w"]) // 2
        out["front"], out["theta"], out["R"] = sim.meniscus(case["res_len"], case["nx"], y0,
                                                            y0 + case["ch_w"])
    return out


# ------------------------------------------------- the same in 64 bits, plain
def _channel_cls(case):
    nx, ny, w = case["nx"], case["ny"], case["ch_w"]
    y0 = (ny - w) // 2
    cls = np.zeros((ny, nx), np.uint8)
    cls[:, case["res_len"]:] = 2
    cls[y0 - 1, case["res_len"]:] = 1
    cls[y0 + w, case["res_len"]:] = 1
    cls[y0:y0 + w, case["res_len"]:] = 0
    return cls


class _Plain:
    """Nodes of all domains in one row; f (less its rest weights) and g as
    [9][nodes], and tables of where each population and each phi neighbour
    comes from.  phi values beyond `nodes` are the wetting ghosts."""

    def __init__(self, case, doms, dev):
        self.dev, self.mrt, self.relax = dev, case["collision"] == "mrt", _relax(case)
        sizes = [d["nx"] * d["ny"] for d in doms]
        self.N = N = sum(sizes)
        self.pull = torch.empty((9, N), dtype=torch.int64, device=dev)
        self.nb = torch.empty((9, N), dtype=torch.int64, device=dev)
        self.fluid = None
        near = torch.zeros(N, dtype=torch.bool, device=dev)
        per = {k: torch.empty(N, dtype=torch.float64, device=dev) for k in ("ta", "tb")}
        gidx, gcnt, gh, off = [], [], [], 0
        for d, n in zip(doms, sizes):
            cls = _channel_cls(case) if case["kind"] == "channel" else None
            hb = 0.0 if cls is not None else d["h"]
            at = sum(len(c) for c in gcnt)
            i, c, h = self._domain(d, cls, off, N + at, near)
            gidx.append(i + off)
            gcnt.append(c)
            gh.append(np.where(h == -1.0, hb, np.where(h == -2.0, 0.0, np.where(h == 1.0, d["h"],
                                                                               0.0))))
            per["ta"][off:off + n] = d["tau_a"]
            per["tb"][off:off + n] = d["tau_b"]
            off += n
        put = lambda v, t: torch.as_tensor(np.concatenate(v), dtype=t, device=dev)  # noqa: E731
        self.gidx, self.gcnt = put(gidx, torch.int64), put(gcnt, torch.float64)
        self.gh = put(gh, torch.float64)
        one = all((d["tau_a"], d["tau_b"]) == (doms[0]["tau_a"], doms[0]["tau_b"]) for d in doms)
        self.ta, self.tb = (doms[0]["tau_a"], doms[0]["tau_b"]) if one else (per["ta"], per["tb"])
        self.near = near if self.mrt and bool(near.any()) else None  # Step 2: MRT only
        self.gamma = doms[0]["gamma"]

    def _domain(self, d, cls, off, ghost0, near):
        """Tables of one domain; returns its ghosts: up to four sources each
        (padded with the last), their count, and -1 / -2 for a bottom / top
        wall ghost or the obstacle's class."""
        nx, ny, dev = d["nx"], d["ny"], self.dev
        n = nx * ny
        own = torch.arange(n, device=dev)
        y, x = own // nx, own % nx
        solid = None if cls is None else torch.as_tensor(cls.reshape(-1) != 0, device=dev)
        idx, cnt, what = [], [], []
        ghost_of = None
        if cls is None:
            if d["walls"]:
                for row, code in ((1, -1.0), (ny - 2, -2.0)):  # the mirror about the boundary row
                    i = row * nx + np.arange(nx)
                    idx.append(np.stack([i] * 4, 1))
                    cnt.append(np.ones(nx))
                    what.append(np.full(nx, code))
        else:
            ghost_of = np.full((ny + 2, nx), -1, np.int64)

            def flu(qx, qy):
                return 0 <= qy < ny and cls[qy, qx % nx] == 0

            for sy in range(-1, ny + 1):
                for sx in range(nx):
                    if flu(sx, sy):
                        continue
                    for dirs in (range(1, 5), range(5, 9)):
                        src = [((sy + 2 * EY[k]) * nx + (sx + 2 * EX[k]) % nx) for k in dirs
                               if flu(sx + EX[k], sy + EY[k])]
                        if src:
                            ghost_of[sy + 1, sx] = len(cnt)
                            idx.append(src + [src[-1]] * (4 - len(src)))
                            cnt.append(float(len(src)))
                            what.append(-1.0 if sy < 0 else (-2.0 if sy >= ny else
                                                             float(cls[sy, sx])))
                            break
            ghost_of = torch.as_tensor(ghost_of.reshape(-1), device=dev)
            idx, cnt, what = [np.array(idx)], [np.array(cnt)], [np.array(what)]
            self.fluid = ~solid
        for i in range(9):
            sx, sy = (x - EX[i]) % nx, y - EY[i]
            out = (sy < 0) | (sy >= ny) if d["walls"] else torch.zeros_like(y, dtype=torch.bool)
            src = (sy % ny) * nx + sx
            if solid is not None:
                out = out | solid[src]
            self.pull[i, off:off + n] = torch.where(out, OPP[i] * self.N + off + own,
                                                    i * self.N + off + src)
            qx, qy = (x + EX[i]) % nx, y + EY[i]
            ins = (qy % ny) * nx + qx + off
            if cls is not None:
                g = ghost_of[(qy + 1) * nx + qx]
                beyond = (qy < 0) | (qy >= ny) | solid[(qy % ny) * nx + qx]
                self.nb[i, off:off + n] = torch.where(beyond, ghost0 + g.clamp(min=0), ins)
                near[off:off + n] |= beyond & ~solid
            elif d["walls"]:
                v = torch.where(qy < 0, ghost0 + qx, ins)
                self.nb[i, off:off + n] = torch.where(qy >= ny, ghost0 + nx + qx, v)
                near[off:off + n] |= (qy < 0) | (qy >= ny)
            else:
                self.nb[i, off:off + n] = ins
        if not cnt:
            return np.zeros((0, 4), np.int64), np.zeros(0), np.zeros(0)
        return np.concatenate(idx), np.concatenate(cnt), np.concatenate(what)

    def stencils(self, phi):
        if len(self.gcnt):
            v = phi[self.gidx]
            total = v[:, 0].clone()
            for k in range(1, 4):
                total += torch.where(self.gcnt > k, v[:, k], torch.zeros_like(total))
            phi = torch.cat((phi, total / self.gcnt - 2.0 * self.gh))
        c, e, w, n, s, ne, sw, nw, se = (phi[self.nb[i]] for i in range(9))
        dx = (4 * (e - w) + (ne - nw) + (se - sw)) / 12
        dy = (4 * (n - s) + (ne - se) + (nw - sw)) / 12
        return dx, dy, (4 * (e + w + n + s) + (ne + nw + se + sw) - 20 * c) / 6

    def equilibria(self, drho, phi, jx, jy, ux, uy, dx, dy, lap):
        """Appendix A with c = 1: f less the rest weights, and g."""
        p2 = phi * phi
        iso = drho / 3 + A * (-0.5 * p2 + 0.75 * p2 * p2) - KAPPA * phi * lap
        mu = A * (p2 * phi - phi) - KAPPA * lap
        xx, yy, xy = jx * ux, jy * uy, jx * uy
        kxx, kyy, kxy = KAPPA * dx * dx, KAPPA * dy * dy, KAPPA * dx * dy
        F, G = [None] * 9, [None] * 9
        for i in range(1, 9):
            ex, ey, w = EX[i], EY[i], (1 / 3 if i < 5 else 1 / 12)
            eu = ex * jx + ey * jy
            q = 1.5 * (ex * ex * xx + ey * ey * yy + 2 * ex * ey * xy) - 0.5 * (xx + yy)
            if i < 5:
                wk = (kxx / 3 - kyy / 6) if ex else (kyy / 3 - kxx / 6)
            else:
                wk = -(kxx + kyy) / 24 + ex * ey * kxy / 4
            F[i] = w * (iso + eu + q) + wk
            gu = ex * ux + ey * uy
            G[i] = w * (self.gamma * mu + phi * (gu + 1.5 * gu * gu - 0.5 * (ux * ux + uy * uy)))
        F[0] = drho - sum(F[1:])
        G[0] = phi - sum(G[1:])
        return torch.stack(F), torch.stack(G)

    def start(self, phi):
        z = torch.zeros_like(phi)
        self.F, self.G = self.equilibria(z, phi, z, z, z, z, *self.stencils(phi))
        if self.fluid is not None:
            self.F *= self.fluid
            self.G *= self.fluid

    def step(self):
        f, g = self.F.view(-1)[self.pull], self.G.view(-1)[self.pull]
        phi, drho = g.sum(0), f.sum(0)
        dx, dy, lap = self.stencils(phi)
        jx = f[1] - f[2] + f[5] - f[6] - f[7] + f[8]
        jy = f[3] - f[4] + f[5] - f[6] + f[7] - f[8]
        jxe, jye = (jx, jy) if self.near is None else (torch.where(self.near, 0.0, jx),
                                                      torch.where(self.near, 0.0, jy))
        fe, ge = self.equilibria(drho, phi, jxe, jye, jxe / (1 + drho), jye / (1 + drho), dx, dy,
                                 lap)
        om = 1 / (self.tb + 0.5 * (phi + 1) * (self.ta - self.tb))
        if self.mrt:
            # S = diag(0,1,1,0,1,0,1,w,w): the two stress moments relax at w, the
            # momentum of a Step-2 node is kept (or, relaxing it, dropped)
            k = f - fe
            m7 = (1 - om) * (k[1] + k[2] - k[3] - k[4]) / 4
            m8 = (1 - om) * (k[5] + k[6] - k[7] - k[8]) / 4
            for i in range(1, 9):
                fe[i] += (m7 if i < 3 else -m7) if i < 5 else (m8 if i < 7 else -m8)
                if self.near is not None and not self.relax:
                    fe[i] += (EX[i] * (jx - jxe) + EY[i] * (jy - jye)) / 6
            fe[0] = drho - fe[1:].sum(0)
        else:
            fe += (1 - om) * (f - fe)
        if self.fluid is not None:
            fe *= self.fluid
            ge *= self.fluid
        self.F, self.G = fe, ge

    def fields(self):
        f = self.F
        rho, phi = 1 + f.sum(0), self.G.sum(0)
        ux = (f[1] - f[2] + f[5] - f[6] - f[7] + f[8]) / rho
        uy = (f[3] - f[4] + f[5] - f[6] + f[7] - f[8]) / rho
        if self.fluid is not None:
            rho, phi = rho * self.fluid, phi * self.fluid
        return rho, phi, ux, uy


def _plain_phi(case, d, dev):
    nx, ny = d["nx"], d["ny"]
    y, x = torch.meshgrid(torch.arange(ny, device=dev, dtype=torch.float64),
                          torch.arange(nx, device=dev, dtype=torch.float64), indexing="ij")
    ell = math.sqrt(2 * KAPPA / A)
    if case["kind"] == "channel":
        phi = torch.tanh(torch.minimum(x - (case["res_len"] // 2 - 0.5),
                                       case["res_len"] - 0.5 - x) / ell)
        phi = torch.where(torch.as_tensor(_channel_cls(case) != 0, device=dev), 0.0, phi)
    elif d["init"] == "random":
        def shr(z, k):  # logical shift of a 64-bit word
            return (z >> k) & ((1 << (64 - k)) - 1)

        def word(v):  # an unsigned 64-bit constant as a signed one
            return v - (1 << 64) if v >= 1 << 63 else v

        k = torch.arange(1, nx * ny + 1, device=dev, dtype=torch.int64)
        z = d["seed"] + k * word(0x9E3779B97F4A7C15)
        z = (z ^ shr(z, 30)) * word(0xBF58476D1CE4E5B9)
        z = (z ^ shr(z, 27)) * word(0x94D049BB133111EB)
        z = z ^ shr(z, 31)
        phi = 0.1 * (2 * (shr(z, 11).double() * 2.0 ** -53) - 1)
    elif d["init"] == "stripe":
        phi = torch.as_tensor(_stripe_phi(d), device=dev)
    else:
        phi = torch.tanh((d["R"] - torch.sqrt((x - d["cx"]) ** 2 + (y + 0.5) ** 2)) / ell)
    return phi.reshape(-1)


def _crossings(phi, fluid):
    """The phi = 0 points on the links of a lattice periodic in x."""
    pts = []
    ny, nx = phi.shape
    for ex, ey in ((1, 0), (0, 1)):
        b = np.roll(phi, -ex, 1) if ex else phi[1:]
        a = phi if ex else phi[:-1]
        ok = fluid & np.roll(fluid, -1, 1) if ex else fluid[:-1] & fluid[1:]
        y, x = np.nonzero((a * b < 0) & ok)
        t = a[y, x] / (a[y, x] - b[y, x])
        pts.append(np.stack([x + ex * t, y + ey * t], 1))
    return np.concatenate(pts)


def _circle(p):
    m = p.mean(0)
    q = p - m
    s = np.linalg.lstsq(np.column_stack([q, np.ones(len(q))]), (q * q).sum(1), rcond=None)[0]
    cx, cy = s[0] / 2, s[1] / 2
    r = math.sqrt(s[2] + cx * cx + cy * cy)
    for _ in range(10):
        dist = np.hypot(q[:, 0] - cx, q[:, 1] - cy)
        J = np.column_stack([-(q[:, 0] - cx) / dist, -(q[:, 1] - cy) / dist, -np.ones(len(q))])
        d = np.linalg.lstsq(J, -(dist - r), rcond=None)[0]
        cx, cy, r = cx + d[0], cy + d[1], r + d[2]
    return cx + m[0], cy + m[1], r


def exact(case, seed):
    doms = _domains(case, seed)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    nodes = sum(d["nx"] * d["ny"] for d in doms)
    if nodes * case["steps"] > 1.2e10:  # some tens of seconds
        return None
    m = _Plain(case, doms, dev)
    m.start(torch.cat([_plain_phi(case, d, dev) for d in doms]))
    if case["kind"] == "ramp":  # the start has the first gradient, the steps the next
        m.gh = torch.where(m.gh == doms[0]["h"], _ramp_h(doms[0], 1), m.gh)
    for _ in range(case["steps"]):
        m.step()
    rho, phi, ux, uy = m.fields()
    shape = (-1,) if case["kind"] == "batch" else (doms[0]["ny"], doms[0]["nx"])
    out = {n: v.reshape(shape) for n, v in zip(("rho", "phi", "ux", "uy"), (rho, phi, ux, uy))}
    out.update(mass=float(rho.sum()), max_u=float(torch.hypot(ux, uy).max()), nonfinite=0)
    if case.get("angle") or case.get("front"):
        fluid = np.ones(shape, bool) if m.fluid is None else m.fluid.reshape(shape).cpu().numpy()
        p = _crossings(out["phi"].cpu().numpy(), fluid)
    if case.get("angle"):
        cx, cy, r = _circle(p[p[:, 1] >= 1.5])
        out["theta"] = 90.0 + math.degrees(math.asin(max(-1.0, min(1.0, (cy + 0.5) / r))))
        out["R"] = r
    if case.get("front"):
        y0 = (case["ny"] - case["ch_w"]) // 2
        wb, wt = y0 - 0.5, y0 + case["ch_w"] - 0.5
        p = p[(p[:, 0] >= case["res_len"]) & (p[:, 0] <= case["nx"] - 1) & (p[:, 1] >= max(y0, wb + 2)) &
              (p[:, 1] <= min(y0 + case["ch_w"] - 1, wt - 2))]
        cx, cy, r = _circle(p)
        sg = 1.0 if cx > p[:, 0].mean() else -1.0
        tb, tt = (math.acos(max(-1.0, min(1.0, sg * v / r))) for v in (cy - wb, wt - cy))
        ym = 0.5 * (wb + wt)
        out["front"] = cx - sg * math.sqrt(max(r * r - (ym - cy) ** 2, 0.0))
        out["theta"], out["R"] = math.degrees(0.5 * (tb + tt)), r
    return out
