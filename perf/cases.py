"""The work a user of the framework has it do, as measurable cases.

A case is a dict of plain values. Kinds:
  solve    steps of one solver context between two looks at it: `steps` time steps, then the state
           snapshot on the device, the probe records of those steps, the time and the next dt (what
           the long-run drivers do between two stop times). A snapshot of the FP64 form is kept in
           double, one of the single-precision forms (FP32 and MIXED) in float, as written to a file.
  batch    an ensemble of independent members advanced together, then every member's snapshot
  coarse   a coarse FP64 solve with the learned correction added every `steps` steps
  predict  the learned correction of a state that the program holds on the device
  train    one optimiser step of the correction network and its updated weights (lr 1e-5: the tail
           of the cosine schedule the training uses)
Sizes and options are those of the workloads in inputs.py, of the tests and of bench.py.

exact() is the same method in plain 64-bit torch, from the same inputs.
"""
import math
import random

import numpy as np
import torch

from paper_2501_15923_gb300 import icarus as ic
from paper_2501_15923_gb300 import inputs as I

PRECISION = {"f64": ic.ICARUS_FP64, "f32": ic.ICARUS_FP32, "mixed": ic.ICARUS_MIXED}
STEP_CELLS = {"f64": 8_400_000, "f32": 42_000_000, "mixed": 42_000_000}   # cell updates of one pass


def _solve(name, flow, n1, n2, n3, precision, limiter=I.LIM_VANLEER, flux=I.FLUX_TVDLF, divb=I.DIVB_LINDE):
    steps = max(1, min(20, STEP_CELLS[precision] // (n1 * n2 * n3)))
    return {"name": name, "kind": "solve", "flow": flow, "n1": n1, "n2": n2, "n3": n3, "precision": precision,
            "limiter": limiter, "flux": flux, "divb": divb, "steps": steps}


def listed():
    return [
        # the smallest run: the static-sheet grid of the smoke test, launch and latency bound
        _solve("f64_static_60x16x32", "static", 60, 16, 32, "f64"),
        # odd and ragged sizes with the other limiter, flux and div-B source
        _solve("f64_ragged_129x17x33", "dynamic", 129, 17, 33, "f64", I.LIM_MC, I.FLUX_HLL, I.DIVB_POWELL),
        # the headline workload in its three precision forms
        _solve("f64_512x64x128", "dynamic", 512, 64, 128, "f64"),
        _solve("mixed_512x64x128", "dynamic", 512, 64, 128, "mixed"),
        _solve("f32_512x64x128", "dynamic", 512, 64, 128, "f32"),
        # an odd grid of ordinary size in single precision
        _solve("f32_ragged_300x33x65", "dynamic", 300, 33, 65, "f32"),
        # the 2019 case: uniform 600 x 64 x 192 grid, two-hour maps (the largest run)
        _solve("mixed_2019_600x64x192", "paper2019", 600, 64, 192, "mixed"),
        # the 2015 case at half its resolution: spherical-cloud CMEs and the CME tracer
        _solve("mixed_2015_300x32x96", "paper2015", 300, 32, 96, "mixed"),
        # a CME ensemble on uneven grids, each member with its own dt
        {"name": "batch_mixed_8", "kind": "batch", "grids": 3, "members": 8, "precision": "mixed", "steps": 4},
        # the coarse solve with the learned correction every ten steps
        {"name": "coarse_256x32x64", "kind": "coarse", "n1": 256, "n2": 32, "n3": 64, "steps": 10},
        # the correction network alone, and one step of its training
        {"name": "predict_256x32x64", "kind": "predict", "n1": 256, "n2": 32, "n3": 64},
        {"name": "train_256x32x64", "kind": "train", "n1": 256, "n2": 32, "n3": 64},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve"] * 6 + ["batch", "coarse", "predict", "train"])
    if kind == "solve":
        flow = rng.choice(["static", "dynamic", "dynamic", "dynamic", "paper2019", "paper2015"])
        c = _solve("", flow, size(40, 600), size(10, 64), size(16, 192), rng.choice(["f64", "f32", "mixed"]),
                   rng.choice([I.LIM_VANLEER] * 3 + [I.LIM_MINMOD, I.LIM_MC]),
                   rng.choice([I.FLUX_TVDLF] * 3 + [I.FLUX_HLL]), rng.choice([I.DIVB_LINDE] * 4 + [I.DIVB_POWELL]))
        del c["name"]
        return c
    if kind == "batch":
        return {"kind": "batch", "grids": rng.randint(4, 10000), "members": rng.randint(2, 6),
                "precision": rng.choice(["f32", "mixed"]), "steps": rng.randint(1, 4)}
    c = {"kind": kind, "n1": size(40, 256), "n2": size(10, 32), "n3": size(16, 64)}
    if kind == "coarse":
        c["steps"] = rng.randint(5, 10)
    return c


# ---- inputs -----------------------------------------------------------------------------------
T0 = I.AU / 1.0e5                                     # code units: 1 AU, 100 km/s, 1 proton per cm^3
RHO0 = I.M_P * 1e6
P0 = RHO0 * 1e10
B0 = math.sqrt(I.MU0 * RHO0) * 1e5


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _workload(case, seed):
    """The drivers of a solve and the time (code units) its pass begins at."""
    g = (case["n1"], case["n2"], case["n3"])
    flow = case.get("flow", "dynamic")
    if flow == "static":
        w, t = I.static_sheet(seed, grid=I.Grid(*g)), 0.0
    elif flow == "dynamic":
        w = I.dynamic_cme(seed, grid=I.Grid(*g), days=4.0)
        t = w.cmes[0, 0] + 3600.0                     # one hour into the CME insertion
    elif flow == "paper2019":
        w = I.paper2019(seed, days=2.0, n_maps=25, grid=I.Grid(*g, stretch=0))
        t = 10.5 * 3600.0
    else:
        w = I.paper2015(seed, days=10.0, grid=I.Grid(*g, stretch=0))
        t = w.cmes[0, 0] + 3600.0
    for k in ("limiter", "flux", "divb"):
        if k in case:
            setattr(w.opts, k, case[k])
    return w, t / T0


def _wave(rnd, r, th, ph):
    """A smooth field with values in [-1, 1]: four random harmonics."""
    s = 0.0
    for _ in range(4):
        a, b, m, p = rnd.uniform(1.0, 8.0), rnd.uniform(1.0, 6.0), rnd.randint(1, 6), rnd.uniform(0.0, 2 * math.pi)
        s = s + 0.25 * torch.cos(a * torch.log(r) + b * th + m * ph + p)
    return s


def _state(w, t, seed):
    """A developed solar wind [8][n3][n2][n1] (code units, double): the boundary map of time t wound
    into a spiral and expanded outwards, with waves in every field."""
    g, dev, rnd = w.grid, _device(), random.Random(seed)
    edges = torch.arange(g.n1 + 1, dtype=torch.float64, device=dev) / g.n1
    edges = g.x1min * (g.x1max / g.x1min) ** edges if g.stretch else g.x1min + (g.x1max - g.x1min) * edges
    r = 0.5 * (edges[1:] + edges[:-1])
    th = torch.from_numpy(g.theta_centres()).to(dev).view(1, -1, 1)
    ph = torch.from_numpy(g.phi_centres()).to(dev).view(-1, 1, 1)
    tm, ts = w.t_maps, t * T0
    m = int(np.clip(np.searchsorted(tm, ts, side="right") - 1, 0, len(tm) - 1))
    n = min(m + 1, len(tm) - 1)
    f = 0.0 if n == m else (ts - tm[m]) / (tm[n] - tm[m])
    maps = torch.from_numpy((1.0 - f) * w.maps[m] + f * w.maps[n]).to(dev)          # [5][n2][n3]
    turn = w.omega * (r - g.x1min) * I.AU / 4.5e5 / (2 * math.pi / g.n3)            # in cells of longitude
    pos = torch.arange(g.n3, dtype=torch.float64, device=dev).view(-1, 1) + turn    # [n3][n1]
    lo = torch.floor(pos)
    a = (pos - lo).unsqueeze(1)
    lo = lo.long() % g.n3
    q = [((1.0 - a) * mm[:, lo].permute(1, 0, 2) + a * mm[:, (lo + 1) % g.n3].permute(1, 0, 2)) for mm in maps]
    r = r.view(1, 1, -1)
    x = g.x1min / r
    wave = lambda amp: amp * _wave(rnd, r, th, ph)  # noqa: E731
    om = w.omega * T0
    v = q[0] / 1e5
    rho = q[1] / 1e6 * x ** 2 * (1.0 + wave(0.1))
    p = q[2] / P0 * x ** (2.0 * w.gamma) * (1.0 + wave(0.1))
    br = q[3] / B0 * x ** 2 * (1.0 + wave(0.02))
    vel = [v * (1.0 + wave(0.05)), v * wave(0.03), -om * r * torch.sin(th) + v * wave(0.03)]
    b = [br, br * wave(0.05), -br * om * r * torch.sin(th) / v * (1.0 + wave(0.05))]
    e = p / (w.gamma - 1.0) + 0.5 * rho * sum(z * z for z in vel) + 0.5 * sum(z * z for z in b)
    return torch.stack([rho] + [rho * z for z in vel] + [e] + b).contiguous()


def _members(case, seed):
    """Drivers and start times of the members, on the uneven grids of the ensemble workload."""
    grids = [w.grid for w in I.ensemble(case["grids"], case["members"], days=1.0)]
    ws = [I.dynamic_cme(seed + 7 * m, grid=g, days=4.0) for m, g in enumerate(grids)]
    return ws, [(w.cmes[0, 0] + 3600.0) / T0 for w in ws]


WIDTHS = ((8, 32), (32, 32), (32, 32), (32, 8))       # channels in and out of the four layers


def _weights(seed):
    """Random weights of the network [out][27][in] and its biases (the padded channels are zero)."""
    rng = np.random.default_rng(seed)
    out = []
    for (ci, co), (pi, po) in zip(WIDTHS, ic.LAYER_SHAPES):
        w, b = np.zeros((po, 27, pi), np.float32), np.zeros(po, np.float32)
        w[:co, :, :ci] = rng.standard_normal((co, 27, ci)) * math.sqrt((2.0 if co == 32 else 0.2) / (27 * ci))
        b[:co] = 0.02 * rng.standard_normal(co)
        out.append((w, b))
    return out


def _network_inputs(case, seed):
    """A coarse state, the correction it should get, weights and normalisation."""
    w, t = _workload(dict(case, flow="dynamic"), seed)
    U = _state(w, t, seed)
    rnd = random.Random(seed + 1)
    ax = [torch.linspace(0.3, 2.0, n, dtype=torch.float64, device=U.device) for n in (case["n1"], case["n2"], case["n3"])]
    dU = torch.stack([1e-5 * u.abs().mean((0, 1)) * _wave(rnd, ax[0].view(1, 1, -1), 3 * ax[1].view(1, -1, 1), 3 * ax[2].view(-1, 1, 1))
                      for u in U]).contiguous()
    mean = U.mean((1, 2))
    scale = (U - mean[:, None, None, :]).square().mean((1, 2)).sqrt()
    oscale = dU.square().mean((1, 2)).sqrt()
    low = lambda a: torch.maximum(a, 1e-12 * a.max()).cpu().numpy()  # noqa: E731
    return w, t, U, dU, _weights(seed), (mean.cpu().numpy(), low(scale), low(oscale))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        w, t = _workload(case, seed)
        s = ic.from_workload(w, precision=PRECISION[case["precision"]])
        U = _state(w, t, seed)
        s.set_state(U.cpu().numpy(), t)
        s.sample(w.traj, cap=1)                       # registers the probes
        return {"kind": kind, "solver": s, "out": U, "steps": case["steps"], "tracer": bool(w.opts.tracer),
                "single": case["precision"] != "f64"}
    if kind == "batch":
        ws, ts = _members(case, seed)
        b = ic.Batch(ws, precision=PRECISION[case["precision"]])
        outs = [_state(w, t, seed + m) for m, (w, t) in enumerate(zip(ws, ts))]
        for m, (U, t) in enumerate(zip(outs, ts)):
            b.set_state(m, U.cpu().numpy(), t)
        return {"kind": kind, "batch": b, "out": outs, "steps": case["steps"]}
    s = ic.from_workload(_workload(dict(case, flow="dynamic"), seed)[0]) if kind == "coarse" else None
    w, t, U, dU, weights, norm = _network_inputs(case, seed)
    net = ic.Closure(case["n1"], case["n2"], case["n3"], seed=seed)
    net.set_weights(weights)
    net.set_norm(*norm)
    if kind == "coarse":
        s.set_state(U.cpu().numpy(), t)
        s.sample(w.traj, cap=1)
        return {"kind": kind, "solver": s, "net": net, "out": U, "steps": case["steps"]}
    return {"kind": kind, "net": net, "U": U, "dU": dU, "out": torch.empty_like(U)}


def run(state):
    kind = state["kind"]
    if kind in ("solve", "coarse"):
        s, n, U = state["solver"], state["steps"], state["out"]
        s.step(n)
        if kind == "coarse":
            state["net"].apply(s.ctx)
        ic.icarus_copy_state(s.ctx, U.data_ptr())
        rec, _ = s.sample(None, cap=n)
        t, dt = s.time()
        got = {"U": U.float() if state.get("single") else U, "probes": rec, "t": t, "dt": dt}
        if state.get("tracer"):
            got["tracer"] = s.get_tracer().astype(np.float32)
        return got
    if kind == "batch":
        b = state["batch"]
        b.step(state["steps"])
        for c, U in zip(b.ctx, state["out"]):
            ic.icarus_copy_state(c, U.data_ptr())
        return [U.float() for U in state["out"]]
    if kind == "predict":
        state["net"].predict(state["U"].data_ptr(), state["out"].data_ptr())
        return state["out"].float()
    loss = state["net"].train_step(state["U"].data_ptr(), state["dU"].data_ptr(), 1e-5)
    return {"loss": np.float32(loss), "weights": state["net"].weights()}


def _sizes(case):
    """(cells, state bytes per value) of each solve of a pass."""
    if case["kind"] == "batch":
        return [(w.grid.ncell, 8 if case["precision"] == "mixed" else 4) for w in _members(case, 0)[0]]
    return [(case["n1"] * case["n2"] * case["n3"], 4 if case.get("precision") == "f32" else 8)]


def work(case):
    """Solves: each step reads and writes the state once, the snapshot is written once; about 190
    operations a face (three a cell) and 130 a cell in each of two stages. The network: the state in,
    the correction out (training: the target in); 2 x 27 products a voxel and pair of channels."""
    steps = case.get("steps", 0)
    nbytes = sum(n * 8 * (2 * size * steps + 8) for n, size in _sizes(case))
    flops = sum(n * steps * 2.0 * (3 * 190 + 130) for n, _ in _sizes(case))
    if case["kind"] in ("coarse", "predict", "train"):
        n = case["n1"] * case["n2"] * case["n3"]
        flops += n * 54.0 * sum(a * b for a, b in WIDTHS) * (3 if case["kind"] == "train" else 1)
        nbytes += 0 if case["kind"] == "coarse" else n * 8 * 8
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- the same in plain 64-bit torch -------------------------------------------------------------
class _Exact:
    """Ideal MHD on the spherical grid: limited linear reconstruction, TVDLF / HLL, SSP-RK2, Linde
    diffusion or the Powell source, driven inner boundary, probes."""

    def __init__(self, w):
        g, self.w, self.o, self.gam = w.grid, w, w.opts, w.gamma
        self.n = (g.n1, g.n2, g.n3)
        self.om, self.gm = w.omega * T0, I.GM_SUN / (I.AU * 1e10)
        dev = self.dev = _device()
        i1, i2, i3 = (np.arange(-2, n + 3, dtype=np.float64) for n in self.n)
        e1 = g.x1min * (g.x1max / g.x1min) ** (i1 / g.n1) if g.stretch else g.x1min + i1 * ((g.x1max - g.x1min) / g.n1)
        self.d2, self.d3 = (g.x2max - g.x2min) / g.n2, (g.x3max - g.x3min) / g.n3
        e2, e3 = g.x2min + i2 * self.d2, g.x3min + i3 * self.d3
        self.rc, self.tc, self.pc = (0.5 * (e[1:] + e[:-1]) for e in (e1, e2, e3))
        R = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev).view(1, 1, -1)  # noqa: E731
        T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev).view(1, -1, 1)  # noqa: E731
        v1, v2 = (e1[1:] ** 3 - e1[:-1] ** 3) / 3.0, np.cos(e2[:-1]) - np.cos(e2[1:])
        q1 = 0.5 * (e1[1:] ** 2 - e1[:-1] ** 2) / v1
        # padded: -2 .. n + 1 (cells), -2 .. n + 2 (faces)
        self.a1, self.iv1, self.q1, self.dr, self.r = R(e1 ** 2), R(1.0 / v1), R(q1), R(np.diff(e1)), R(self.rc)
        self.a2, self.iv2, self.q2 = T(np.sin(e2)), T(1.0 / v2), T(self.d2 / v2)
        self.sn, self.cs = T(np.sin(self.tc)), T(np.cos(self.tc))
        self.tmaps = w.t_maps / T0
        unit = np.array([1e5, 1e6, P0, B0, B0]).reshape(1, 5, 1, 1)
        self.maps = torch.from_numpy(w.maps / unit).to(dev).permute(0, 1, 3, 2)      # [m][5][n3][n2]
        th, ph = self.tc[2:-2][None, :], self.pc[2:-2][:, None]
        self.dirs = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th) + 0 * ph])

    def prims(self, U):
        rho = U[0]
        v = U[1:4] / rho
        p = (self.gam - 1.0) * (U[4] - 0.5 * (U[1:4] * v).sum(0) - 0.5 * U[5:8].square().sum(0))
        return torch.cat([rho[None], v, p[None], U[5:8]])

    def inner(self, tau):
        """(rho, v_r, p, B_r, B_phi) [n3][n2] of the driven face at time tau."""
        tm = self.tmaps
        m = int(np.clip(np.searchsorted(tm, tau, side="right") - 1, 0, len(tm) - 1))
        n = min(m + 1, len(tm) - 1)
        f = 0.0 if n == m else min(max((tau - tm[m]) / (tm[n] - tm[m]), 0.0), 1.0)
        v, rho, p, br, bp = ((1.0 - f) * self.maps[m] + f * self.maps[n]).clone()
        for on, dur, lat, lon, hw, speed, dens, temp in self.w.cmes:
            on, dur, vel = on / T0, dur / T0, speed / 1e5
            ax = np.array([math.cos(lat) * math.cos(lon), math.cos(lat) * math.sin(lon), math.sin(lat)])
            thr = math.cos(hw)
            if self.o.cme_model == I.CME_SPHERE:
                r0 = self.w.grid.x1min
                rad = r0 * math.sin(hw)
                dur = 2.0 * rad / vel
                d = r0 - rad + vel * (tau - on)
                thr = (r0 * r0 + d * d - rad * rad) / (2.0 * r0 * d)
            if on <= tau < on + dur:
                hit = torch.from_numpy((self.dirs * ax[:, None, None]).sum(0) >= thr).to(self.dev)
                for q, x in ((rho, dens / 1e6), (v, vel), (p, 2.0 * dens * I.K_B * temp / P0)):
                    q[hit] = x
        return rho, v, p, br, bp

    def padded(self, W, tau):
        n1, n2, n3 = self.n
        P = torch.empty((8, n3 + 4, n2 + 4, n1 + 4), dtype=torch.float64, device=self.dev)
        P[:, 2:-2, 2:-2, 2:-2] = W
        rho, v, p, br, bp = self.inner(tau)
        for gh in (1, 2):
            mir = W[..., gh - 1]
            P[:, 2:-2, 2:-2, 2 - gh] = torch.stack([rho, v, -mir[2], -mir[3], p, br, -mir[6], bp])
            P[:, 2:-2, 2:-2, n1 + 1 + gh] = W[..., -1]
            P[5, 2:-2, 2:-2, n1 + 1 + gh] *= (self.rc[n1 + 1] / self.rc[n1 + 1 + gh]) ** 2
        P[:, 2:-2, :2] = P[:, 2:-2, 2:3]
        P[:, 2:-2, -2:] = P[:, 2:-2, -3:-2]
        for gh in (0, 1):                                                         # periodic in longitude
            P[:, gh] = P[:, 2 + (gh - 2) % n3]
            P[:, n3 + 2 + gh] = P[:, 2 + gh % n3]
        return P

    def slope(self, a, b):
        same, s = a * b > 0, a + b
        if self.o.limiter == I.LIM_VANLEER:
            return torch.where(same, 2.0 * a * b / torch.where(same, s, torch.ones_like(s)), 0.0)
        if self.o.limiter == I.LIM_MINMOD:
            m = torch.where(a.abs() < b.abs(), a, b)
        else:
            m = torch.sign(a) * torch.minimum(2.0 * torch.minimum(a.abs(), b.abs()), 0.5 * s.abs())
        return torch.where(same, m, 0.0)

    def side(self, w, d):
        """Conserved state, flux and fast speed along d of primitives w."""
        rho, v, p, b = w[0], w[1:4], w[4], w[5:8]
        bb, bv, vn, bn = b.square().sum(0), (b * v).sum(0), v[d], b[d]
        m, pt = rho * v, p + 0.5 * bb
        e = p / (self.gam - 1.0) + 0.5 * rho * v.square().sum(0) + 0.5 * bb
        fm, fb = m * vn - b * bn, vn * b - bn * v
        fm[d] += pt
        fb[d] = 0.0
        a2 = self.gam * p / rho
        s = a2 + bb / rho
        cf = torch.sqrt(0.5 * (s + torch.sqrt(torch.clamp(s * s - 4.0 * a2 * bn * bn / rho, min=0.0))))
        return torch.cat([rho[None], m, e[None], b]), torch.cat([(rho * vn)[None], fm, ((e + pt) * vn - bn * bv)[None], fb]), cf

    def flux(self, P, d):
        """Fluxes through the n + 1 faces along d (0: r, 1: theta, 2: phi)."""
        n, ax = self.n[d], 3 - d
        A = P[(slice(None),) + tuple(slice(None) if 2 - k == d else slice(2, -2) for k in range(3))]
        c, lo, hi = A.narrow(ax, 1, n + 2), A.narrow(ax, 0, n + 2), A.narrow(ax, 2, n + 2)
        h = 0.5 * self.slope(c - lo, hi - c)
        wl, wr = (c + h).narrow(ax, 0, n + 1), (c - h).narrow(ax, 1, n + 1)
        first = (wl[0] <= 0) | (wr[0] <= 0) | (wl[4] <= 0) | (wr[4] <= 0)
        wl, wr = torch.where(first, c.narrow(ax, 0, n + 1), wl), torch.where(first, c.narrow(ax, 1, n + 1), wr)
        (ul, fl, cl), (ur, fr, cr) = self.side(wl, d), self.side(wr, d)
        if self.o.flux == I.FLUX_TVDLF:
            c = torch.maximum(wl[1 + d].abs() + cl, wr[1 + d].abs() + cr)
            return 0.5 * (fl + fr) - 0.5 * c * (ur - ul)
        sl, sr = torch.minimum(wl[1 + d] - cl, wr[1 + d] - cr), torch.maximum(wl[1 + d] + cl, wr[1 + d] + cr)
        mid = (sr * fl - sl * fr + sl * sr * (ur - ul)) / torch.where(sr > sl, sr - sl, torch.ones_like(sr))
        return torch.where(sl >= 0, fl, torch.where(sr <= 0, fr, mid))

    def stage(self, U, P, dt):
        """U + dt L(P), with the Linde increment."""
        n1, n2, n3 = self.n
        x, y = slice(2, -2), slice(2, -2)
        W = P[:, 2:-2, 2:-2, 2:-2]
        a1m, a1p, iv1, q1 = self.a1[..., 2:-3], self.a1[..., 3:-2], self.iv1[..., x], self.q1[..., x]
        a2m, a2p, iv2, q2 = self.a2[:, 2:-3], self.a2[:, 3:-2], self.iv2[:, y], self.q2[:, y]
        f = self.flux(P, 0)
        L = -(a1p * f[..., 1:] - a1m * f[..., :-1]) * iv1
        f = self.flux(P, 1)
        L -= (a2p * f[:, :, 1:] - a2m * f[:, :, :-1]) * iv2 * q1
        f = self.flux(P, 2)
        L -= (f[:, 1:] - f[:, :-1]) * q1 * q2 / self.d3
        del f
        rho, vr, vt, vp, p, br, bt, bp = W
        r, sn, cs = self.r[..., x], self.sn[:, y], self.cs[:, y]
        ir, cot, pt = 1.0 / r, cs / sn, p + 0.5 * (br * br + bt * bt + bp * bp)
        L[1] += pt * (a1p - a1m) * iv1 + (rho * (vt * vt + vp * vp) - (bt * bt + bp * bp)) * ir
        L[2] += pt * q1 * (a2p - a2m) * iv2 + (-(rho * vr * vt - br * bt) + cot * (rho * vp * vp - bp * bp)) * ir
        L[3] -= ((rho * vp * vr - bp * br) + cot * (rho * vp * vt - bp * bt)) * ir
        L[6] += (vr * bt - vt * br) * ir
        L[7] += ((vr * bp - vp * br) + cot * (vt * bp - vp * bt)) * ir
        cen, vpar, om = rho * self.om ** 2 * r * sn, vr * sn + vt * cs, self.om
        L[1] += cen * sn + 2.0 * rho * om * vp * sn
        L[2] += cen * cs + 2.0 * rho * om * vp * cs
        L[3] -= 2.0 * rho * om * vpar
        L[4] += cen * vpar
        if self.o.gravity:
            gr = self.gm / r ** 2
            L[1] -= rho * gr
            L[4] -= rho * vr * gr
        # div B of the cells -1 .. n
        b1, b2, b3 = P[5, 1:-1, 1:-1], P[6, 1:-1, :, 1:-1], P[7, :, 1:-1, 1:-1]
        f1, f2 = 0.5 * (b1[..., 1:] + b1[..., :-1]), 0.5 * (b2[:, 1:] + b2[:, :-1])
        D = (self.a1[..., 2:-1] * f1[..., 1:] - self.a1[..., 1:-2] * f1[..., :-1]) * self.iv1[..., 1:-1]
        D += (self.a2[:, 2:-1] * f2[:, 1:] - self.a2[:, 1:-2] * f2[:, :-1]) * self.iv2[:, 1:-1] * self.q1[..., 1:-1]
        D += 0.5 * (b3[2:] - b3[:-2]) * self.q1[..., 1:-1] * self.q2[:, 1:-1] / self.d3
        if self.o.divb == I.DIVB_POWELL:
            dc = D[1:-1, 1:-1, 1:-1]
            L[1:4] -= dc * W[5:8]
            L[4] -= dc * (vr * br + vt * bt + vp * bp)
            L[5:8] -= dc * W[1:4]
        out = U + dt * L
        if self.o.divb == I.DIVB_LINDE and dt > 0:
            coef = self.o.divb_coef / (self.dr[..., x] ** -2 + (r * self.d2) ** -2 + (r * sn * self.d3) ** -2)
            g1 = (D[1:-1, 1:-1, 2:] - D[1:-1, 1:-1, :-2]) / (self.r[..., 3:-1] - self.r[..., 1:-3])
            g2 = (D[1:-1, 2:, 1:-1] - D[1:-1, :-2, 1:-1]) / (2.0 * self.d2) * ir
            g3 = (D[2:, 1:-1, 1:-1] - D[:-2, 1:-1, 1:-1]) / (2.0 * self.d3) * ir / sn
            lb = coef * torch.stack([g1, g2, g3])
            out[4] += (W[5:8] * lb).sum(0)
            out[5:8] += lb
        return out

    def floors(self, U):
        U[0].clamp_(min=self.o.rho_floor)
        W = self.prims(U)
        low = W[4] < self.o.p_floor
        if bool(low.any()):
            e = self.o.p_floor / (self.gam - 1.0) + 0.5 * U[1:4].square().sum(0) / U[0] + 0.5 * U[5:8].square().sum(0)
            U[4] = torch.where(low, e, U[4])
            W[4].clamp_(min=self.o.p_floor)
        return W

    def cfl_dt(self, W):
        x, y = slice(2, -2), slice(2, -2)
        width = (self.dr[..., x], self.r[..., x] * self.d2, self.r[..., x] * self.sn[:, y] * self.d3)
        return self.o.cfl / float(sum((W[1 + d].abs() + self.side(W, d)[2]) / width[d] for d in range(3)).max())

    def probes(self, W, t):
        """Records of every probe at time t."""
        (n1, n2, n3), out, ts = self.n, [], t * T0
        rc, tc, pc = self.rc[2:-2], self.tc[2:-2], self.pc[2:-2]
        for kn in self.w.traj:
            rm, lat, lon = (float(np.interp(ts, kn[:, 0], kn[:, q])) for q in (1, 2, 3))
            r, th, ph = rm / I.AU, math.pi / 2 - lat, (lon - self.w.omega * ts) % (2 * math.pi)
            i = int(np.clip(np.searchsorted(rc, r, side="right") - 1, 0, n1 - 2))
            j = int(np.clip(np.searchsorted(tc, th, side="right") - 1, 0, n2 - 2))
            k = int(np.searchsorted(pc, ph, side="right")) - 1
            wr, wt = (r - rc[i]) / (rc[i + 1] - rc[i]), (th - tc[j]) / (tc[j + 1] - tc[j])
            wp = (ph - (pc[k] if k >= 0 else pc[-1] - 2 * math.pi)) / self.d3
            k = k % n3
            wr, wt, wp = (min(max(z, 0.0), 1.0) for z in (wr, wt, wp))
            box = W[:, [k, (k + 1) % n3]][:, :, j:j + 2, i:i + 2].cpu().numpy()
            a = np.einsum("vkji,k,j,i->v", box, [1 - wp, wp], [1 - wt, wt], [1 - wr, wr])
            b = a[5:8] * B0
            out.append([ts, a[0] * 1e6, a[1] * 1e5, a[2] * 1e5, (a[3] + self.om * r * math.sin(th)) * 1e5, *b, a[4] * P0,
                        math.sqrt((b * b).sum()), i, j, k])
        return np.array(out)

    def steps(self, U, t, n):
        """n steps from U at time t: (U, probe records, t, next dt)."""
        W, rec = self.prims(U), []
        dt = self.cfl_dt(W)
        for _ in range(n):
            U1 = self.stage(U, self.padded(W, t), dt)
            W1 = self.floors(U1)
            U = 0.5 * U + 0.5 * self.stage(U1, self.padded(W1, t + dt), dt)
            W = self.floors(U)
            t, dt = t + dt, self.cfl_dt(W)
            rec.append(self.probes(W, t))
        return U, np.stack(rec), t, dt


def _network(x, wb):
    """The four layers on x [n3][n2][n1][8] (circular in longitude, replicated in r and colatitude)."""
    for l, (w, b) in enumerate(wb):
        p = torch.cat([x[-1:], x, x[:1]])
        p = torch.cat([p[:, :1], p, p[:, -1:]], 1)
        p = torch.cat([p[:, :, :1], p, p[:, :, -1:]], 2)
        n3, n2, n1 = x.shape[:3]
        y = b
        for t in range(27):
            d1, d2, d3 = t % 3, (t // 3) % 3, t // 9
            y = y + p[d3:d3 + n3, d2:d2 + n2, d1:d1 + n1] @ w[:, t].T
        x = torch.relu(y) if l < 3 else y
    return x


def _wb64(weights, dev):
    return [[torch.from_numpy(w[:co, :, :ci].astype(np.float64)).to(dev), torch.from_numpy(b[:co].astype(np.float64)).to(dev)]
            for (w, b), (ci, co) in zip(weights, WIDTHS)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        w, t = _workload(case, seed)
        U, rec, t, dt = _Exact(w).steps(_state(w, t, seed), t, case["steps"])
        got = {"U": U, "probes": rec, "t": t, "dt": dt}
        if w.opts.tracer:
            got["tracer"] = None
        return got
    if kind == "batch":
        ws, ts = _members(case, seed)
        return [_Exact(w).steps(_state(w, t, seed + m), t, case["steps"])[0] for m, (w, t) in enumerate(zip(ws, ts))]
    w, t, U, dU, weights, norm = _network_inputs(case, seed)
    mean, scale, oscale = (torch.from_numpy(a).to(U.device)[:, None, None, :] for a in norm)
    wb = _wb64(weights, U.device)
    if kind == "coarse":
        U, rec, t, _ = _Exact(w).steps(U, t, case["steps"])
    x = ((U - mean) / scale).permute(1, 2, 3, 0)
    if kind == "coarse":
        U = U + _network(x, wb).permute(3, 0, 1, 2) * oscale
        m = _Exact(w)
        return {"U": U, "probes": rec, "t": t, "dt": m.cfl_dt(m.prims(U))}
    if kind == "predict":
        return _network(x, wb).permute(3, 0, 1, 2) * oscale
    flat = [v.requires_grad_() for layer in wb for v in layer]
    loss = (_network(x, wb) - (dU / oscale).permute(1, 2, 3, 0)).square().mean()
    grads = torch.autograd.grad(loss, flat)
    out = [(w.astype(np.float64), b.astype(np.float64)) for w, b in weights]
    for q, gr in enumerate(grads):                    # the first Adam step: m / c1 = g, v / c2 = g^2
        gr = gr.cpu().numpy()
        new, (ci, co) = out[q // 2][q % 2], WIDTHS[q // 2]
        part = new[:co, :, :ci] if q % 2 == 0 else new[:co]
        part -= 1e-5 * gr / (np.abs(gr) + 1e-8)
    return {"loss": float(loss.detach()), "weights": out}
