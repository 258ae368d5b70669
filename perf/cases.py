"""The work that users have this framework do, as cases that can be timed and compared.

Each case is a dict of plain values.  The kinds:

``solve1d``      steps of a batch of independent 1D GPE instances (hfs.Solver.step)
``diag1d``       norm and energy of such a batch (hfs.Solver.norm, .energy)
``solve3d``      steps of one 3D GPE instance
``fno_forward``  inference of the learned surrogate (fno.Fno.forward)
``fno_train``    one optimizer step of the surrogate (fno.Fno.train_step)

A solver pass continues in time from where the pass before it ended, as a
simulation does between two of its outputs; the state stays on the device.
``exact`` integrates the same composition unmerged, sub-flow by sub-flow, in
64 bits with torch's own transforms.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1007_3470_gb300 import hfs
from paper_1007_3470_gb300 import workloads as W
from paper_1007_3470_gb300.fno import Fno, FnoConfig

FLOWS = {"lemma2": hfs.HFS_FLOW_LEMMA2, "cf4": hfs.HFS_FLOW_CF4, "m6": hfs.HFS_FLOW_M6}
SPLITS = {"ho": hfs.HFS_SPLIT_HO, "fourier": hfs.HFS_SPLIT_FOURIER}
LAWS = {"const": W.OMEGA_CONST, "sin": W.OMEGA_SIN, "cos_sq": W.OMEGA_COS_SQ}
KINDS = {"none": W.VI_NONE, "x4": W.VI_X4, "cos": W.VI_COS}
STAGES = {"strang": 1, "srkn6_4": 6, "ni4_82": 4, "ni5_84": 5}


def _solve1d(**kw):
    c = {"kind": "solve1d", "count": 1, "nmin": 256, "nmax": 256, "steps": 1, "h": 0.005, "scheme": "strang",
         "flow": "cf4", "split": "ho", "law": "sin", "vi": "cos", "off_centre": False, "precision": "c64",
         "streaming": False, "projection": False, "graphs": False, "reuse": False}
    c.update(kw)
    return c


def _fno(kind, batch, name=None, grid=256, width=64, modes=32, layers=4, proj=128):
    c = {"kind": kind, "batch": batch, "grid": grid, "width": width, "modes": modes, "layers": layers, "in_ch": 7,
         "proj": proj, "out_ch": 2}
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # one step of one instance: a program that looks at psi, or couples to it, after every step
        _solve1d(name="single_step_1024", nmin=1024, nmax=1024, steps=1),
        # the paper's coherent state in a quartic-perturbed trap: one small instance over a long time
        _solve1d(name="coherent_256", nmin=256, nmax=256, steps=1000, h=0.01, flow="lemma2", law="const", vi="x4"),
        # the time-dependent GPE with the five-stage composition in the FP64 parity mode: a reference solution
        _solve1d(name="gpe_1024_c128", nmin=1024, nmax=1024, steps=25, h=0.04, scheme="ni5_84", precision="c128"),
        # training targets of the surrogate: a chunk of 4096 trajectories of one grid size to T = 1
        _solve1d(name="family_256", count=4096, nmin=256, nmax=256, steps=200),
        # the headline batch: mixed grid sizes, 500 steps, replayed from a graph, next call's schedule prefetched
        _solve1d(name="batch_4096", count=4096, nmin=128, nmax=4096, steps=500, projection=True, graphs=True,
                 reuse=True),
        # a batch larger than L2 advanced one step per call (each call one pass over device memory)
        _solve1d(name="monitor_16384", count=16384, nmin=128, nmax=4096, steps=1, projection=True, streaming=True),
        # norm and energy of the headline batch, as a run logs them
        {"name": "diagnostics_4096", "kind": "diag1d", "count": 4096, "nmin": 128, "nmax": 4096, "precision": "c64"},
        # 3D: the mid-size grid
        {"name": "grid3d_64", "kind": "solve3d", "n": 64, "steps": 50, "h": 0.005, "scheme": "strang", "flow": "cf4",
         "precision": "c64", "projection": False, "graphs": True},
        # 3D: the headline grid, half a solve
        {"name": "grid3d_128", "kind": "solve3d", "n": 128, "steps": 100, "h": 0.005, "scheme": "strang",
         "flow": "cf4", "precision": "c64", "projection": True, "graphs": True},
        # the surrogate asked for one solution
        _fno("fno_forward", 1, "fno_forward_1"),
        # the surrogate over a large batch
        _fno("fno_forward", 4096, "fno_forward_4096"),
        # the surrogate's training batch
        _fno("fno_train", 256, "fno_train_256"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# grid-point-sub-stages of the largest listed 1D and 3D cases
_MOST_1D, _MOST_3D = 2.0e9, 2.0e8


def draw(rng):
    kind = rng.choice(["solve1d", "solve1d", "solve1d", "diag1d", "solve3d", "solve3d", "fno_forward", "fno_train"])
    if kind in ("solve1d", "diag1d"):
        i = rng.randrange(6)
        j = rng.choice([i, rng.randrange(i, 6)])
        nmin, nmax = 128 << i, 128 << j
        precision = rng.choice(["c64", "c64", "c64", "c128"])
        if kind == "diag1d":
            return {"kind": kind, "count": _log(rng, 1, 4096), "nmin": nmin, "nmax": nmax, "precision": precision}
        scheme = rng.choice(["strang", "strang", "strang", "srkn6_4", "ni4_82", "ni5_84"])
        streaming = rng.random() < 0.15
        # FP64 runs at a small fraction of the FP32 rate
        most = _MOST_1D / (40.0 if precision == "c128" else 1.0) / STAGES[scheme] / math.sqrt(nmin * nmax)
        count = _log(rng, 1, int(min(16384 if streaming else 4096, most)))
        steps = _log(rng, 1, int(max(1, min(20 if streaming else 500, most / count))))
        split = rng.choice(["ho", "ho", "ho", "fourier"])
        return _solve1d(count=count, nmin=nmin, nmax=nmax, steps=steps, scheme=scheme,
                        h=rng.choice([0.0025, 0.005, 0.01] if scheme == "strang" else [0.01, 0.02, 0.04]),
                        flow=rng.choice(["cf4", "cf4", "lemma2", "m6"]), split=split,
                        law=rng.choice(["sin", "sin", "const", "cos_sq"]), vi=rng.choice(["cos", "cos", "none", "x4"]),
                        off_centre=rng.random() < 0.15, precision=precision, streaming=streaming,
                        projection=precision == "c64" and rng.random() < 0.5, graphs=rng.random() < 0.4,
                        reuse=rng.random() < 0.3)
    if kind == "solve3d":
        n = rng.choice([32, 64, 128])
        precision = rng.choice(["c64", "c64", "c128"])
        scheme = rng.choice(["strang", "strang", "srkn6_4", "ni4_82"])
        most = _MOST_3D / (40.0 if precision == "c128" else 1.0) / STAGES[scheme] / n ** 3
        return {"kind": kind, "n": n, "steps": _log(rng, 1, int(max(1, min(200, most)))), "h": rng.choice([0.0025, 0.005]),
                "scheme": scheme, "flow": rng.choice(["cf4", "cf4", "lemma2", "m6"]), "precision": precision,
                "projection": n == 128 and precision == "c64" and rng.random() < 0.5, "graphs": rng.random() < 0.6}
    batch = _log(rng, 1, 4096 if kind == "fno_forward" else 512)
    return rng.choice([_fno(kind, batch), _fno(kind, batch),
                       _fno(kind, batch, grid=64, width=16, modes=8, layers=2, proj=32),
                       _fno(kind, batch, grid=64, width=64, modes=8, layers=2, proj=128)])


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _sizes(case):
    """Grid sizes of a batch: equally many of each, their order left to the seed."""
    sizes = np.asarray([n for n in (128, 256, 512, 1024, 2048, 4096) if case["nmin"] <= n <= case["nmax"]])
    return sizes[((np.arange(case["count"]) + 0.5) * len(sizes) / case["count"]).astype(int)]


def _batch(case, seed):
    """Parameters of a 1D batch, one array per parameter: the batched GPE family (half-width 8 + N/64)."""
    rng = np.random.default_rng(seed)
    count = case["count"]
    sizes = _sizes(case)
    p = {"n": rng.permutation(sizes), "w0": rng.uniform(0.5, 2.0, count),
         "sigma": rng.uniform(-1.0, 20.0, count), "eps": rng.uniform(0.0, 0.1, count),
         "k": rng.uniform(1.0, 4.0, count), "x0": rng.uniform(-1.0, 1.0, count),
         "shift": rng.uniform(-2.0, 2.0, count)}
    half = 8.0 + p["n"] / 64.0
    centre = p["shift"] if case.get("off_centre") else np.zeros(count)
    p["lo"], p["hi"] = centre - half, centre + half
    if case.get("vi", "cos") == "none":
        p["eps"] = np.zeros(count)
    p["groups"] = [(n, np.nonzero(p["n"] == n)[0]) for n in np.unique(sizes).tolist()]
    return p


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grid(p, n, idx):
    """x_j of every instance of one grid size, and its parameters as columns, FP64."""
    def col(v):
        return torch.from_numpy(np.ascontiguousarray(v[idx])).to(_device())[:, None]
    lo, hi = col(p["lo"]), col(p["hi"])
    x = lo + (hi - lo) / n * torch.arange(n, dtype=torch.float64, device=_device())
    return x, col, (hi - lo) / n


def _psi0(p):
    """Normalised Gaussians exp(-w0 (x - x0)^2 / 2) of every grid size: {n: (instances, complex128)}."""
    out = {}
    for n, idx in p["groups"]:
        x, col, dx = _grid(p, n, idx)
        g = torch.exp(-0.5 * col(p["w0"]) * (x - col(p["x0"])) ** 2)
        out[n] = (idx, (g / torch.sqrt(dx * (g * g).sum(1, keepdim=True))).to(torch.complex128))
    return out


def _flat(p, groups):
    """One vector, instance after instance, of the rows of every grid size."""
    off = np.concatenate([[0], np.cumsum(p["n"])])
    out = torch.empty(int(off[-1]), dtype=torch.complex128, device=_device())
    for n, (idx, v) in groups.items():
        at = torch.from_numpy(off[idx]).to(_device())[:, None] + torch.arange(n, device=_device())
        out[at] = v
    return out


def _instances(case, p):
    law, vi = LAWS[case.get("law", "sin")], KINDS[case.get("vi", "cos")]
    pars = [0.0, 0.0, 0.0] if law == W.OMEGA_CONST else [0.3, 1.0, 0.0]
    return [W.Instance(n=[n], a=[lo], b=[hi], omega_law=law, w0=w0, law=pars, eps=eps, vi_kind=vi, vi_k=k, sigma=sg)
            for n, lo, hi, w0, eps, k, sg in zip(*(p[key].tolist() for key in ("n", "lo", "hi", "w0", "eps", "k", "sigma")))]


def _state(psi, precision):
    return psi if precision == "c128" else psi.to(torch.complex64)


def _box3d(seed):
    """Parameters of the 3D GPE: a repulsive gas in an anisotropic trap, started off the trap's ground state."""
    rng = np.random.default_rng(seed)
    return {"sigma": float(rng.uniform(50.0, 100.0)), "eps": float(rng.uniform(0.02, 0.08)), "k": 2.0,
            "x0": rng.uniform(-0.5, 0.5, 3), "scale": [1.0, 1.5, 2.0], "half": 12.0}


def _psi0_3d(case, p):
    n = case["n"]
    x = -p["half"] + 2.0 * p["half"] / n * torch.arange(n, dtype=torch.float64, device=_device())
    gx, gy, gz = (torch.exp(-0.5 * s * (x - o) ** 2) for s, o in zip(p["scale"], p["x0"].tolist()))
    g = gz[:, None, None] * gy[None, :, None] * gx[None, None, :]
    return (g / torch.sqrt((2.0 * p["half"] / n) ** 3 * (g * g).sum())).to(torch.complex128)


def _fno_shapes(c):
    C, M, P = c["width"], c["modes"], c["proj"]
    s = [("Pin", (c["in_ch"], C)), ("bin", (C,))]
    for l in range(c["layers"]):
        s += [("Rre%d" % l, (M, C, C)), ("Rim%d" % l, (M, C, C)), ("W%d" % l, (C, C)), ("b%d" % l, (C,))]
    return s + [("P1", (C, P)), ("c1", (P,)), ("P2", (P, c["out_ch"])), ("c2", (c["out_ch"],))]


def _fno_inputs(c, seed):
    """Parameters (one FP32 vector), features of random 1D problems and the states that a free rotation in the trap gives."""
    rng = np.random.default_rng(seed)
    parts = []
    for name, sh in _fno_shapes(c):
        fan = 1.0 / 0.1 if len(sh) == 1 else c["width"] if name.startswith("R") else math.sqrt(sh[0])
        parts.append(rng.uniform(-1.0, 1.0, int(np.prod(sh))) / fan)
    params = torch.from_numpy(np.concatenate(parts).astype(np.float32)).to(_device())
    B, L = c["batch"], c["grid"]
    u = torch.from_numpy(np.stack([rng.uniform(lo, hi, B) for lo, hi in
                                   ((0.5, 2.0), (-1.0, 20.0), (0.0, 0.1), (1.0, 4.0), (-1.0, 1.0))])).to(_device())
    w0, sigma, eps, k, x0 = (v[:, None].expand(B, L) for v in u)
    pos = (-12.0 + 24.0 / L * torch.arange(L, dtype=torch.float64, device=_device())).expand(B, L)
    amp = (w0 / math.pi) ** 0.25
    psi = amp * torch.exp(-0.5 * w0 * (pos - x0) ** 2)
    x = torch.stack([psi, torch.zeros_like(psi), pos / 12.0, w0, sigma / 20.0, eps / 0.1, k / 4.0], 2)
    # the coherent state of the unperturbed trap at T = 1
    q, mom = x0 * torch.cos(w0), -w0 * x0 * torch.sin(w0)
    env, ph = amp * torch.exp(-0.5 * w0 * (pos - q) ** 2), mom * (pos - 0.5 * q) - 0.5 * w0
    y = torch.stack([env * torch.cos(ph), env * torch.sin(ph)], 2)
    return params, x.float().contiguous(), y.float().contiguous()


# a learning rate of the last epochs of a cosine schedule from 2e-3
LEARNING_RATE = 2e-6


_streams = []


def _stream():
    """The one stream of a program that calls the framework: its passes follow one another."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve1d", "diag1d"):
        p = _batch(case, seed)
        steps = case.get("steps", 1)
        s = hfs.Solver(_instances(case, p), precision=case["precision"], chunk_steps=min(steps, 512),
                       stream=_stream())
        if kind == "solve1d":
            s.set_schedule(case["h"], case["scheme"], FLOWS[case["flow"]], SPLITS[case["split"]])
            if case["streaming"]:
                s.set_mode(hfs.HFS_MODE_STREAMING, 1)
            if case["projection"]:
                s.set_norm_projection(True)
            if case["reuse"]:
                s.set_schedule_reuse(True)
            if case["graphs"]:
                s.set_graphs(True)
        psi = _state(_flat(p, _psi0(p)), case["precision"])
        torch.cuda.synchronize()  # the solver copies it on its own stream
        s.set_psi(psi)
        return {"kind": kind, "solver": s, "steps": steps}
    if kind == "solve3d":
        p, n = _box3d(seed), case["n"]
        inst = W.Instance(n=[n] * 3, a=[-p["half"]] * 3, b=[p["half"]] * 3, omega_law=W.OMEGA_SIN, w0=1.0,
                          law=[0.3, 1.0, 0.0], axis_scale=p["scale"], eps=p["eps"], vi_kind=W.VI_COS, vi_k=p["k"],
                          sigma=p["sigma"])
        s = hfs.Solver([inst], dim=3, precision=case["precision"], chunk_steps=case["steps"], stream=_stream())
        s.set_schedule(case["h"], case["scheme"], FLOWS[case["flow"]])
        if case["projection"]:
            s.set_norm_projection(True)
        if case["graphs"]:
            s.set_graphs(True)
        psi = _state(_psi0_3d(case, p).reshape(-1), case["precision"])
        torch.cuda.synchronize()
        s.set_psi(psi)
        return {"kind": kind, "solver": s, "steps": case["steps"]}
    params, x, y = _fno_inputs(case, seed)
    cfg = FnoConfig(grid=case["grid"], width=case["width"], modes=case["modes"], layers=case["layers"],
                    in_ch=case["in_ch"], proj=case["proj"], out_ch=case["out_ch"])
    m = Fno(cfg, max_batch=case["batch"], train=kind == "fno_train", seed=None, stream=_stream())
    m.set_params(params)
    torch.cuda.synchronize()
    return {"kind": kind, "model": m, "x": x, "y": y}


def run(state):
    kind = state["kind"]
    if kind in ("solve1d", "solve3d"):
        state["solver"].step(state["steps"])
        return state["solver"].psi
    if kind == "diag1d":
        return {"norm": state["solver"].norm(), "energy": state["solver"].energy()}
    if kind == "fno_forward":
        return state["model"].forward(state["x"])
    loss = state["model"].train_step(state["x"], state["y"], LEARNING_RATE)
    return {"loss": loss, "params": state["model"].params}


# ---------------------------------------------------------------------------
# work of a pass
# ---------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("solve1d", "diag1d"):
        sizes = _sizes(case)
        pts = float(sizes.sum())
        lg = float((sizes * np.log2(sizes)).sum()) / pts
        es = 16 if case["precision"] == "c128" else 8
        if kind == "diag1d":  # one read; one transform and about 20 operations a point for the two sums
            return {"bytes": pts * es, "flops": pts * (5.0 * lg + 20.0)}
        # per sub-stage a forward and an inverse transform and two pointwise phases
        return {"bytes": 2.0 * pts * es, "flops": pts * case["steps"] * STAGES[case["scheme"]] * (10.0 * lg + 22.0)}
    if kind == "solve3d":
        pts = case["n"] ** 3
        es = 16 if case["precision"] == "c128" else 8
        return {"bytes": 2.0 * pts * es,
                "flops": pts * case["steps"] * STAGES[case["scheme"]] * (30.0 * math.log2(case["n"]) + 34.0)}
    B, L, C, M, P, NL = (case[k] for k in ("batch", "grid", "width", "modes", "proj", "layers"))
    params = sum(int(np.prod(sh)) for _, sh in _fno_shapes(case))
    # lift, truncated transform, complex mixing, inverse transform, pointwise product, projection
    flops = 2.0 * B * (L * case["in_ch"] * C + NL * (2 * M * L * C + 4 * M * C * C + 2 * M * L * C + L * C * C)
                       + L * C * P + L * P * case["out_ch"])
    io = 4.0 * B * L * (case["in_ch"] + case["out_ch"])
    if kind == "fno_forward":
        return {"bytes": io + 4.0 * params, "flops": flops}
    # forward and the two products of each contraction backward; parameters and two moments read and written
    return {"bytes": io + 24.0 * params, "flops": 3.0 * flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _composition(scheme):
    """a_i (drifts) and b_i (kicks, one more) of the BAB compositions."""
    if scheme == "strang":
        return [1.0], [0.5, 0.5]
    if scheme == "srkn6_4":
        b1, b2, b3 = 0.0829844064174052, 0.396309801498368, -0.0390563049223486
        a1, a2 = 0.245298957184271, 0.604872665711080
        a3 = 0.5 - (a1 + a2)
        return [a1, a2, a3, a3, a2, a1], [b1, b2, b3, 1.0 - 2.0 * (b1 + b2 + b3), b3, b2, b1]
    if scheme == "ni4_82":
        b1, b2 = 1.0 / 20.0, 49.0 / 180.0
        a1 = 0.5 - math.sqrt(3.0 / 28.0)
        return [a1, 0.5 - a1, 0.5 - a1, a1], [b1, b2, 1.0 - 2.0 * (b1 + b2), b2, b1]
    b1, b2 = 0.811862738544516, -0.677480399532169
    a1, a2 = -0.00758691311877447, 0.317218277973169
    b3 = 0.5 - (b1 + b2)
    return [a1, a2, 1.0 - 2.0 * (a1 + a2), a2, a1], [b1, b2, b3, b3, b2, b1]


def _omega2(law, w0, t):
    if law == "sin":
        return (w0 * (1.0 + 0.3 * np.sin(t))) ** 2
    if law == "cos_sq":
        return w0 ** 2 * (1.0 + 0.3 * np.cos(t))
    return w0 ** 2 * np.ones_like(t)


def _half(w, t):
    """cos, sin / sqrt(w) and 1 - cos of sqrt(w) t, continued to w <= 0."""
    r = np.sqrt(np.abs(w))
    pos = w > 0
    s = np.where(pos, np.sin(0.5 * r * t), np.sinh(0.5 * r * t))
    c = np.where(pos, np.cos(0.5 * r * t), np.cosh(0.5 * r * t))
    omc = np.where(pos, 2.0 * s * s, -2.0 * s * s)
    return 1.0 - omc, np.where(r * np.abs(t) > 0, 2.0 * s * c / np.where(r > 0, r, 1.0), t), omc


def _flow(flow, law, w0, tau, s):
    """Kick f, drift g, kick e (e first) of the harmonic flow over [tau, tau + s] for mass 1."""
    def at(c):
        return _omega2(law, w0, tau + c * s)
    if flow == "lemma2":
        om = np.sqrt(at(0.0))
        f = om * np.tan(0.5 * om * s)
        return f, np.sin(om * s) / om, f
    if flow == "cf4":
        w1, w2, al = at(0.5 - math.sqrt(3.0) / 6.0), at(0.5 + math.sqrt(3.0) / 6.0), 0.5 - 1.0 / math.sqrt(3.0)
        wl, wr = al * w1 + (1.0 - al) * w2, (1.0 - al) * w1 + al * w2
        cl, sl, ol = _half(wl, 0.5 * s)
        cr, sr, orr = _half(wr, 0.5 * s)
        g = sl * cr + cl * sr
        omcc = ol + cl * orr
        return (omcc + wl * sl * sr) / g, g, (omcc + wr * sl * sr) / g
    d = math.sqrt(15.0) / 10.0
    w1, w2, w3 = at(0.5 - d), at(0.5), at(0.5 + d)
    avg = 5.0 * w1 + 8.0 * w2 + 5.0 * w3
    al = avg / 18.0 + s * s / 486.0 * (4.25 * (w1 * w1 + w3 * w3) + 8.0 * w2 * w2 + w1 * w2 + w2 * w3 - 18.5 * w1 * w3)
    be = s * math.sqrt(5.0 / 3.0) * (w3 - w1) * (1.0 / 12.0 + s * s / 3240.0 * avg)
    ga = 1.0 + s * s / 54.0 * (w1 - 2.0 * w2 + w3)
    _, S, omc = _half(al * ga - be * be, s)
    return (omc + be * S) / (ga * S), ga * S, (omc - be * S) / (ga * S)


def _coefficients(case, w0, law, split):
    """f, g, e of every stage and omega^2 at the start of every B flow: arrays (steps, stages, instances)."""
    a, b = _composition(case["scheme"])
    h, m = case["h"], len(a)
    cum = np.concatenate([[0.0], np.cumsum(a)])
    tau = h * (np.arange(case["steps"])[:, None] + cum[None, :])[:, :, None]  # (steps, m + 1, 1)
    w0 = np.asarray(w0)[None, None, :]
    s = h * np.asarray(a)[None, :, None]
    if split == "fourier":
        g = np.broadcast_to(s, (case["steps"], m, w0.shape[2]))
        return np.zeros_like(g), g, np.zeros_like(g), _omega2(law, w0, tau), a, b
    f, g, e = _flow(case["flow"], law, w0, tau[:, :m], s)
    return f, g, e, None, a, b


def _to(v):
    return torch.from_numpy(np.ascontiguousarray(v)).to(_device())


def _phase(angle):
    return torch.polar(torch.ones_like(angle), angle)


def _exact1d(case, p):
    done = {}
    for n, (idx, u) in _psi0(p).items():
        if case["precision"] == "c64":
            u = u.to(torch.complex64).to(torch.complex128)
        x, col, dx = _grid(p, n, idx)
        k = 2.0 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device=_device()) / dx
        V = {"none": torch.zeros_like(x), "x4": x ** 4, "cos": torch.cos(col(p["k"]) * x)}[case["vi"]] * col(p["eps"])
        f, g, e, w2, a, b = _coefficients(case, p["w0"][idx], case["law"], case["split"])
        f, g, e = _to(f)[..., None], _to(g)[..., None], _to(e)[..., None]
        w2 = None if w2 is None else _to(w2)[..., None]
        hx2, hk2, sig = 0.5 * x * x, 0.5 * k * k, col(p["sigma"])
        m, h = len(a), case["h"]
        for step in range(case["steps"]):
            for i in range(m + 1):
                pot = V + sig * (u.real ** 2 + u.imag ** 2)
                if w2 is not None:
                    pot = pot + w2[step, i] * hx2
                if i == m:
                    u = u * _phase(-b[i] * h * pot)
                    break
                u = u * _phase(-b[i] * h * pot - e[step, i] * hx2)
                u = torch.fft.ifft(torch.fft.fft(u) * _phase(-g[step, i] * hk2)) * _phase(-f[step, i] * hx2)
        done[n] = (idx, u)
    return _flat(p, done)


def _exact3d(case, p):
    n, h = case["n"], case["h"]
    u = _psi0_3d(case, p)
    if case["precision"] == "c64":
        u = u.to(torch.complex64).to(torch.complex128)
    x = -p["half"] + 2.0 * p["half"] / n * torch.arange(n, dtype=torch.float64, device=_device())
    k = 2.0 * math.pi * torch.fft.fftfreq(n, 2.0 * p["half"] / n, dtype=torch.float64, device=_device())
    f, g, e, _, a, b = _coefficients(case, p["scale"], "sin", "ho")

    def on_axes(v, q):  # sum over the axes of v_d q^2 / 2; axis 0 of the problem is the last of the array
        hq = 0.5 * q * q
        return v[2] * hq[:, None, None] + v[1] * hq[None, :, None] + v[0] * hq[None, None, :]

    c = p["eps"] * torch.cos(p["k"] * x)
    V = c[:, None, None] + c[None, :, None] + c[None, None, :]
    for step in range(case["steps"]):
        for i in range(len(a) + 1):
            pot = -b[i] * h * (V + p["sigma"] * (u.real ** 2 + u.imag ** 2))
            if i == len(a):
                u = u * _phase(pot)
                break
            u = u * _phase(pot - on_axes(e[step, i].tolist(), x))
            u = torch.fft.ifftn(torch.fft.fftn(u) * _phase(-on_axes(g[step, i].tolist(), k)))
            u = u * _phase(-on_axes(f[step, i].tolist(), x))
    return u.reshape(-1)


def _exact_diag(case, p):
    norm, energy = (np.zeros(case["count"]) for _ in range(2))
    for n, (idx, u) in _psi0(p).items():
        if case["precision"] == "c64":
            u = u.to(torch.complex64).to(torch.complex128)
        x, col, dx = _grid(p, n, idx)
        k = 2.0 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device=_device()) / dx
        d = u.real ** 2 + u.imag ** 2
        V = 0.5 * col(p["w0"]) ** 2 * x * x + col(p["eps"]) * torch.cos(col(p["k"]) * x)
        kin = 0.5 * (k * torch.fft.fft(u).abs()).square().sum(1) / n
        norm[idx] = (dx[:, 0] * d.sum(1)).cpu().numpy()
        energy[idx] = (dx[:, 0] * (kin + (V * d + 0.5 * col(p["sigma"]) * d * d).sum(1))).cpu().numpy()
    return {"norm": norm, "energy": energy}


def _fno_model(c, vec, x):
    q, o = {}, 0
    for name, sh in _fno_shapes(c):
        size = int(np.prod(sh))
        q[name] = vec[o:o + size].view(sh)
        o += size
    H = x @ q["Pin"] + q["bin"]
    for l in range(c["layers"]):
        S = torch.fft.fft(H, dim=1)[:, :c["modes"]]
        Y = torch.einsum("bkc,kco->bko", S, torch.complex(q["Rre%d" % l], q["Rim%d" % l]))
        # the real inverse takes twice the real part of every mode but the constant one
        weight = torch.full((c["modes"], 1), 2.0, dtype=torch.float64, device=Y.device)
        weight[0] = 1.0
        U = torch.fft.ifft(Y * weight, n=c["grid"], dim=1).real
        Z = H @ q["W%d" % l] + q["b%d" % l] + U
        H = torch.nn.functional.gelu(Z) if l < c["layers"] - 1 else Z
    return torch.nn.functional.gelu(H @ q["P1"] + q["c1"]) @ q["P2"] + q["c2"]


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve1d":
        return _exact1d(case, _batch(case, seed))
    if kind == "diag1d":
        return _exact_diag(case, _batch(case, seed))
    if kind == "solve3d":
        return _exact3d(case, _box3d(seed))
    params, x, y = (v.double() for v in _fno_inputs(case, seed))
    if kind == "fno_forward":
        with torch.no_grad():
            return torch.cat([_fno_model(case, params, part) for part in x.split(512)])
    params.requires_grad_(True)
    out = _fno_model(case, params, x)
    loss = ((out - y).flatten(1).norm(dim=1) / y.flatten(1).norm(dim=1)).mean()
    grad, = torch.autograd.grad(loss, params)
    # the first step of Adam (0.9, 0.999, 1e-8): the bias corrections leave g / (|g| + eps)
    with torch.no_grad():
        return {"loss": float(loss), "params": params - LEARNING_RATE * grad / (grad.abs() + 1e-8)}
