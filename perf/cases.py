"""Performance cases of the GB300 adaptive wavelet TRiSK library.

Every case is one call sequence of a program that uses the Python binding: a
forecast (initial fields already on the GPU, adaptation, Runge-Kutta steps, the
resulting state read back), an ensemble of forecasts, one trend evaluation, a
forward and inverse wavelet transform, or one training epoch or evaluation of the
refinement proposal's perceptron.  The sizes are those of the library's workload
configurations, tests and benchmark.

A program keeps its grids and handles and loads new initial conditions into
them, so they are built once per process here (``_base``, ``_handles``); the
inputs of a state (fields, training samples) come from its seed alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1404_0405_gb300 as sww

R, OMEGA, G, DEPTH = 6.371e6, 7.292e-5, 9.80616, 1.0e4
U_SOLID = 2.0 * math.pi * R / (12.0 * 86400.0)   # one rotation in 12 days
F64 = torch.float64


# ---------------------------------------------------------------- cases

def _forecast(name, **kw):
    c = {"name": name, "kind": "forecast", "jmin": 4, "jmax": 8, "patch": 8, "precision": "fp64", "rk": "rk4",
         "field": "jet", "out": 9, "eps": 1e-2, "members": 1, "spread": 0, "learned": False, "adapt": True,
         "steps": 20, "nu": 0.0, "advect": False}
    c.update(kw)
    c["out"] = min(c["out"], c["jmax"])
    return c


def listed():
    return [
        # one trend evaluation on a small adapted grid (the size of the parity tests): the
        # shortest call, launches and barriers only
        {"name": "trend_j2_4_fp64", "kind": "trend", "jmin": 2, "jmax": 4, "patch": 4, "precision": "fp64",
         "field": "jet", "eps": 1e-2},
        # the non-adaptive configuration: uniform J=5, harmonic depth, FP64, CFL steps on a fixed grid
        _forecast("uniform_j5_fp64", jmin=5, jmax=5, field="harmonic", eps=0.0, adapt=False),
        # the adaptive FP64 configuration, a handle stepping alone: the plain form of the benchmark
        _forecast("jet_j4_8_fp64"),
        # the precision form: the same jet in FP32 with the finest level at 9; it refines to level 8 in
        # these steps, where the result is read
        _forecast("jet_j4_9_fp32", jmax=9, precision="fp32", out=8),
        # the learned-mask configuration's kind of flow: a random field with small scales everywhere, a
        # large active grid, the proposal on
        _forecast("turbulence_j4_9_fp32", jmax=9, precision="fp32", field="turbulence", eps=5e-3, learned=True,
                  steps=8),
        # the advection test: a prescribed velocity carries a smooth bell, third-order SSP scheme
        _forecast("advect_j4_7_fp64", jmax=7, field="bell", eps=2e-3, advect=True, rk="ssp43"),
        # the viscous form on small 4 x 4 patches
        _forecast("viscous_j3_6_fp64", jmin=3, jmax=6, patch=4, nu=2.0e5),
        # a small ensemble with the exact criterion (batched phases)
        _forecast("ensemble8_j4_7_fp32", jmax=7, precision="fp32", members=8),
        # the batched configuration: 64 members, Jmax 6..9, eps 1e-2 and 3e-3, learned proposal (the
        # benchmark's chosen form from initial fields to the result), every member read on level 7
        _forecast("ensemble64_j4_9_fp32", jmax=9, precision="fp32", members=64, spread=3, learned=True, out=7),
        # analysis of a full field: forward and inverse wavelet transform, every point live
        {"name": "transform_j4_8_fp32", "kind": "transform", "jmin": 4, "jmax": 8, "patch": 8, "precision": "fp32",
         "field": "jet", "eps": 0.0},
        # training of the proposal: one full-batch epoch on a million patch samples
        {"name": "train_1m", "kind": "train", "n": 1_000_000},
        # evaluation of the proposal on one adaptation's patches (levels 5..9)
        {"name": "predict_54k", "kind": "predict", "n": 54_565},
    ]


def draw(rng):
    kind = rng.choice(["trend", "forecast", "forecast", "ensemble", "transform", "train", "predict"])
    prec = rng.choice(["fp64", "fp32"])
    grids = [(2, 4, 4), (3, 6, 4), (3, 6, 16)]
    if kind in ("train", "predict"):
        return {"kind": kind, "n": int(round(math.exp(rng.uniform(math.log(1e3), math.log(1e6)))))}
    if kind == "trend":
        jmin, jmax, patch = rng.choice(grids + [(4, rng.randint(5, 7), 8)])
        return {"kind": kind, "jmin": jmin, "jmax": jmax, "patch": patch, "precision": prec,
                "field": rng.choice(["jet", "harmonic", "turbulence"]), "eps": math.exp(rng.uniform(-6.0, -3.9))}
    if kind == "transform":
        jmin, jmax, patch = rng.choice(grids[1:] + 2 * [(4, rng.randint(5, 8), 8)])
        return {"kind": kind, "jmin": jmin, "jmax": jmax, "patch": patch, "precision": prec,
                "field": rng.choice(["jet", "harmonic", "turbulence"]),
                "eps": math.exp(rng.uniform(-6.0, -3.9)) if rng.random() < 0.5 else 0.0}
    if kind == "forecast":
        field = rng.choice(["jet", "jet", "harmonic", "turbulence", "bell"])
        adapt = rng.random() < 0.8
        # large active grids in FP64 or without adaptation stop at level 7
        top = 7 if not adapt or (field == "turbulence" and prec == "fp64") else 9
        jmin, jmax, patch = rng.choice(grids[1:] + 2 * [(4, rng.randint(5, top), 8)])
        bell = field == "bell"
        c = _forecast("", jmin=jmin, jmax=jmax, patch=patch, precision=prec, rk=rng.choice(["rk4", "ssp43"]),
                      field=field, eps=math.exp(rng.uniform(-6.0, -3.9)), steps=rng.randint(1, 20),
                      learned=rng.random() < 0.3, adapt=adapt, advect=bell,
                      nu=2.0e5 if not bell and jmax <= 6 and rng.random() < 0.3 else 0.0)
    else:
        field = rng.choice(["jet", "turbulence"])
        jmax = rng.randint(6, 9 if field == "jet" else 7)
        most = 32 if field == "jet" else 8
        c = _forecast("", jmax=jmax, precision=prec if jmax < 9 else "fp32", field=field,
                      eps=math.exp(rng.uniform(-5.8, -3.9)), steps=rng.randint(1, 12), out=7,
                      members=int(round(math.exp(rng.uniform(math.log(2), math.log(most))))),
                      spread=rng.randint(0, jmax - 6), learned=rng.random() < 0.5)
    del c["name"]
    return c


# ---------------------------------------------------------------- grids and handles a program keeps

@functools.lru_cache(maxsize=None)
def _base(jmin, jmax, patch):
    """The handle whose grid the others share: levels 4..9 with 8 x 8 patches, else the case's own."""
    return sww.Model(jmin, jmax, patch=patch, eps=1e-2)


def _grid_of(c):
    return _base(4, 9, 8) if (c["jmin"], c["patch"]) == (4, 8) else _base(c["jmin"], c["jmax"], c["patch"])


def _model(c, jmax, eps, H=DEPTH):
    phased = c.get("members", 1) > 1
    m = sww.Model(c["jmin"], jmax, H=H, patch=c["patch"], rk=c.get("rk", "rk4"), eps=eps, share=_grid_of(c),
                  precision=c["precision"], persistent="phased" if phased else True, blocks_per_sm=2 if phased else 0,
                  nu=c.get("nu", 0.0), advect=c.get("advect", False))
    if c.get("learned"):
        m.set_learned(2, _proposal(), 0.9)
    return m


_kept = {}


def _handles(c):
    """The case's handles, built once: a program loads new initial conditions into them.  Members of an
    ensemble with spread s have finest levels jmax - s..jmax in turn, and eps or 0.3 eps."""
    key = tuple(sorted((k, v) for k, v in c.items() if k not in ("name", "field", "out", "steps", "adapt")))
    if key not in _kept:
        if len(_kept) >= 4:   # a few handles of earlier cases at most
            for m in _kept.pop(next(iter(_kept))):
                m.close()
        ms = []
        for k in range(c["members"]):
            jmax = c["jmax"] - k % (c["spread"] + 1)
            eps = c["eps"] * (0.3 if c["spread"] and (k // (c["spread"] + 1)) % 2 else 1.0)
            ms.append(_model(c, jmax, eps, 0.0 if c["advect"] else DEPTH))
        _kept[key] = ms
    return _kept[key]


def _proposal():
    """Parameters of a perceptron that proposes a patch when a neighbour's coefficients are a few times the
    threshold."""
    W1 = np.zeros((sww.MLP_FEATURES, sww.MLP_HIDDEN))
    b1 = np.zeros(sww.MLP_HIDDEN)
    w2 = np.zeros(sww.MLP_HIDDEN)
    W1[4, 0] = W1[5, 1] = 1.0
    b1[:2] = -0.75
    w2[:2] = 4.0
    return np.concatenate([W1.ravel(), b1, w2, [-2.0]]).astype(np.float32)


# ---------------------------------------------------------------- initial fields (on the GPU)

@functools.lru_cache(maxsize=16)
def _points(jmin, jmax, patch, level):
    """Node positions, edge midpoints and unit edge tangents of a level, in the library's order."""
    xyz, en = _base(jmin, jmax, patch).grid(level)
    x = torch.from_numpy(xyz).cuda()
    e = torch.from_numpy(en.astype(np.int64)).cuda()
    a, b = x[e[:, 0]], x[e[:, 1]]
    mid = torch.nn.functional.normalize(a + b, dim=1)
    return x, mid, torch.nn.functional.normalize(b - a, dim=1)


def _jet(x, mid, tan, rng):
    """Zonal jet of 80 m/s and 7 degrees width in gradient-wind balance, and three height bumps of 120 m."""
    lat0 = math.radians(rng.uniform(20.0, 60.0))
    wind = lambda la: 80.0 * torch.exp(-((la - lat0) / math.radians(7.0)) ** 2)
    n = 20001
    la = torch.linspace(-math.pi / 2, math.pi / 2, n, dtype=F64, device="cuda")
    u = wind(la)
    f = -R * u * (2.0 * OMEGA * torch.sin(la) + u * torch.tan(la.clamp(-1.57, 1.57)) / R) / G
    step = math.pi / (n - 1)
    h = torch.cat([torch.zeros(1, dtype=F64, device="cuda"), torch.cumsum(0.5 * (f[1:] + f[:-1]) * step, 0)])
    h = h - (h * torch.cos(la)).sum() * step / 2.0
    s = ((torch.asin(x[:, 2].clamp(-1, 1)) + math.pi / 2) / step).clamp(0, n - 1.000001)
    i = s.long()
    dh = h[i] + (s - i) * (h[i + 1] - h[i])
    for _ in range(3):
        lon, lat = rng.uniform(-math.pi, math.pi), math.radians(rng.uniform(-70.0, 70.0))
        b = torch.tensor([math.cos(lat) * math.cos(lon), math.cos(lat) * math.sin(lon), math.sin(lat)], dtype=F64,
                         device="cuda")
        dh += 120.0 * torch.exp(-(torch.acos((x @ b).clamp(-1, 1)) * R / 5.0e5) ** 2)
    east = (mid[:, 0] * tan[:, 1] - mid[:, 1] * tan[:, 0]) / torch.hypot(mid[:, 0], mid[:, 1]).clamp_min(1e-12)
    return dh, wind(torch.asin(mid[:, 2].clamp(-1, 1))) * east


def _ridges(x, mid, tan, rng, lo, hi, speed, power):
    """A geostrophic sum of waves cos(l x.n + phase) about random axes n, wavenumbers lo..hi, stream function
    amplitudes l^-power, scaled to an rms velocity (or, for speed 0, to 100 m of depth)."""
    psi = torch.zeros(len(x), dtype=F64, device="cuda")
    grad = torch.zeros_like(mid)
    for _ in range(48):
        n = rng.normal(size=3)
        n = torch.from_numpy(n / np.linalg.norm(n)).cuda()
        l, ph = float(rng.uniform(lo, hi)), float(rng.uniform(0, 2 * math.pi))
        a = l ** -power
        psi += a * torch.cos(l * (x @ n) + ph)
        grad += (-a * l * torch.sin(l * (mid @ n) + ph))[:, None] * n
    f0 = 2.0 * OMEGA * math.sin(math.pi / 4)
    u = (torch.linalg.cross(mid, grad) * tan).sum(1) / R      # psi in m^2/s after the scaling below
    scale = speed / (u.square().mean().sqrt() * math.sqrt(2.0)) if speed else 100.0 * G / f0 / psi.abs().max()
    return scale * f0 / G * (psi - psi.mean()), scale * u


def _bell(x, mid, tan, rng):
    """Smooth bell of 1000 m and radius R/3 at a random point of the equator, carried by solid-body rotation
    about an axis tilted from the pole."""
    lon, al = rng.uniform(-math.pi, math.pi), rng.uniform(0.0, math.pi / 4)
    c = torch.tensor([math.cos(lon), math.sin(lon), 0.0], dtype=F64, device="cuda")
    axis = torch.tensor([-math.sin(al), 0.0, math.cos(al)], dtype=F64, device="cuda")
    L = R / 3.0
    r = R * torch.acos((x @ c).clamp(-1, 1))
    r = torch.where(r < math.sqrt(2.0) * L, r, torch.zeros_like(r))
    h = torch.where(r > 0, 1000.0 * torch.exp(r * r / (r * r - 2.0 * L * L)), torch.zeros_like(r))
    return h, U_SOLID * (torch.linalg.cross(axis.expand_as(mid), mid) * tan).sum(1)


def _fields(c, level, seed):
    base = (4, 9, 8) if (c["jmin"], c["patch"]) == (4, 8) else (c["jmin"], c["jmax"], c["patch"])
    x, mid, tan = _points(*base, level)
    rng = np.random.default_rng([seed, 7])
    if c["field"] == "jet":
        dh, u = _jet(x, mid, tan, rng)
    elif c["field"] == "harmonic":
        dh, u = _ridges(x, mid, tan, rng, 1.0, 8.0, 0.0, 1.0)
    elif c["field"] == "turbulence":
        dh, u = _ridges(x, mid, tan, rng, 12.0, 96.0, 20.0, 2.0)
    else:
        dh, u = _bell(x, mid, tan, rng)
    return dh.contiguous(), u.contiguous()


# ---------------------------------------------------------------- training samples

def _samples(n, seed):
    """Patch features as the library computes them (logs of coefficient ratios, most patches quiet; a live
    fraction; a level) and labels that follow the neighbours' coefficients."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = lambda *s: torch.rand(*s, generator=g, device="cuda")
    X = torch.empty(n, sww.MLP_FEATURES, device="cuda")
    X[:, :6] = torch.relu(6.0 * r(n, 6) - 4.0 + 2.0 * r(n, 1))
    X[:, 4:6] = torch.maximum(X[:, 4:6], X[:, 0:2])
    X[:, 6] = (r(n) * 64.0).floor() / 64.0
    X[:, 7] = (1.0 + (r(n) * 5.0).floor()) / 5.0
    y = ((X[:, 4] + X[:, 5] + r(n)) > 3.0).float()
    return X, y


def _params(seed):
    rng = np.random.default_rng([seed, 3])
    F, H = sww.MLP_FEATURES, sww.MLP_HIDDEN
    p = np.concatenate([rng.normal(0, math.sqrt(2.0 / F), F * H), rng.normal(0, 0.1, H),
                        rng.normal(0, math.sqrt(1.0 / H), H), [-1.0]])
    return torch.from_numpy(p.astype(np.float32)).cuda()


# ---------------------------------------------------------------- the path

def prepare(case, seed):
    k = case["kind"]
    if k in ("train", "predict"):
        X, y = _samples(case["n"], seed)
        s = {"X": X, "params": _params(seed)}
        if k == "predict":
            s["out"] = torch.empty(case["n"], device="cuda")
        else:
            z = lambda n: torch.zeros(n, device="cuda")
            s.update(y=y, m=z(sww.MLP_PARAMS), v=z(sww.MLP_PARAMS), work=z(sww.MLP_WORK), out=z(sww.MLP_PARAMS + 1),
                     t=0)
    elif k == "forecast":
        hs = _handles(case)
        s = {"handles": hs,
             "fields": [_fields(case, h.jmax, seed * 1000 + i) for i, h in enumerate(hs)]}
    else:
        # a handle that holds a state, on an adapted grid or (eps 0) with every point live
        h = _model(case, case["jmax"], case["eps"])
        h.set_state(*_fields(case, case["jmax"], seed))
        if case["eps"] > 0:
            h.adapt()
        s = {"handle": h}
    s["case"] = case
    torch.cuda.synchronize()
    return s


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "predict":
        sww.mlp_predict(state["X"], state["params"], state["out"])
        return state["out"]
    if k == "train":
        s = state
        s["t"] += 1
        sww.mlp_loss_grad(s["X"], s["y"], s["params"], 4.0, s["work"], s["out"])
        sww.mlp_adam(s["params"], s["out"], s["m"], s["v"], s["t"], 1e-2)
        return [s["out"], s["params"], s["m"], s["v"]]
    if k == "trend":
        h = state["handle"]
        h.rhs()
        return [h.get(j, q) for j in range(c["jmin"], c["jmax"] + 1) for q in (sww.DH_T, sww.U_T)]
    if k == "transform":
        h = state["handle"]
        h.forward()
        h.inverse()
        return list(h.get_state(c["jmax"]))
    hs = state["handles"]
    for h, (dh, u) in zip(hs, state["fields"]):
        h.set_state(dh, u)
        if c["adapt"]:
            h.adapt()
    if len(hs) > 1:
        sww.step_ensemble(hs, -1.0, c["steps"], c["adapt"])
    else:
        hs[0].step(-1.0, c["steps"], c["adapt"])
    got = [h.get_state(min(c["out"], h.jmax)) for h in hs]
    live = np.array([h.live_nodes() for h in hs])
    return [np.concatenate([g[0] for g in got]), np.concatenate([g[1] for g in got]), live]


# ---------------------------------------------------------------- work

def _cells(c, jmax):
    """Live cells over all levels, roughly: the whole hierarchy without adaptation, else the fraction that
    these fields leave at such thresholds."""
    full = sum(10 * 4 ** j + 2 for j in range(c["jmin"], jmax + 1))
    if c["eps"] == 0 or not c.get("adapt", True):
        return full
    return min(full, {"jet": 20_000, "harmonic": 6_000, "turbulence": 400_000, "bell": 50_000}[c["field"]])


def work(case):
    """Bytes and operations of one pass at the least: the initial fields read and the result written, and per
    live cell (a node, three edges, two triangles) and Runge-Kutta stage the state and its base read, the new
    state written and 17 words of FP64 geometry; about 400 operations a cell and stage."""
    k = case["kind"]
    if k in ("train", "predict"):
        n, F, H = case["n"], sww.MLP_FEATURES, sww.MLP_HIDDEN
        if k == "train":
            return {"bytes": 4 * n * (F + 1) + 4 * 8 * sww.MLP_PARAMS, "flops": n * (4 * F * H + 8 * H)}
        return {"bytes": 4 * n * (F + 1), "flops": n * (2 * F * H + 4 * H)}
    w = 8 if case["precision"] == "fp64" else 4
    if k == "transform":
        n = _cells(case, case["jmax"])
        return {"bytes": n * (3 * 4 * w) + 8 * 4 * 10 * 4 ** case["jmax"], "flops": n * 3 * 12 * 2 * 2}
    if k == "trend":
        n = _cells(case, case["jmax"])
        return {"bytes": n * (2 * 4 * w + 136), "flops": n * 400}
    b = f = 0
    for i in range(case["members"]):
        jmax = case["jmax"] - i % (case["spread"] + 1)
        n = _cells(case, jmax)
        b += 8 * 40 * 4 ** jmax + 8 * 40 * 4 ** min(case["out"], jmax)
        b += n * case["steps"] * 4 * (12 * w + 136)
        f += n * case["steps"] * 4 * 400
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- 64-bit values

def _mlp64(X, params):
    """Logits, hidden activations and pre-activations in 64 bits (weights rounded to BF16 for use)."""
    F, H = sww.MLP_FEATURES, sww.MLP_HIDDEN
    bf = lambda p: p.to(torch.bfloat16).double()
    W1 = bf(params[: F * H]).reshape(F, H)
    b1, w2, b2 = params[F * H: F * H + H].double(), bf(params[F * H + H: F * H + 2 * H]), params[-1].double()
    z = X.double() @ W1 + b1
    a = torch.relu(z)
    return a @ w2 + b2, a, z, w2


def exact(case, seed):
    k = case["kind"]
    if k == "predict":
        X, _ = _samples(case["n"], seed)
        return torch.sigmoid(_mlp64(X, _params(seed))[0])
    if k == "train":
        X, y = _samples(case["n"], seed)
        params, t, w = _params(seed), y.double(), 4.0
        logit, a, z, w2 = _mlp64(X, params)
        p = torch.sigmoid(logit)
        g = w * t * (p - 1.0) + (1.0 - t) * p
        sp = torch.nn.functional.softplus(logit)
        loss = (w * t * (sp - logit) + (1.0 - t) * sp).mean()
        dz = torch.where(z > 0, g[:, None] * w2, torch.zeros_like(z))
        n = len(X)
        grad = torch.cat([(X.double().T @ dz).reshape(-1) / n, dz.mean(0), (a.T @ g) / n, g.mean().reshape(1)])
        m, v = 0.1 * grad, 0.001 * grad * grad
        new = params.double() - 1e-2 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
        return [torch.cat([grad, loss.reshape(1)]), new, m, v]
    if k == "transform" and case["eps"] == 0:
        # the inverse transform of the forward transform is the field itself
        dh, u = _fields(case, case["jmax"], seed)
        return [dh, u]
    return None   # a forecast, a trend or an adapted grid has no value without a solver of its own
