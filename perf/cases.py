"""Performance cases of the library: what its users run, over the sizes they run it at.

Every pass starts from a state handed in as a CUDA tensor (set_state), sets
the draw counters, runs the forecast, analysis, batch or network calls a twin
experiment makes, and reads the state back (get_state), so that a pass on the
same inputs repeats bit for bit.  `exact` restates the same mathematics in
64-bit torch and numpy.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1910_01031_gb300 import iewpf

DEV = "cuda" if torch.cuda.is_available() else "cpu"
PHYS = {"dx": 2000.0, "dy": 2000.0, "g": 9.81, "f": 1.2e-4, "H": 230.0, "theta": 1.3, "dt": 60.0, "q0": 5e-4}
SIGMA = 2.3                    # observation error of hu, hv: 0.01 m/s times the depth
FLOP_STEP = 338                # of one scheme step per cell, a fused multiply-add as two
FLOP_NET = 2 * 9 * (3 * 64 + 4 * 64 * 64 + 64 * 3)   # of one network call per pixel


def listed():
    return [
        # the smallest twin experiment: one observation cycle's forecast (4 model
        # steps with model error, the fifth without) and its analysis
        _forecast("forecast_64_ne10", 64, 64, 10),
        _analysis("analysis_64_ne10_1drifter", 64, 64, 10, "drifter", 1),
        # the paper's ensemble: 512 x 512 cells, 100 particles, 64 drifters
        _forecast("forecast_512_ne100", 512, 512, 100),
        _analysis("analysis_512_ne100_64drifters", 512, 512, 100, "drifter", 64),
        # a quarter of the largest ensemble (1024 x 1024): one model step, and the
        # analysis of the 1521 moorings every 26 cells
        _forecast("forecast_1024_ne256", 1024, 1024, 256, steps_err=1, steps_plain=0),
        _analysis("analysis_1024_ne256_1521moorings", 1024, 1024, 256, "mooring", 1521, spacing=26),
        # moorings close enough to couple: the dense factor fills in
        _analysis("analysis_624_ne1000_1521coupled", 624, 624, 1000, "mooring", 1521, spacing=16),
        # whole cycles of many small problems in one batch, and of the ragged
        # 500 x 300 experiments (c_omega 5, Courant number 0.8, 120 moorings)
        # that rank histograms are made from
        _batch("batch_64x64_ne10_x64", " ".join(["64x64x10x1"] * 64), "drifter"),
        _batch("batch_500x300_ne40_x8", " ".join(["500x300x40x120"] * 8), "mooring", c_omega=5, courant=0.8),
        # the learned surrogate: a network call over an ensemble on the device, the
        # loss and gradients of one training batch, and half an hour of drift forecast
        {"name": "surrogate_apply_256_n256", "kind": "apply", "nx": 256, "ny": 256, "n": 256},
        {"name": "surrogate_grad_64_n32", "kind": "grad", "nx": 64, "ny": 64, "n": 32},
        _drift("drift_surrogate_256_ne100", 256, 256, 100, 64, 1800.0, True),
    ]


def _forecast(name, nx, ny, ne, steps_err=4, steps_plain=1, c_omega=3, courant=0.45):
    return {"name": name, "kind": "forecast", "nx": nx, "ny": ny, "ne": ne, "steps_err": steps_err,
            "steps_plain": steps_plain, "c_omega": c_omega, "courant": courant}


def _analysis(name, nx, ny, ne, obs, n_obs, spacing=0, c_omega=3, scheme=0, dense=1):
    return {"name": name, "kind": "analysis", "nx": nx, "ny": ny, "ne": ne, "obs": obs, "n_obs": n_obs,
            "spacing": spacing, "c_omega": c_omega, "scheme": scheme, "dense": dense}


def _batch(name, problems, obs, c_omega=3, courant=0.45):
    """problems: "nx x ny x particles x observations" of each, separated by blanks."""
    return {"name": name, "kind": "batch", "problems": problems, "obs": obs, "c_omega": c_omega, "courant": courant}


def _drift(name, nx, ny, ne, nd, seconds, surrogate):
    return {"name": name, "kind": "drift", "nx": nx, "ny": ny, "ne": ne, "nd": nd, "seconds": seconds,
            "every": 600.0, "surrogate": surrogate}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forecast", "forecast", "analysis", "analysis", "batch", "apply", "grad", "drift"])
    if kind == "forecast":
        nx, ny = _log(rng, 48, 1024), _log(rng, 48, 1024)
        ne = max(1, min(_log(rng, 4, 1000), 60_000_000 // (nx * ny)))
        return dict(_forecast("", nx, ny, ne, steps_err=rng.randint(0, 4), steps_plain=1, c_omega=rng.choice([1, 3]),
                              courant=rng.choice([0.45, 0.8])))
    if kind == "analysis":
        c = rng.choice([1, 3])
        if rng.random() < 0.5:
            nx, ny = _log(rng, 48, 1024), _log(rng, 48, 1024)
            ne = max(1, min(_log(rng, 4, 500), 60_000_000 // (nx * ny)))
            # the local blocks and the random part are scaled by the state: beta stays positive
            n_obs = max(1, min(_log(rng, 1, 128), nx * ny // 600))
            return _analysis("", nx, ny, ne, "drifter", n_obs, c_omega=c, scheme=rng.choice([0, 0, 1]),
                             dense=rng.choice([1, 1, 0]))
        m = rng.randint(3, 39)
        spacing = rng.choice([16, 18, 21, 26])
        n = m * spacing + rng.randint(16, 40)
        ne = max(1, min(_log(rng, 8, 500), 60_000_000 // (n * n)))
        return _analysis("", n, n, ne, "mooring", m * m, spacing=spacing, c_omega=3, scheme=rng.choice([0, 0, 1]))
    if kind == "batch":
        parts = []
        for _ in range(rng.randint(2, 24)):
            nx, ny = _log(rng, 48, 300), _log(rng, 48, 300)
            parts.append("%dx%dx%dx%d" % (nx, ny, rng.randint(4, 40), max(1, min(rng.randint(1, 64), nx * ny // 600))))
        return _batch("", " ".join(parts), "drifter")
    if kind == "apply":
        nx, ny = rng.choice([64, 128, 256, 384, 512]), 16 * rng.randint(2, 24)
        return {"name": "", "kind": "apply", "nx": nx, "ny": ny, "n": max(1, min(_log(rng, 4, 400), 16_000_000 // (nx * ny)))}
    if kind == "grad":
        nx, ny = rng.choice([64, 128, 192]), 16 * rng.randint(2, 8)
        return {"name": "", "kind": "grad", "nx": nx, "ny": ny, "n": max(1, min(_log(rng, 2, 64), 600_000 // (nx * ny)))}
    nx, ny = _log(rng, 64, 400), _log(rng, 64, 400)
    return _drift("", nx, ny, max(1, min(_log(rng, 10, 300), 6_000_000 // (nx * ny))), rng.randint(1, 64), 1800.0, False)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + k)


def _state(nx, ny, ne, seed, k=0):
    """Two opposite zonal jets in geostrophic balance with white noise of 1 mm in
    eta and, as model errors leave them, smooth balanced perturbations."""
    P, w = PHYS, 8.0 * PHYS["dy"]
    y = (torch.arange(ny, device=DEV, dtype=torch.float64) + 0.5) * P["dy"]
    a1, a2 = (y - ny * P["dy"] / 4) / w, (y - 3 * ny * P["dy"] / 4) / w
    eta = 0.05 * (torch.tanh(a1) - torch.tanh(a2))
    hu = -(P["g"] * P["H"] / P["f"]) * 0.05 / w * (1 / torch.cosh(a1) ** 2 - 1 / torch.cosh(a2) ** 2)
    U = torch.zeros((ne, 3, ny, nx), device=DEV)
    U[:, 0] = (eta - eta.mean()).float()[:, None]
    U[:, 1] = hu.float()[:, None]
    g = _gen(seed, k)
    s = P["g"] * P["H"] / P["f"]
    for p0 in range(0, ne, 64):
        V = U[p0:p0 + 64]
        r = torch.randn((V.shape[0], ny, nx), generator=g, device=DEV) * (1e-3 / 0.053)
        for d in (1, 2, 4):
            for ax in (1, 2):
                r = 0.5 * r + 0.25 * (r.roll(d, ax) + r.roll(-d, ax))
        V[:, 0] += r + 1e-3 * torch.randn(r.shape, generator=g, device=DEV)
        V[:, 1] -= s / (2 * P["dy"]) * (r.roll(-1, 1) - r.roll(1, 1))
        V[:, 2] += s / (2 * P["dx"]) * (r.roll(-1, 2) - r.roll(1, 2))
    return U


def _drifters(nx, ny, n, seed):
    """A k x k lattice of positions, each moved by up to two cells."""
    k = math.ceil(math.sqrt(n))
    rng = np.random.default_rng(int(seed))
    xy = np.array([[(i % k + 0.5) * nx / k, (i // k + 0.5) * ny / k] for i in range(n)]) + rng.uniform(-2, 2, (n, 2))
    return xy * [PHYS["dx"], PHYS["dy"]]


def _moorings(nx, ny, n, spacing):
    """Cell centres of a lattice: square with the given spacing, or the western half of a 20 x 12 one."""
    if spacing:
        m = math.isqrt(n)
        ox, oy = (nx - spacing * (m - 1)) // 2, (ny - spacing * (m - 1)) // 2
        c = [(ox + spacing * p, oy + spacing * q) for q in range(m) for p in range(m)]
    else:
        c = [(nx // 40 + nx // 20 * p, ny // 24 + ny // 12 * q) for q in range(12) for p in range(10)][:n]
    return (np.array(c, np.float64) + 0.5) * [PHYS["dx"], PHYS["dy"]]


def _cells(xy, nx, ny):
    return np.floor(xy / [PHYS["dx"], PHYS["dy"]]).astype(np.int64) % [nx, ny]


def _observe(xy, nx, ny, seed, k):
    """(hu, hv) of another draw of the initial state at the positions, with noise."""
    T = _state(nx, ny, 1, seed, 7919 + k)[0].double().cpu().numpy()
    c = _cells(xy, nx, ny)
    e = T[0][c[:, 1], c[:, 0]]
    v = np.stack([T[1][c[:, 1], c[:, 0]], T[2][c[:, 1], c[:, 0]]], 1) * (PHYS["H"] / (PHYS["H"] + e))[:, None]
    return v + SIGMA * np.random.default_rng(1000 * int(seed) + k).standard_normal(v.shape)


def _params(nx, ny, ne, c_omega=3, courant=0.45, obs="drifter", n_obs=0, scheme=0, dense=1, nd=0, inst=0):
    P = PHYS
    return iewpf.Params(nx, ny, P["dx"], P["dy"], P["g"], P["f"], P["H"], P["theta"], courant, P["dt"], c_omega, P["q0"],
                        0.75 * c_omega * P["dx"], 0x191001031, ne,
                        iewpf.OBS_MOORING if obs == "mooring" else iewpf.OBS_DRIFTER, n_obs, SIGMA, dense, inst, nd,
                        scheme)


def _counters(seed):
    return 100 + int(seed) % 1000, 20 + int(seed) % 1000


def _problems(case):
    return [tuple(int(v) for v in p.split("x")) for p in case["problems"].split()]


def _batch_inputs(case, seed):
    """Per problem: state, observed positions and values."""
    out = []
    for i, (nx, ny, ne, n) in enumerate(_problems(case)):
        xy = _moorings(nx, ny, n, 0) if case["obs"] == "mooring" else _drifters(nx, ny, n, seed + i)
        out.append((_state(nx, ny, ne, seed, i + 1), xy, _observe(xy, nx, ny, seed, i + 1)))
    return out


IN_SCALE, OUT_SCALE = (10.0, 0.05, 0.05), (2e-4, 0.02, 0.02)


def _weights(seed, depth=6):
    """He-normal weights, the last layer scaled by 0.1 as a new network's, biases a little off zero; flat,
    per layer [3][3][cout][cin] (3 padded to 16) and bias."""
    rng = np.random.default_rng(77 + int(seed))
    flat = []
    for l in range(depth):
        ci, co = (16 if l == 0 else 64), (16 if l == depth - 1 else 64)
        ri, ro = min(ci, 3) if l == 0 else 64, min(co, 3) if l == depth - 1 else 64
        W = np.zeros((3, 3, co, ci), np.float32)
        W[:, :, :ro, :ri] = rng.standard_normal((3, 3, ro, ri)) * math.sqrt(2 / (9 * ri)) * (0.1 if l == depth - 1 else 1)
        b = np.zeros(co, np.float32)
        b[:ro] = 0.05 * rng.standard_normal(ro)
        flat += [W.ravel(), b]
    return np.concatenate(flat)


def _network(case, seed):
    s = iewpf.Surrogate(case["nx"], case["ny"])
    s.set_params(_weights(seed))
    s.set_scales(IN_SCALE, OUT_SCALE)
    return s


def _pairs(case, seed):
    """Host states and the states ten model steps on, as a training set holds them (the change as random as OUT_SCALE)."""
    X = _state(case["nx"], case["ny"], case["n"], seed)
    D = torch.randn(X.shape, generator=_gen(seed, 5), device=DEV) * torch.tensor(OUT_SCALE, device=DEV)[:, None, None]
    return X.cpu().numpy(), (X + D).cpu().numpy()


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "ctr": _counters(seed)}
    if kind == "batch":
        data = _batch_inputs(case, seed)
        probs = _problems(case)
        P = [_params(nx, ny, ne, case["c_omega"], case["courant"], case["obs"], n, inst=i)
             for i, (nx, ny, ne, n) in enumerate(probs)]
        moor = case["obs"] == "mooring"
        s["b"] = iewpf.Batch(P, [d[1] for d in data] if moor else None)
        s["U"] = [d[0] for d in data]
        s["out"] = [torch.empty_like(u) for u in s["U"]]
        s["obs"] = [(None if moor else d[1], d[2]) for d in data]
        s["b"].tune()
        return s
    if kind == "grad":
        s["sur"] = _network(case, seed)
        s["X"], s["Y"] = _pairs(case, seed)
        return s
    if kind == "apply":
        s["sur"] = _network(case, seed)
        s["U"] = _state(case["nx"], case["ny"], case["n"], seed)
        s["out"] = torch.empty_like(s["U"])
        return s
    nx, ny, ne = case["nx"], case["ny"], case["ne"]
    s["U"] = _state(nx, ny, ne, seed)
    s["out"] = torch.empty_like(s["U"])
    if kind == "forecast":
        s["e"] = iewpf.Ensemble(_params(nx, ny, ne, case["c_omega"], case["courant"]))
        s["e"].tune()
    elif kind == "analysis":
        moor = case["obs"] == "mooring"
        xy = _moorings(nx, ny, case["n_obs"], case["spacing"]) if moor else _drifters(nx, ny, case["n_obs"], seed)
        s["e"] = iewpf.Ensemble(_params(nx, ny, ne, case["c_omega"], 0.45, case["obs"], case["n_obs"], case["scheme"],
                                        case["dense"]), xy if moor else None)
        s["xy"], s["y"] = (None if moor else xy), _observe(xy, nx, ny, seed, 0)
    else:
        s["e"] = iewpf.Ensemble(_params(nx, ny, ne, nd=case["nd"]))
        s["xy"] = _drifters(nx, ny, case["nd"], seed)
        if case["surrogate"]:
            s["sur"] = _network(case, seed)
            s["e"].set_surrogate(s["sur"], 10)
        s["e"].tune()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        return s["sur"].apply_device(s["U"], s["out"])
    if kind == "grad":
        loss, grad = s["sur"].loss_grad(s["X"], s["Y"])
        return {"loss": loss, "grad": grad}
    if kind == "batch":
        for e, u in zip(s["b"].instances, s["U"]):
            e.set_state(u)
            e.set_counters(*s["ctr"])
        diag = s["b"].cycle(5, s["obs"])
        # target weights and betas, logged in single precision
        return {"diag": diag[:, :2].astype(np.float32),
                "state": torch.cat([e.get_state(o).view(-1) for e, o in zip(s["b"].instances, s["out"])])}
    e = s["e"]
    e.set_state(s["U"])
    e.set_counters(*s["ctr"])
    if kind == "forecast":
        if case["steps_err"]:
            e.forecast(case["steps_err"], True)
        if case["steps_plain"]:
            e.forecast(case["steps_plain"], False)
        return e.get_state(s["out"])
    if kind == "analysis":
        d = e.assimilate(s["xy"], s["y"])
        return {"state": e.get_state(s["out"]), "diag": d}
    traj = e.drifter_forecast(s["xy"], case["seconds"] / 3600.0, case["every"], case["surrogate"])
    return {"traj": traj.astype(np.float32), "state": e.get_state(s["out"])}


def _n_sub(courant):
    return math.ceil(PHYS["dt"] * 4 / courant * (math.sqrt(PHYS["g"] * PHYS["H"]) + 0.5) / PHYS["dx"])


def work(case):
    kind = case["kind"]
    if kind in ("apply", "grad"):
        pix = case["nx"] * case["ny"] * case["n"]
        return {"bytes": 24 * pix, "flops": FLOP_NET * pix * (1 if kind == "apply" else 3)}
    if kind == "batch":
        cells = sum(nx * ny * ne for nx, ny, ne, _ in _problems(case))
        return {"bytes": 24 * cells, "flops": 5 * _n_sub(case["courant"]) * FLOP_STEP * cells}
    cells = case["nx"] * case["ny"] * case["ne"]
    if kind == "forecast":
        return {"bytes": 24 * cells,
                "flops": (case["steps_err"] + case["steps_plain"]) * _n_sub(case["courant"]) * FLOP_STEP * cells}
    if kind == "analysis":
        # the update's interpolation and differences per cell, and two normals per coarse point
        return {"bytes": 24 * cells, "flops": 30 * cells + 100 * cells / case["c_omega"] ** 2}
    if case["surrogate"]:
        return {"bytes": 24 * cells, "flops": case["seconds"] / 600.0 * FLOP_NET * cells}
    return {"bytes": 24 * cells, "flops": case["seconds"] / 60.0 * _n_sub(0.45) * FLOP_STEP * cells}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
D = torch.float64


def _minmod(a, b):
    t = PHYS["theta"]
    m = torch.minimum(torch.minimum(t * a.abs(), t * b.abs()), 0.5 * (a + b).abs())
    return torch.where(a * b > 0, torch.sign(a) * m, torch.zeros_like(m))


def _flux(eL, nL, tL, eR, nR, tR):
    g, H = PHYS["g"], PHYS["H"]
    hL, hR = H + eL, H + eR
    uL, uR = nL / hL, nR / hR
    cL, cR = (g * hL).sqrt(), (g * hR).sqrt()
    ap = torch.maximum(uL + cL, uR + cR).clamp(min=0)
    am = torch.minimum(uL - cL, uR - cR).clamp(max=0)
    w = 1 / (ap - am)
    F0 = (ap * nL - am * nR + ap * am * (eR - eL)) * w
    F1 = (ap * (nL * uL + g * eL * (H + eL / 2)) - am * (nR * uR + g * eR * (H + eR / 2)) + ap * am * (nR - nL)) * w
    return F0, F1, F0 * torch.where(F0 >= 0, tL / hL, tR / hR)


def _rhs(U):
    """Central-upwind right-hand side of the rotating shallow-water equations, eta reconstructed through the
    potentials g eta - f V (in x) and g eta + f U (in y)."""
    P = PHYS
    e, qu, qv = U[:, 0], U[:, 1], U[:, 2]
    h = P["H"] + e
    out = [0, 0, 0]
    for ax, d, n, t, vel, sgn in ((2, P["dx"], qu, qv, qv / h, -1.0), (1, P["dy"], qv, qu, qu / h, 1.0)):
        def fwd(a):
            return a.roll(-1, ax) - a
        K = P["g"] * fwd(e) + sgn * 0.5 * P["f"] * d * (vel + vel.roll(-1, ax))
        dn, dt = fwd(n), fwd(t)
        ex = (_minmod(K.roll(1, ax), K) - sgn * P["f"] * d * vel) / (2 * P["g"])
        sn, st = 0.5 * _minmod(dn.roll(1, ax), dn), 0.5 * _minmod(dt.roll(1, ax), dt)
        fl = _flux(e + ex, n + sn, t + st, (e - ex).roll(-1, ax), (n - sn).roll(-1, ax), (t - st).roll(-1, ax))
        for q, x in zip((0, 1, 2) if ax == 2 else (0, 2, 1), fl):
            out[q] = out[q] - (x - x.roll(1, ax)) / d
    return torch.stack([out[0], out[1] + P["f"] * qv, out[2] - P["f"] * qu], 1)


def _model_step(U, courant, each=None):
    """One model step of every particle, each with its own number of scheme steps; each(U, p, dt) after each."""
    P = PHYS
    h = P["H"] + U[:, 0]
    c = (P["g"] * h).sqrt()
    a = torch.maximum(((U[:, 1] / h).abs() + c).amax((1, 2)) / P["dx"], ((U[:, 2] / h).abs() + c).amax((1, 2)) / P["dy"])
    n = torch.ceil(P["dt"] / (courant * 0.25 / a)).long().clamp(min=1)
    for k in n.unique().tolist():
        p = (n == k).nonzero()[:, 0]
        V, dt = U[p], P["dt"] / k
        for _ in range(k):
            V1 = V + dt * _rhs(V)
            V = 0.5 * (V + V1 + dt * _rhs(V1))
            if each:
                each(V, p, dt)
        U[p] = V
    return U


def _normals(seed, p, t, stream, n):
    """Philox4x32-10 (Salmon et al., SC'11) and Box-Muller: [len(p)][n]."""
    M = 0xFFFFFFFF
    nb = (n + 3) // 4
    z = torch.zeros((len(p), nb), dtype=torch.int64, device=DEV)
    c = [z + torch.arange(nb, device=DEV), z + torch.as_tensor(p, device=DEV)[:, None], z + t, z + stream]
    k0, k1 = seed & M, seed >> 32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & M) ^ c[1] ^ k0, b & M, ((a >> 32) & M) ^ c[3] ^ k1, a & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    out = []
    for a, b in ((c[0], c[1]), (c[2], c[3])):
        r = (-2 * torch.log((a.to(D) + 0.5) / 2 ** 32)).sqrt()
        th = 2 * math.pi * ((b.to(D) + 0.5) / 2 ** 32)
        out += [r * th.cos(), r * th.sin()]
    return torch.stack(out, 2).reshape(len(p), -1)[:, :n]


def _coarse(n, c):
    """Fine positions of the coarse points, periodic: (count, position of any index)."""
    nR = (n - 1 - c // 2) // c + 1
    return nR, lambda a: c // 2 + c * (a % nR) + a // nR * n


def _cubic(t):
    return [0.5 * (-t ** 3 + 2 * t ** 2 - t), 0.5 * (3 * t ** 3 - 5 * t ** 2 + 2), 0.5 * (-3 * t ** 3 + 4 * t ** 2 + t),
            0.5 * (t ** 3 - t ** 2)]


def _soar_w(d, c):
    L0 = 0.75 * c * PHYS["dx"]
    return PHYS["q0"] * (1 + d / L0) * np.exp(-d / L0)


def _interval(j, nR, pos, c):
    a = np.where(j < c // 2, -1, np.minimum((j - c // 2) // c, nR - 1))
    return a, pos(a), pos(a + 1)


class _Q:
    """Q^{1/2}: SOAR on the coarse grid, bicubic to the fine one, momentum in geostrophic balance."""

    def __init__(self, nx, ny, c):
        self.nRx, px = _coarse(nx, c)
        self.nRy, py = _coarse(ny, c)
        a, b = np.arange(self.nRx), np.arange(self.nRy)
        self.w = {}
        for db in range(-2, 3):
            for da in range(-2, 3):
                d = np.hypot((px(a + da) - px(a))[None] * PHYS["dx"], (py(b + db) - py(b))[:, None] * PHYS["dy"])
                self.w[da, db] = torch.as_tensor(_soar_w(d, c), device=DEV)
        self.A = [self._interp(nx, self.nRx, px, c), self._interp(ny, self.nRy, py, c)]

    @staticmethod
    def _interp(n, nR, pos, c):
        j = np.arange(n)
        a, x0, x1 = _interval(j, nR, pos, c)
        A = np.zeros((n, nR))
        for k, w in enumerate(_cubic((j - x0) / (x1 - x0))):
            np.add.at(A, (j, (a - 1 + k) % nR), w)
        return torch.as_tensor(A, device=DEV)

    def add(self, U, x):
        x = x.reshape(-1, self.nRy, self.nRx)
        f = sum(w * x.roll((-db, -da), (1, 2)) for (da, db), w in self.w.items())
        f = self.A[1] @ f @ self.A[0].T
        s = PHYS["g"] * PHYS["H"] / PHYS["f"]
        U[:, 0] += f
        U[:, 1] -= s / (2 * PHYS["dy"]) * (f.roll(-1, 1) - f.roll(1, 1))
        U[:, 2] += s / (2 * PHYS["dx"]) * (f.roll(-1, 2) - f.roll(1, 2))
        return U


def _stencil(c):
    """Q H^T of a unit hu and a unit hv observation around its cell: [2][3][2R+1][2R+1], R = 7 c."""
    P, n, R = PHYS, 21, 7 * c
    s = P["g"] * P["H"] / P["f"]
    o = np.arange(-R - 1, R + 2)
    b = o // c
    A = np.zeros((len(o), n))
    for k, w in enumerate(_cubic((o - b * c) / c)):
        A[np.arange(len(o)), 10 + b - 1 + k] += w
    K = np.zeros((2, 3, 2 * R + 1, 2 * R + 1))
    for comp in range(2):
        e = np.zeros((n, n))
        if comp == 0:
            e[11, 10], e[9, 10] = -s / (2 * c * P["dy"]), s / (2 * c * P["dy"])
        else:
            e[10, 11], e[10, 9] = s / (2 * c * P["dx"]), -s / (2 * c * P["dx"])
        for _ in range(2):
            e = sum(_soar_w(np.hypot(i * c * P["dx"], j * c * P["dy"]), c) * np.roll(e, (j, i), (0, 1))
                    for i in range(-2, 3) for j in range(-2, 3))
        f = A @ e @ A.T
        K[comp] = [f[1:-1, 1:-1], -s * (f[2:, 1:-1] - f[:-2, 1:-1]) / (2 * P["dy"]),
                   s * (f[1:-1, 2:] - f[1:-1, :-2]) / (2 * P["dx"])]
    return K


def _block_root(c):
    """Symmetric root of I - B^T (B B^T + R)^{-1} B, B = H Q^{1/2} on the 7 x 7 coarse points around an observation."""
    P = PHYS
    s = P["g"] * P["H"] / P["f"]
    my, mx = (v.ravel() for v in np.mgrid[-3:4, -3:4])

    def w(ax, ay):
        near = (abs(ax - mx) <= 2) & (abs(ay - my) <= 2)
        return near * _soar_w(np.hypot((ax - mx) * c * P["dx"], (ay - my) * c * P["dy"]), c)
    B = np.stack([-s / (2 * c * P["dy"]) * (w(0, 1) - w(0, -1)), s / (2 * c * P["dx"]) * (w(1, 0) - w(-1, 0))])
    lam, V = np.linalg.eigh(np.eye(49) - B.T @ np.linalg.solve(B @ B.T + SIGMA ** 2 * np.eye(2), B))
    return (V * np.sqrt(lam.clip(0))) @ V.T


def _alpha(gamma, cstar, N):
    """-N/gamma W0(-gamma/N exp(-gamma/N) exp(-c*/N)) through s = 1 + W0: -s - log(1 - s) = q."""
    x = gamma / N
    q = (x - 1 - torch.log1p(x - 1)) + cstar.clamp(min=0) / N
    lo, hi = torch.zeros_like(q), torch.ones_like(q)
    for _ in range(200):
        m = 0.5 * (lo + hi)
        low = -m - torch.log1p(-m) < q
        lo, hi = torch.where(low, m, lo), torch.where(low, hi, m)
    return torch.where(q > 0, 1 - 0.5 * (lo + hi), torch.ones_like(q)) / x


def _assimilate(U, nx, ny, xy, y, c, t, stream, scheme, dense):
    """The implicit equal-weights analysis of the ensemble U (changed in place); its diagnostics."""
    P, ne = PHYS, U.shape[0]
    Q, cells, R = _Q(nx, ny, c), _cells(xy, nx, ny), 7 * c
    K = torch.as_tensor(_stencil(c), device=DEV)
    cj, ck = (torch.as_tensor(cells[:, k].copy(), device=DEV) for k in (0, 1))
    s = (P["H"] + U[:, 0][:, ck, cj]) / P["H"]
    yt = torch.as_tensor(y, device=DEV)
    d = torch.stack([yt[:, 0] * s - U[:, 1][:, ck, cj], yt[:, 1] * s - U[:, 2][:, ck, cj]], 2).reshape(ne, -1)
    no = len(cells)
    ox, oy = (((q[:, None] - q[None] + n // 2) % n) - n // 2 for q, n in ((cj, nx), (ck, ny)))
    ox, oy = torch.where(2 * ox == -nx, -ox, ox), torch.where(2 * oy == -ny, -oy, oy)
    near = (ox.abs() <= R) & (oy.abs() <= R)
    if not dense:
        near &= torch.eye(no, dtype=torch.bool, device=DEV)
    A = torch.zeros((no, 2, no, 2), dtype=D, device=DEV)
    for a in range(2):
        for b in range(2):
            A[:, a, :, b] = near * K[b, 1 + a][oy.clamp(-R, R) + R, ox.clamp(-R, R) + R]
    A = A.reshape(2 * no, 2 * no)
    A = 0.5 * (A + A.T) + SIGMA ** 2 * torch.eye(2 * no, dtype=D, device=DEV)
    Sd = torch.cholesky_solve(d.T.contiguous(), torch.linalg.cholesky(A)).T
    phi = (d * Sd).sum(1)
    cc = phi + math.log(ne)
    NR, N = Q.nRx * Q.nRy, 3.0 * nx * ny
    xi, nt = (_normals(0x191001031, range(ne), t, stream + k, NR) for k in (1, 2))
    xx, nn, xn = (xi * xi).sum(1), (nt * nt).sum(1), (xi * nt).sum(1)
    gamma, zeta = xx * N / NR, nn * N / NR
    if scheme:
        target, beta = cc.max(), torch.zeros((), dtype=D, device=DEV)
        cstar = target - cc
    else:
        target = cc.mean()
        beta = ((target - cc) / zeta + 1).min()
        cstar = target - cc - (beta - 1) * zeta
    alpha = _alpha(gamma, cstar, N)
    nlw = (alpha - 1) * gamma - N * torch.log(alpha) + cc + (0 if scheme else (beta - 1) * zeta)
    a = xn / xx
    nu = (nn / (nn - a * xn)).sqrt()[:, None] * (nt - a[:, None] * xi)
    r = beta.clamp(min=0).sqrt() * nu + alpha.sqrt()[:, None] * xi
    M = torch.as_tensor(_block_root(c), device=DEV)
    near_pt = []
    for q, n, nR in ((cells[:, 0], nx, Q.nRx), (cells[:, 1], ny, Q.nRy)):
        ai, x0, x1 = _interval(q, nR, _coarse(n, c)[1], c)
        near_pt.append(np.where(q - x0 <= x1 - q, ai, ai + 1))
    o7 = np.arange(-3, 4)
    idx = torch.as_tensor((((near_pt[1][:, None] + o7) % Q.nRy * Q.nRx)[:, :, None]
                           + ((near_pt[0][:, None] + o7) % Q.nRx)[:, None, :]).reshape(no, 49), device=DEV)
    for l in range(no):
        r[:, idx[l]] = r[:, idx[l]] @ M.T
    off = torch.arange(-R, R + 1, device=DEV)
    for l in range(no):
        rows, cols = (ck[l] + off) % ny, (cj[l] + off) % nx
        U[:, :, rows[:, None], cols] += torch.einsum("pk,kfyx->pfyx", Sd[:, 2 * l:2 * l + 2], K)
    for p0 in range(0, ne, 32):
        Q.add(U[p0:p0 + 32], r[p0:p0 + 32])
    return {"phi": phi, "c": cc, "gamma": gamma, "zeta": zeta, "alpha": alpha, "neglogw": nlw,
            "cbar": float(cc.mean()), "beta": float(beta), "w_target": float(target)}


def _advance(U, nx, ny, c, courant, t, stream, errs, p0=0, each=None):
    """Model steps of the particles p0.. (errs: whether each is followed by its model error)."""
    Q = _Q(nx, ny, c)
    for k, err in enumerate(errs):
        U = _model_step(U, courant, each)
        if err:
            Q.add(U, _normals(0x191001031, range(p0, p0 + len(U)), t + k, stream, Q.nRx * Q.nRy))
    return U


def _chunked(U, nx, ny, *args):
    step = max(1, 8_000_000 // (nx * ny))
    return torch.cat([_advance(U[p:p + step].to(D), nx, ny, *args, p0=p) for p in range(0, len(U), step)])


def _net64(flat, x, depth=6):
    off = 0
    for l in range(depth):
        ci, co = (16 if l == 0 else 64), (16 if l == depth - 1 else 64)
        W = flat[off:off + 9 * ci * co].view(3, 3, co, ci).permute(2, 3, 0, 1)
        off += 9 * ci * co
        b = flat[off:off + co]
        off += co
        if l == 0:
            W = W[:, :3]
        if l == depth - 1:
            W, b = W[:3], b[:3]
        x = F.conv2d(F.pad(x, (1, 1, 1, 1), mode="circular"), W, b)
        if l < depth - 1:
            x = F.silu(x)
    return x


def _scale(v):
    return torch.tensor(v, dtype=D, device=DEV)[:, None, None]


def _apply64(U, flat):
    step = max(1, 500_000 // U[0, 0].numel())
    return torch.cat([U[p:p + step].to(D) + _scale(OUT_SCALE) * _net64(flat, _scale(IN_SCALE) * U[p:p + step].to(D))
                      for p in range(0, len(U), step)])


def _drift64(U, xy, dt, scale=1.0):
    """Drifter velocities (times scale dt) in their cells, added to xy [n][nd][2] in place."""
    n, _, ny, nx = U.shape
    c = torch.floor(xy / torch.tensor([PHYS["dx"], PHYS["dy"]], dtype=D, device=DEV)).long()
    j, k = c[..., 0] % nx, c[..., 1] % ny
    p = torch.arange(n, device=DEV)[:, None]
    h = PHYS["H"] + U[p, 0, k, j]
    return scale * dt * torch.stack([U[p, 1, k, j] / h, U[p, 2, k, j] / h], -1)


def exact(case, seed):
    kind = case["kind"]
    t, cyc = _counters(seed)
    if work(case)["flops"] > (6e12 if kind in ("apply", "grad", "drift") else 2.5e12):
        return None     # over the time that is worth waiting for
    if kind == "batch":
        diag, states = [], []
        for i, ((nx, ny, _, _), (U, xy, y)) in enumerate(zip(_problems(case), _batch_inputs(case, seed))):
            U = _chunked(U, nx, ny, case["c_omega"], case["courant"], t, 16 * i, [1, 1, 1, 1, 0])
            d = _assimilate(U, nx, ny, xy, y, case["c_omega"], cyc, 16 * i, 0, 1)
            diag.append([d["w_target"], d["beta"]])
            states.append(U.reshape(-1))
        return {"diag": np.array(diag), "state": torch.cat(states)}
    if kind == "grad":
        X, Y = (torch.as_tensor(v, device=DEV).to(D) for v in _pairs(case, seed))
        flat = torch.as_tensor(_weights(seed), device=DEV).to(D).requires_grad_()
        loss = ((_net64(flat, _scale(IN_SCALE) * X) - (Y - X) / _scale(OUT_SCALE)) ** 2).mean()
        loss.backward()
        return {"loss": float(loss.detach()), "grad": flat.grad.detach()}
    nx, ny = case["nx"], case["ny"]
    U = _state(nx, ny, case["n"] if kind == "apply" else case["ne"], seed)
    if kind == "apply":
        return _apply64(U, torch.as_tensor(_weights(seed), device=DEV).to(D))
    if kind == "forecast":
        return _chunked(U, nx, ny, case["c_omega"], case["courant"], t, 0,
                        [1] * case["steps_err"] + [0] * case["steps_plain"])
    if kind == "analysis":
        moor = case["obs"] == "mooring"
        xy = _moorings(nx, ny, case["n_obs"], case["spacing"]) if moor else _drifters(nx, ny, case["n_obs"], seed)
        U = U.to(D)
        d = _assimilate(U, nx, ny, xy, _observe(xy, nx, ny, seed, 0), case["c_omega"], cyc, 0, case["scheme"],
                        case["dense"])
        return {"state": U, "diag": d}
    U = U.to(D)
    pos = torch.as_tensor(_drifters(nx, ny, case["nd"], seed), device=DEV).expand(len(U), -1, -1).clone()
    traj = [pos.clone()]
    flat = torch.as_tensor(_weights(seed), device=DEV).to(D)
    Q = _Q(nx, ny, 3)

    def each(V, p, dt):
        pos[p] += _drift64(V, pos[p], dt)
    for o in range(int(case["seconds"] / case["every"])):
        if case["surrogate"]:
            V = _apply64(U, flat)
            pos += _drift64(U, pos, 600.0, 0.5) + _drift64(V, pos, 600.0, 0.5)
            U = V
            for k in range(10):
                Q.add(U, _normals(0x191001031, range(len(U)), t + 10 * o + k, 0, Q.nRx * Q.nRy))
        else:
            U = _advance(U, nx, ny, 3, 0.45, t + 10 * o, 0, [1] * 10, each=each)
        traj.append(pos.clone())
    return {"traj": torch.stack(traj), "state": U}
