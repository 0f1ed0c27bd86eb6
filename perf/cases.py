"""Performance cases: the runs a user of the history engine makes, through its
Python entry points (engine.Scene and engine.TransportFn).

A plain case is one estimate: reset the tallies, run the histories, read mean
and standard error of every tally.  A gradient case is one step of a fit:
TransportFn forward (set the instance parameters, run with the score-function
accumulators, means of every bin) and backward.  Scenes, their materials and
the launch chosen at a scene's first run are what a program keeps between
estimates; prepare() makes them."""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_2304_06226_gb300.engine import Scene, TransportFn

# Lane operations of the method per history (random numbers, cross sections,
# flight, next boundary, crossing, collision), from the event, collision and
# crossing counts of each workload at its default parameters.
OPS_PER_HISTORY = {"slab": 1016, "powder": 1194, "guide": 395, "total_scattering": 850, "chopper": 334,
                   "moderator": 430, "imaging": 826, "batched": 2935}


def listed():
    return [
        # a check run of a scene being set up: few histories, FP64, answer wanted at once
        {"name": "slab_f64_check", "workload": "slab", "histories": 20_000, "precision": "f64", "g": 3.0},
        # the biasing study of a slab, FP64
        {"name": "slab_f64", "workload": "slab", "histories": 1_000_000, "precision": "f64", "g": 3.0},
        # a first look at a diffractogram
        {"name": "powder_f32_look", "workload": "powder", "histories": 99_991, "precision": "f32", "g": 1.0,
         "bins": 3600},
        # the diffractometer at full statistics (the benchmark's size)
        {"name": "powder_f32", "workload": "powder", "histories": 100_000_000, "precision": "f32", "g": 1.0,
         "bins": 3600},
        # the same instrument in FP64, to validate the FP32 one
        {"name": "powder_f64", "workload": "powder", "histories": 2_000_000, "precision": "f64", "g": 1.0,
         "bins": 3600},
        # supermirror guide at full statistics
        {"name": "guide_f32", "workload": "guide", "histories": 100_000_000, "precision": "f32", "m": 2.0,
         "length": 2000.0},
        # scattering-order study, default size
        {"name": "total_scattering_f32", "workload": "total_scattering", "histories": 10_000_000,
         "precision": "f32", "g": 1.0, "radius": 1.2, "lam": 1.0},
        # time-of-flight chopper study, default size
        {"name": "chopper_f32", "workload": "chopper", "histories": 10_000_000, "precision": "f32", "bins": 1000},
        # a moderator gun looked at through a slit, default size
        {"name": "moderator_f32", "workload": "moderator", "histories": 1_000_000, "precision": "f32",
         "temperature": 293.15},
        # a radiograph of 1000 primitives with biased absorption
        {"name": "imaging_f32", "workload": "imaging", "histories": 20_000_000, "precision": "f32", "prims": 1000,
         "bins": 512, "abs_bias": 0.1, "grad": False},
        # one step of a density fit to a radiograph
        {"name": "imaging_grad_f32", "workload": "imaging", "histories": 20_000_000, "precision": "f32",
         "prims": 1000, "bins": 512, "abs_bias": 0.0, "grad": True},
        # one step of a fit of radius, scale and density of many samples at once
        {"name": "batched_grad_f32", "workload": "batched", "histories": 120_000_000, "precision": "f32",
         "instances": 256, "bins": 3600, "grad": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["slab", "powder", "powder", "guide", "total_scattering", "chopper", "moderator", "imaging",
                       "imaging", "batched"])
    g = rng.choice([1.0, 1.0, round(rng.uniform(0.5, 4.0), 2)])
    if kind == "slab":
        f64 = rng.random() < 0.7
        return {"workload": kind, "histories": _log_int(rng, 1e4, 4e6 if f64 else 1e8),
                "precision": "f64" if f64 else "f32", "g": rng.choice([1.0, 3.0, round(rng.uniform(0.5, 4.0), 2)])}
    if kind == "powder":
        f64 = rng.random() < 0.3
        return {"workload": kind, "histories": _log_int(rng, 1e4, 1e7 if f64 else 1e8),
                "precision": "f64" if f64 else "f32", "g": g, "bins": _log_int(rng, 360, 7200)}
    if kind == "guide":
        return {"workload": kind, "histories": _log_int(rng, 1e5, 1e8), "precision": "f32",
                "m": round(rng.uniform(1.0, 4.0), 2), "length": round(rng.uniform(500.0, 4000.0), 1)}
    if kind == "total_scattering":
        return {"workload": kind, "histories": _log_int(rng, 1e5, 1e8), "precision": "f32", "g": g,
                "radius": round(rng.uniform(0.3, 2.0), 3), "lam": round(rng.uniform(0.8, 3.0), 3)}
    if kind == "chopper":
        return {"workload": kind, "histories": _log_int(rng, 1e5, 1e8), "precision": "f32",
                "bins": _log_int(rng, 100, 2500)}
    if kind == "moderator":
        return {"workload": kind, "histories": _log_int(rng, 1e5, 1e8), "precision": "f32",
                "temperature": rng.choice([0.0, round(rng.uniform(25.0, 600.0), 2)])}
    if kind == "imaging":
        return {"workload": kind, "histories": _log_int(rng, 1e5, 5e7), "precision": "f32",
                "prims": _log_int(rng, 100, 1200), "bins": _log_int(rng, 64, 512),
                "abs_bias": rng.choice([0.0, 0.1, round(rng.uniform(0.1, 1.0), 2)]), "grad": rng.random() < 0.5}
    return {"workload": kind, "histories": _log_int(rng, 1e6, 1.2e8), "precision": "f32",
            "instances": _log_int(rng, 4, 256), "bins": _log_int(rng, 360, 3600), "grad": True}


def _describe(case, seed):
    n, prec, kind = case["histories"], case["precision"], case["workload"]
    if kind == "slab":
        d = W.slab(g=case["g"], n_histories=n, precision=prec)
    elif kind == "powder":
        d = W.powder(n_histories=n, precision=prec, g=(case["g"],) * 3, nbins=case["bins"])
    elif kind == "guide":
        d = W.guide(n_histories=n, precision=prec, m=case["m"], length=case["length"])
    elif kind == "total_scattering":
        d = W.total_scattering(g=case["g"], n_histories=n, precision=prec, radius=case["radius"], lam=case["lam"])
    elif kind == "chopper":
        d = W.chopper(n_histories=n, precision=prec, tof_bins=case["bins"])
    elif kind == "moderator":
        d = W.moderator_test(n_histories=n, precision=prec, temperature=case["temperature"] or None)
    elif kind == "imaging":
        d = W.imaging(n_histories=n, precision=prec, n_prims=case["prims"], psd_bins=case["bins"], seed=seed,
                      abs_bias=case["abs_bias"] or None)
    else:
        # uneven counts (a factor of 100 between instances), scaled to the wanted total
        d = W.batched(n_instances=case["instances"], seed=seed, precision=prec, nbins=case["bins"])
        c = d["instances"]["counts"].astype(np.float64)
        d["instances"]["counts"] = np.maximum(1, np.rint(c * (n / c.sum()))).astype(np.int64)
    d["seed"] = int(seed)
    return d


def prepare(case, seed):
    desc = _describe(case, seed)
    scene = Scene(desc)
    state = {"scene": scene, "names": [t["name"] for t in desc["tallies"]], "params": None}
    if case.get("grad"):
        state["params"] = torch.tensor(desc["instances"]["params"], dtype=torch.float64, device="cuda",
                                       requires_grad=True)
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        # gradient of a loss with respect to every bin
        state["weights"] = torch.rand(scene.n_inst, scene.total_bins, dtype=torch.float64, device="cuda",
                                      generator=gen)
    scene.run(want_grad=bool(case.get("grad")))   # a scene's first run picks its launch
    scene.reset()
    return state


def run(state):
    scene = state["scene"]
    if state["params"] is not None:
        means = TransportFn.apply(state["params"], scene)
        (grad,) = torch.autograd.grad(means, state["params"], state["weights"])
        return {"means": means.detach(), "grad": grad}
    scene.reset()
    scene.run()
    out = {}
    for t, name in enumerate(state["names"]):
        out[name + "_mean"], out[name + "_err"] = scene.tally(t)
    return out


def work(case):
    bins = {"slab": 182, "guide": 10_000, "total_scattering": 808, "moderator": 1660}.get(case["workload"])
    if bins is None:
        b = case["bins"]
        bins = {"powder": b, "batched": b, "chopper": 2 * b + 1, "imaging": b * b}[case["workload"]]
    bins *= case.get("instances", 1)
    return {"bytes": 16.0 * bins, "flops": float(OPS_PER_HISTORY[case["workload"]]) * case["histories"]}


# ---------------------------------------------------------------------------
# The same histories in 64-bit torch, for the scenes whose transport is short
# ---------------------------------------------------------------------------
_MASK = 0xFFFFFFFF


def _philox(event, sub, hid, seed):
    """Philox4x32-10 blocks of counter (event, sub, hid, 0); int64 tensors in [0, 2^32)."""
    zero = torch.zeros_like(hid)
    c = [zero + event, zero + sub, hid, zero]
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK

    def mul(a, b):
        p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
        return (p1 + (p0 >> 16)) >> 16, (p0 + ((p1 & 0xFFFF) << 16)) & _MASK

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c


def _uniform(a, precision):
    if precision == "f64":
        return (a.double() + 0.5) * 2.0 ** -32
    return ((a >> 8).double() + 0.5) * 2.0 ** -24


def _bins(x, lo, hi, n):
    b = torch.floor((x - lo) * (n / (hi - lo))).long().clamp_(max=n - 1)
    return torch.where((x >= lo) & (x < hi), b, torch.full_like(b, -1))


class _Tally:
    def __init__(self, nbins, device):
        self.sums = torch.zeros(2, nbins, dtype=torch.float64, device=device)

    def add(self, b, w):
        keep = b >= 0
        self.sums[0].index_add_(0, b[keep], w[keep])
        self.sums[1].index_add_(0, b[keep], w[keep] ** 2)

    def result(self, n):
        mean = self.sums[0] / n
        return mean, torch.sqrt(torch.clamp(self.sums[1] / n - mean * mean, min=0.0) / (n - 1.0))


_KT_MEV, _E_MEV, _H_OVER_M = 0.08617333, 81.80420, 395603.4012


def _moderator_rays(desc, hid, precision):
    """Position, direction and wavelength of the moderator guns."""
    s = desc["source"]
    a = [_uniform(v, precision) for v in _philox(0, 0, hid, desc["seed"])]
    b = [_uniform(v, precision) for v in _philox(0, 1, hid, desc["seed"])]
    x = [s["centre"][i] + s["half"][i] * (2 * a[i] - 1) for i in (0, 1)] + [torch.full_like(a[0], s["centre"][2])]
    if s["temperature"] > 0:
        e = _KT_MEV * s["temperature"] * (-torch.log(a[2]) - torch.log(a[3]) * torch.cos(0.5 * math.pi * b[3]) ** 2)
        lam = torch.sqrt(_E_MEV / e)
    else:
        lam = s["lambda"][0] + (s["lambda"][1] - s["lambda"][0]) * a[2]
    d = [s["centre"][i] + s["slit_half"][i] * (2 * b[1 + i] - 1) - x[i] for i in (0, 1)]
    d.append(s["slit_z"] - x[2])
    r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    return x, [v / r for v in d], lam


def _exact_moderator(desc, hid, precision, device):
    psd, spectrum = desc["tallies"]
    x, u, lam = _moderator_rays(desc, hid, precision)
    p = desc["prims"][0]
    t = (p["centre"][2] - p["params"][2] - x[2]) / u[2]
    q = [x[i] + t * u[i] for i in (0, 1)]
    one = torch.ones_like(t)
    a, b = _Tally(psd["bins"][0] * psd["bins"][1], device), _Tally(spectrum["bins"][0], device)
    bx, by = (_bins(q[i], psd["lo"][i], psd["hi"][i], psd["bins"][i]) for i in (0, 1))
    a.add(torch.where((bx >= 0) & (by >= 0), bx * psd["bins"][1] + by, torch.full_like(bx, -1)), one)
    bl = _bins(lam, spectrum["lo"][0], spectrum["hi"][0], spectrum["bins"][0])
    b.add(torch.where(_bins(q[0], spectrum["lo"][1], spectrum["hi"][1], 1) >= 0, bl, torch.full_like(bl, -1)), one)
    return [a, b]


def _exact_chopper(desc, hid, precision, device):
    before, after, _ = desc["tallies"]
    x, u, lam = _moderator_rays(desc, hid, precision)
    p = desc["prims"][0]
    c = p["chopper"]
    t = [(p["centre"][2] + s * p["params"][2] - x[2]) / u[2] for s in (-1, 1)]   # front and rear of the disk
    q = [x[i] + t[0] * u[i] - p["centre"][i] for i in (0, 1)]
    psi = (torch.atan2(q[1], q[0]) - c["phase"]) * (c["n"] / (2 * math.pi)) - c["n"] * c["freq"] * t[0] * lam / _H_OVER_M
    is_open = ((psi - torch.round(psi)).abs() <= c["n"] * c["theta0"] / (4 * math.pi)) & \
        (q[0] ** 2 + q[1] ** 2 >= c["r_black"] ** 2)
    one = torch.ones_like(psi)
    tallies = [_Tally(before["bins"][0], device), _Tally(after["bins"][0], device), _Tally(1, device)]
    tallies[0].add(_bins(t[0] * lam / _H_OVER_M, before["lo"][0], before["hi"][0], before["bins"][0]), one)
    tallies[1].add(_bins(t[1] * lam / _H_OVER_M, after["lo"][0], after["hi"][0], after["bins"][0])[is_open], one[is_open])
    tallies[2].add(torch.zeros_like(hid)[is_open], one[is_open])
    return tallies


def _exact_slab(desc, hid, precision, device):
    box, world, mat = desc["prims"][0], desc["world"], desc["materials"][0]
    g = [float(v) for v in desc["bias"][0]]
    lam = desc["source"]["lambda"][0]
    sig = (mat["sigma_abs_ref"] * lam / 1.8, mat["sigma_inc"])
    sig_t, sig_g = sum(sig), g[0] * sig[0] + g[1] * sig[1]
    nudge = 1e-9 if precision == "f64" else 1e-5
    half = torch.tensor(box["params"], dtype=torch.float64, device=device)
    centre = torch.tensor(box["centre"], dtype=torch.float64, device=device)
    tallies = [_Tally(1, device), _Tally(1, device), _Tally(desc["tallies"][2]["bins"][0], device)]

    def step_over(x, u):
        return x + nudge * x.abs().amax(dim=1, keepdim=True).clamp(min=1.0) * u

    # event 1: from the source to the slab's front face
    n = hid.numel()
    x = torch.zeros(n, 3, dtype=torch.float64, device=device)
    u = torch.zeros_like(x)
    u[:, 2] = 1.0
    x[:, 2] = box["centre"][2] - box["params"][2]
    x = step_over(x, u)
    w = torch.ones(n, dtype=torch.float64, device=device)
    nscat = torch.zeros(n, dtype=torch.int64, device=device)
    for k in range(2, desc["event_cap"] + 1):
        if not hid.numel():
            break
        r = [_uniform(v, precision) for v in _philox(k, 0, hid, desc["seed"])]
        length = -torch.log(r[0]) / sig_g
        t = torch.where(u > 0, (half - (x - centre)) / u, torch.where(u < 0, (-half - (x - centre)) / u, math.inf))
        db, axis = t.min(dim=1)
        out = length >= db
        d = torch.where(out, db, length)
        x = x + d[:, None] * u
        w = w * torch.exp((sig_g - sig_t) * d)
        # leaving: the rear-face counts, then the flight to the world's sphere
        rear = out & (axis == 2) & (u[:, 2] > 0)
        zero = torch.zeros_like(hid)
        tallies[0].add(zero[rear & (nscat == 0)], w[rear & (nscat == 0)])
        tallies[1].add(zero[rear], w[rear])
        xe, ue = step_over(x[out], u[out]), u[out]
        v = xe - torch.tensor(world["centre"], dtype=torch.float64, device=device)
        vu = (v * ue).sum(1)
        p = v + (-vu + torch.sqrt(vu * vu - (v * v).sum(1) + world["params"][1] ** 2))[:, None] * ue
        theta = torch.atan2(torch.sqrt(p[:, 0] ** 2 + p[:, 1] ** 2), p[:, 2])
        tallies[2].add(_bins(theta, 0.0, math.pi, tallies[2].sums.shape[1]), w[out])
        # collisions: absorbed, or a new isotropic direction
        stay = ~out & ~(r[1] * sig_g < g[0] * sig[0])
        mu, phi = 2 * r[2] - 1, 2 * math.pi * r[3]
        st = torch.sqrt(torch.clamp(1 - mu * mu, min=0.0))
        u = torch.stack([st * torch.cos(phi), st * torch.sin(phi), mu], dim=1)[stay]
        x, w, nscat, hid = x[stay], w[stay] / g[1], nscat[stay] + 1, hid[stay]
    return tallies


_EXACT = {"moderator": _exact_moderator, "chopper": _exact_chopper, "slab": _exact_slab}


def exact(case, seed):
    follow = _EXACT.get(case["workload"])
    if follow is None:   # a whole instrument, history by history: minutes in plain torch
        return None
    desc = _describe(case, seed)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    n, total = case["histories"], None
    for lo in range(0, n, 4_000_000):
        hid = torch.arange(lo, min(n, lo + 4_000_000), dtype=torch.int64, device=device)
        part = follow(desc, hid, case["precision"], device)
        if total is None:
            total = part
        else:
            for a, b in zip(total, part):
                a.sums += b.sums
    out = {}
    for t, tally in zip(desc["tallies"], total):
        out[t["name"] + "_mean"], out[t["name"] + "_err"] = tally.result(float(n))
    return out
