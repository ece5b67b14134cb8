"""The performance cases of the track fit: what a program that uses this
library has it do, through the public entry points, over the range of sizes
and options it is used with.

A case is a dict of plain values; its "entry" says which call it makes:

  fit       Fitter.run (fit_propagate_update): the fused fit of a call's events
  plan      fit_plan_run: uneven events of both modes in one persistent launch
  noalloc   fit_propagate_update_noalloc with per-event counters
  f64       fit_propagate_update_f64
  find      fit_find_tracks: the best of several candidate hits per layer
  adjoint   fit.chi2 and its gradient through autograd
  seeded    Fitter.run on a handle with the learned path-length seed attached
  train     fit_mlp_set_params, fit_mlp_train, fit_mlp_get_params
  host      fit_propagate_update_host on page-locked host arrays

Tracks, hits, candidate hits and training samples follow the distributions of
paper_2409_09228_gb300/inputs.py, drawn on the GPU so that preparing a case is
quick.  One thing differs: the azimuth is drawn uniformly where a track ends,
0.02 rad away from the jump of phi at +-pi (20 times the spread of a fitted
azimuth), so that two results can be compared as numbers.

exact() is the same fit in plain torch, in 64 bits: full 6x6 matrices, the
closed-form crossing polished by Newton's method, gradients by autograd.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2409_09228_gb300 import fit, inputs

P2R, P2Z = inputs.MODE_R, inputs.MODE_Z
KA, B_FIELD = 0.00299792458, float(np.float32(3.8))
SIGMA_RPHI, SIGMA_2 = 0.01, 0.1  # hit errors [cm]: azimuthal; along z (p2r) or radial (p2z)
SIGMA0 = (0.01, 0.01, 0.1, 0.05, 0.01, 0.01)  # of the start state, that of w relative
SIGMA_STATE = (0.01, 0.01, 0.1, 0.01, 1e-3, 1e-3)  # of a filtered state (training samples)
GATE = 30.0
MLP_SHAPES = ((64, 8), (64,), (64, 64), (64,), (1, 64), (1,))
PAIRS = [(i, j) for i in range(6) for j in range(i + 1)]


# ---- the cases --------------------------------------------------------------------------


def listed():
    return [
        # The smallest call: one p2r event of 1024 tracks, as an online program
        # has it, where the launch and the layers' latency count.
        dict(name="fit_event", entry="fit", sizes="even", nevt=1, ntrk=1024, modes="r", nlayer=20),
        # Two ordinary events, one of each detector part, odd track counts.
        dict(name="fit_pair", entry="fit", sizes="even", nevt=2, ntrk=8191, modes="rz", nlayer=20),
        # Bulk reprocessing: 100 events of 9600 tracks in either part, one call.
        dict(name="fit_bulk", entry="fit", sizes="even", nevt=200, ntrk=9600, modes="rrzz",
             nlayer=20),
        # A recorded stream: uneven events, barrel and endcap in random order.
        dict(name="fit_uneven", entry="fit", sizes="uneven", nevt=500, ntrk=2000, modes="mixed",
             nlayer=20),
        # The same kind of stream with its structure fixed in a plan, replayed.
        dict(name="plan_uneven", entry="plan", sizes="uneven", nevt=2000, ntrk=2000,
             modes="mixed", nlayer=20, layout=0),
        # A trigger farm's call: small mixed events, no allocation, counters per event.
        dict(name="noalloc_trigger", entry="noalloc", sizes="uneven", nevt=32, ntrk=500,
             modes="mixed", nlayer=20),
        # A reference fit in double.
        dict(name="f64_events", entry="f64", sizes="even", nevt=10, ntrk=9600, modes="rz",
             nlayer=20),
        # Pattern recognition: four candidate hits per layer.
        dict(name="find_events", entry="find", sizes="even", nevt=50, ntrk=9600, modes="rrzz",
             nlayer=20, ncand=4),
        # Alignment: chi2 and its gradient with respect to hits and start states.
        dict(name="adjoint", entry="adjoint", sizes="even", nevt=1, ntrk=100000, modes="r",
             nlayer=20),
        # The fit with the learned path-length seed.
        dict(name="seeded_fit", entry="seeded", sizes="even", nevt=1, ntrk=250001, modes="r",
             nlayer=20),
        # Training that seed: one pass over the samples in batches of 4096.
        dict(name="seed_training", entry="train", n=262144, batch=4096, epochs=1),
        # Events that arrive in page-locked host memory.
        dict(name="host_events", entry="host", sizes="even", nevt=10, ntrk=9600, modes="rrzz",
             nlayer=20),
    ]


# The most track-layers (tracks x layers; for "train", samples) a drawn case of
# an entry has, and its least tracks.
DRAWN = {"fit": (4e7, 200), "plan": (4e7, 2000), "noalloc": (4e6, 200), "f64": (4e6, 500),
         "find": (8e6, 500), "adjoint": (2e6, 300), "seeded": (5e6, 1000), "train": (2.6e5, 8192),
         "host": (4e6, 2000)}


def draw(rng):
    entry = rng.choice(["fit", "fit", "fit"] + [e for e in DRAWN if e != "fit"])
    most, least = DRAWN[entry]
    log = lambda lo, hi: int(math.exp(rng.uniform(math.log(lo), math.log(hi))))  # noqa: E731
    if entry == "train":
        n = log(least, most)
        return dict(entry=entry, n=n, batch=min(n, rng.choice([1024, 2048, 4096, 8192])),
                    epochs=rng.choice([1, 2]))
    nlayer = rng.choice([10, 13, 20, 20, 20, 27, 40])
    tracks = log(least, most / nlayer)
    if entry in ("adjoint", "seeded"):
        modes = rng.choice(["r", "r", "z"]) if entry == "adjoint" else "r"
    else:
        modes = rng.choice(["r", "z", "rz", "rrzz", "mixed", "mixed"])
    nevt = min(log(1, 600), max(1, tracks // 60))
    if entry == "noalloc":
        nevt = min(nevt, 128)
    case = dict(entry=entry, sizes=rng.choice(["even", "uneven"]), nevt=nevt,
                ntrk=max(1, tracks // nevt), modes=modes, nlayer=nlayer)
    if entry == "plan":
        case["layout"] = rng.choice([0, 1])
    if entry == "find":
        case["ncand"] = rng.choice([1, 2, 3, 4, 4, 6])
        case["ntrk"] = max(1, case["ntrk"] // case["ncand"])
    return case


def events(case, seed):
    """Track counts and modes of the case's events (numpy int64 and int32)."""
    nevt, ntrk, modes = case["nevt"], case["ntrk"], case["modes"]
    if case["sizes"] == "even":
        nt = np.full(nevt, ntrk, np.int64)
    else:  # log-normal as inputs.uneven_event_sizes, around ntrk / e^(1/2), total kept
        g = np.random.Generator(np.random.Philox(key=1000003))
        x = np.clip(np.exp(g.standard_normal(nevt)), 0.025, 10.0)
        nt = np.maximum(1, np.rint(x * (ntrk / x.mean()))).astype(np.int64)
    if modes == "mixed":
        g = np.random.Generator(np.random.Philox(key=1000033))
        md = np.where(g.random(nevt) < 0.5, P2R, P2Z)
    else:  # a run of events for each letter, in order
        md = np.array([P2R if c == "r" else P2Z for c in modes])
        md = md[np.arange(nevt) * len(md) // nevt] if nevt >= len(md) else md[:nevt]
    return nt, md.astype(np.int32)


def work(case):
    if case["entry"] == "train":
        n = (case["n"] // case["batch"]) * case["batch"] * case["epochs"]
        return {"bytes": 36.0 * case["n"], "flops": 6.0 * 4801 * n}
    nt, md = events(case, 0)
    nr, nz = int(nt[md == P2R].sum()), int(nt[md == P2Z].sum())
    nl, size = case["nlayer"], 8 if case["entry"] == "f64" else 4
    rows = 5 * nz + 9 * nr  # hit components that the update reads
    state = (27 * 2 + 1) * size + 2 * 4 + 1
    flops = nl * (580.0 * nz + 650.0 * nr)
    if case["entry"] == "find":  # a trial of a candidate is about 40 operations
        nbytes = nl * (case["ncand"] * rows * size + (nr + nz)) + state * (nr + nz)
        flops += nl * 40.0 * (case["ncand"] - 1) * (nr + nz)
    elif case["entry"] == "adjoint":  # hits read; gradients of the hits and the start state
        nbytes = nl * (rows + 3 * (nr + nz)) * size + (28 + 28 + 28) * size * (nr + nz)
        flops *= 3.0
    else:
        nbytes = nl * rows * size + state * (nr + nz)
    if case["entry"] == "seeded":  # the network before every layer
        flops += nl * 2.0 * 4801 * nr
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- inputs -------------------------------------------------------------------------------


def surfaces(mode, nlayer):
    lo, hi = (4.0, 110.0) if mode == P2R else (10.0, 270.0)
    return np.linspace(lo, hi, nlayer).astype(np.float32)


class Tracks:
    """The truth of n tracks on nlayer surfaces (float64 on the GPU), mode[t]
    the mode of track t, and the draws that smear it."""

    def __init__(self, mode, nlayer, seed):
        dev = mode.device
        self.g = torch.Generator(dev).manual_seed(int(seed))
        self.mode, self.n = mode, mode.shape[0]
        self.isr = mode == P2R
        self.surf = [torch.from_numpy(surfaces(m, nlayer).astype(np.float64)).to(dev)
                     for m in (P2R, P2Z)]
        eta = self.uniform(-1.0, 1.0)
        self.theta = 2.0 * torch.atan(torch.exp(-torch.where(self.isr, eta, 2.0 + 0.5 * eta)))
        # pT ~ U[0.5, 10] GeV; p2r tracks reach the last cylinder at 0.9 of its limit at most
        lo = torch.where(self.isr, KA * B_FIELD * 110.0 / 1.8, 0.5)
        self.pt = lo + (10.0 - lo) * self.uniform(0.0, 1.0)
        self.q = torch.where(self.uniform(0.0, 1.0) < 0.5, -1.0, 1.0)
        self.rho = self.pt / (KA * B_FIELD)
        self.phi0 = self.uniform(-math.pi + 0.02, math.pi - 0.02) + self.q * self.turn(nlayer - 1)

    def uniform(self, lo, hi):
        return lo + (hi - lo) * torch.rand(self.n, generator=self.g, device=self.mode.device,
                                           dtype=torch.float64)

    def normal(self):
        return torch.randn(self.n, generator=self.g, device=self.mode.device, dtype=torch.float64)

    def at(self, layer):
        return torch.where(self.isr, self.surf[0][layer], self.surf[1][layer])

    def turn(self, layer):
        """How far the direction has turned at a surface."""
        s = self.at(layer)
        half_r = torch.asin(torch.clamp(s / (2.0 * self.rho), max=1.0))
        return torch.where(self.isr, 2.0 * half_r, s * torch.tan(self.theta) / self.rho)

    def crossing(self, layer):
        """(radius, azimuth, z) of the truth on a surface."""
        s, turn = self.at(layer), self.turn(layer)
        r = torch.where(self.isr, s, 2.0 * self.rho * torch.sin(0.5 * turn))
        z = torch.where(self.isr, self.rho * turn / torch.tan(self.theta), s)
        return r, self.phi0 - 0.5 * self.q * turn, z

    def hit(self, layer, spread=1.0):
        """A hit smeared by `spread` times its errors: (position 3, covariance 6)."""
        r, phi, z = self.crossing(layer)
        return self.near(r, phi, z, spread * self.normal(), spread * self.normal())

    def near(self, r, phi, z, n1, n2):
        phi = phi + n1 * SIGMA_RPHI / r
        r = torch.where(self.isr, r, r + n2 * SIGMA_2)
        z = torch.where(self.isr, z + n2 * SIGMA_2, z)
        c, s = torch.cos(phi), torch.sin(phi)
        a, b = SIGMA_RPHI ** 2, SIGMA_2 ** 2
        br = torch.where(self.isr, 0.0, b)  # p2z: the second error is radial
        zero = torch.zeros_like(c)
        cov = (a * s * s + br * c * c, (br - a) * s * c, a * c * c + br * s * s, zero, zero, b - br)
        return (r * c, r * s, z), cov

    def start(self):
        """The smeared start state: par (6, n) and the diagonal of its covariance."""
        w = 1.0 / self.pt
        zero = torch.zeros_like(w)
        sig = [SIGMA0[0] + zero, SIGMA0[1] + zero, SIGMA0[2] + zero, SIGMA0[3] * w,
               SIGMA0[4] + zero, SIGMA0[5] + zero]
        par = [m + s * self.normal() for m, s in zip((zero, zero, zero, w, self.phi0, self.theta), sig)]
        return par, [s * s for s in sig]


def track_inputs(case, seed, device="cuda"):
    """(ntrk, mode, arrays): the case's events and par, cov, q, hpos, hcov (or
    the candidates' cpos, ccov), track fastest, ld a multiple of 32."""
    nt, md = events(case, seed)
    n, nl = int(nt.sum()), case["nlayer"]
    ld = (n + 31) // 32 * 32
    mode = torch.from_numpy(np.repeat(md, nt)).to(device)
    t = Tracks(mode, nl, seed)
    dtype = torch.float64 if case["entry"] == "f64" else torch.float32
    new = lambda *shape: torch.zeros(shape + (ld,), dtype=dtype, device=device)  # noqa: E731
    a = {"par": new(6), "cov": new(21), "q": torch.ones(ld, dtype=torch.int32, device=device)}
    par, var = t.start()
    for k in range(6):
        # (in double, too, the inputs are numbers that a float holds)
        a["par"][k, :n] = par[k].float()
        a["cov"][k * (k + 1) // 2 + k, :n] = var[k].float()
    a["q"][:n] = t.q.to(torch.int32)
    if case["entry"] != "find":
        a["hpos"], a["hcov"] = new(nl, 3), new(nl, 6)
        for l in range(nl):
            pos, cov = t.hit(l)
            for k in range(3):
                a["hpos"][l, k, :n] = pos[k].float()
            for k in range(6):
                a["hcov"][l, k, :n] = cov[k].float()
        return nt, md, a
    # the track's own hit with probability 0.95 in a random slot, noise within
    # 20 times the hit errors of it in the others
    nc = case["ncand"]
    a["cpos"], a["ccov"] = new(nl, nc, 3), new(nl, nc, 6)
    for l in range(nl):
        r, phi, z = t.crossing(l)
        n1, n2 = t.normal(), t.normal()
        slot = torch.floor(t.uniform(0.0, nc))
        slot = torch.where(t.uniform(0.0, 1.0) < 0.95, slot, -1.0)
        for c in range(nc):
            m1, m2 = n1 + 20.0 * t.normal(), n2 + 20.0 * t.normal()
            pos, cov = t.near(r, phi, z, torch.where(slot == c, n1, m1), torch.where(slot == c, n2, m2))
            for k in range(3):
                a["cpos"][l, c, k, :n] = pos[k].float()
            for k in range(6):
                a["ccov"][l, c, k, :n] = cov[k].float()
    return nt, md, a


def train_inputs(n, seed, device="cuda"):
    """Network inputs (n, 8) and targets (n,) of p2r propagations from the
    state a fit holds before a layer drawn uniformly (float32), as
    fit_mlp_prepare makes them."""
    nl = 20
    t = Tracks(torch.full((n,), P2R, dtype=torch.int32, device=device), nl, seed)
    layer = torch.floor(t.uniform(0.0, nl)).long()
    prev = t.surf[0][torch.clamp(layer - 1, min=0)]
    half = torch.asin(prev / (2.0 * t.rho))
    az, w = t.phi0 - t.q * half, 1.0 / t.pt
    first = (layer == 0).double()
    mean = [(1 - first) * prev * torch.cos(az), (1 - first) * prev * torch.sin(az),
            (1 - first) * 2.0 * t.rho * half / torch.tan(t.theta), w,
            t.phi0 - 2.0 * t.q * half * (1 - first), t.theta]
    sig = [torch.where(layer == 0, SIGMA0[k], SIGMA_STATE[k]) * (w if k == 3 else 1.0)
           for k in range(6)]
    x, y, z, w, phi, theta = (m + s * t.normal() for m, s in zip(mean, sig))
    R = t.surf[0][layer]
    kappa = -t.q * KA * B_FIELD * w
    h, _ = path_length(x, y, phi, kappa, R)
    b0 = x * torch.cos(phi) + y * torch.sin(phi)
    line = torch.sqrt(b0 * b0 + R * R - x * x - y * y) - b0
    r0 = torch.sqrt(x * x + y * y)
    psi = phi - torch.atan2(y, x)
    f = [r0 / R, z / R, 0.5 * KA * B_FIELD * w * R, torch.cos(psi), torch.sin(psi),
         torch.cos(theta), t.q, R / 100.0]
    return torch.stack(f, 1).float().contiguous(), ((h - line) / (0.5 * kappa * line * line)).float()


def start_params(seed):
    """He-uniform weights and zero biases, the float32 vector fit_mlp_set_params takes."""
    g = np.random.Generator(np.random.Philox(key=int(seed)))
    return np.concatenate([g.uniform(-1.0, 1.0, s).ravel() * math.sqrt(6.0 / s[1]) if len(s) == 2
                           else np.zeros(s) for s in MLP_SHAPES]).astype(np.float32)


@functools.lru_cache(maxsize=1)
def trained_params():
    """The network that a program keeps for its seeded fits: trained once."""
    x, y = train_inputs(1 << 17, 4)
    params, _ = train64(x, y, start_params(4), 8192, 96, 4, lr=4e-3)
    return params.float().cpu().numpy()


# ---- what a program keeps, and its call --------------------------------------------------


def prepare(case, seed):
    if case["entry"] == "train":
        x, y = train_inputs(case["n"], seed)
        return {"case": case, "x": x, "y": y, "net": fit.fit_mlp_create(0, seed=1),
                "params": start_params(seed + 1)}
    nt, md, a = track_inputs(case, seed)
    n, nl, entry = int(nt.sum()), case["nlayer"], case["entry"]
    ld = a["par"].shape[-1]
    tol = 1e-12 if entry == "f64" else 1e-6
    start = fit.FIT_START_LINE if entry == "seeded" else fit.FIT_START_CROSSING
    geo = [fit.Geometry(B_FIELD, surfaces(m, nl), tol=tol, start=start) for m in (P2R, P2Z)]
    s = {"case": case, "nt": nt, "md": md, "n": n, "geo": geo, **a}
    if entry == "noalloc":
        f = None
        s["out"] = {"par": torch.zeros(6, ld, device="cuda"), "cov": torch.zeros(21, ld, device="cuda"),
                    "q": torch.zeros(ld, dtype=torch.int32, device="cuda"),
                    "chi2": torch.zeros(ld, device="cuda"),
                    "status": torch.zeros(ld, dtype=torch.uint8, device="cuda")}
    else:
        f = s["fitter"] = fit.Fitter(geo[0], geo[1], device=0)
        s["out"] = f.outputs(n, ld=ld)
    if entry == "f64":
        s["out"].update({k: s["out"][k].double() for k in ("par", "cov", "chi2")})
    elif entry == "find":
        s["chosen"] = torch.zeros((nl, ld), dtype=torch.int8, device="cuda")
    elif entry == "adjoint":
        s["weight"] = torch.ones(ld, device="cuda")
        for k in ("hpos", "par", "cov"):
            s[k].requires_grad_(True)
    elif entry == "seeded":
        net = fit.fit_mlp_create(0, seed=1)
        fit.fit_mlp_set_params(net, trained_params())
        fit.fit_mlp_attach(f.h, net)
        torch.cuda.synchronize()
        fit.fit_mlp_destroy(net)
    elif entry == "host":
        for k in ("par", "cov", "q", "hpos", "hcov"):
            s[k] = s[k].cpu().pin_memory()
        s["out"] = {k: torch.zeros(v.shape, dtype=v.dtype, pin_memory=True)
                    for k, v in s["out"].items() if v is not None}
    elif entry == "plan":
        s["plan"] = fit.fit_plan_create(f.h, nt, md, nl, layout=case["layout"])
        if case["layout"] == fit.FIT_LAYOUT_AOSOA32:
            for k in ("par", "cov", "hpos", "hcov"):
                tiles = torch.empty_like(s[k])
                fit.fit_relayout(s[k], fit.FIT_LAYOUT_SOA, tiles, fit.FIT_LAYOUT_AOSOA32)
                s[k] = tiles
    return s


def run(s):
    entry = s["case"]["entry"]
    if entry == "train":
        c = s["case"]
        fit.fit_mlp_set_params(s["net"], s["params"])
        curve = fit.fit_mlp_train(s["net"], s["x"], s["y"], epochs=c["epochs"], batch=c["batch"],
                                  lr=2e-3, lr_final=1e-4, seed=7)
        return {"params": fit.fit_mlp_get_params(s["net"]), "loss": curve}
    n, out, nt, md = s["n"], s["out"], s["nt"], s["md"]
    if entry == "adjoint":
        chi2, par, cov = fit.chi2(s["fitter"], s["hpos"], s["par"], s["cov"], s["q"], s["hcov"], nt, md)
        g = torch.autograd.grad(chi2, (s["hpos"], s["par"], s["cov"]), s["weight"])
        return {"chi2": chi2[:n], "par": par[:, :n], "cov": cov[:, :n], "g_hpos": g[0][..., :n],
                "g_par": g[1][:, :n], "g_cov": g[2][:, :n]}
    bufs = dict(par_out=out["par"], cov_out=out["cov"], q_out=out["q"], chi2=out["chi2"],
                status=out["status"])
    if entry in ("fit", "seeded"):
        s["fitter"].run(s["par"], s["cov"], s["q"], s["hpos"], s["hcov"], nt, md, out=out)
    elif entry == "plan":
        fit.fit_plan_run(s["plan"], s["par"], s["cov"], s["q"], s["hpos"], s["hcov"], **bufs)
    elif entry == "f64":
        fit.fit_propagate_update_f64(s["fitter"].h, s["par"], s["cov"], s["q"], s["hpos"], s["hcov"],
                                     nt, md, **bufs)
    elif entry == "host":
        fit.fit_propagate_update_host(s["fitter"].h, s["par"], s["cov"], s["q"], s["hpos"],
                                      s["hcov"], nt, md, **bufs)
    elif entry == "find":
        fit.fit_find_tracks(s["fitter"].h, s["par"], s["cov"], s["q"], s["cpos"], s["ccov"], nt, md,
                            GATE, s["chosen"], **bufs)
    elif entry == "noalloc":
        per_event = fit.fit_propagate_update_noalloc(s["geo"][0], s["geo"][1], s["par"], s["cov"],
                                                     s["q"], s["hpos"], s["hcov"], nt, md, **bufs)
    # the tracks of the events (a leading dimension may be longer; in tiles of
    # 32 tracks the arrays are returned whole up to the tile that ends it)
    if entry == "plan" and s["case"]["layout"] == fit.FIT_LAYOUT_AOSOA32:
        res = {k: out[k].view(-1, out[k].shape[0], 32)[:n // 32] for k in ("par", "cov")}
        res["chi2"], res["q"], res["status"] = out["chi2"][:n], out["q"][:n], out["status"][:n]
    else:
        res = {k: out[k][..., :n] for k in ("par", "cov", "chi2", "q", "status")}
    if entry == "find":
        res["chosen"] = s["chosen"][:, :n]
    elif entry == "noalloc":
        res["counters"] = np.array([list(c.values()) for c in per_event], np.int64)
    return res


# ---- the same in 64 bits ------------------------------------------------------------------


def path_length(x, y, phi, kappa, R):
    """(first forward crossing of the helix with the cylinder R, whether it
    reaches it): the closed form in tan(kappa h / 2), polished by Newton."""
    cph, sph = torch.cos(phi), torch.sin(phi)
    b0, t0 = x * cph + y * sph, y * cph - x * sph
    c0 = x * x + y * y - R * R
    X = b0 * b0 - c0 * (1.0 + kappa * (t0 + 0.25 * kappa * c0))
    sq = torch.sqrt(torch.clamp(X, min=0.0))
    period = 2.0 * math.pi / kappa.abs()
    h = torch.full_like(x, math.inf)
    for den in (b0 + sq, b0 - sq):
        hk = 2.0 * torch.atan2(-0.5 * kappa * c0, den) / kappa
        hk = hk - torch.floor(hk / period) * period
        h = torch.minimum(h, torch.where(hk > 0.0, hk, hk + period))
    for _ in range(3):
        px, py, c1, s1 = helix(x, y, cph, sph, kappa, h)[:4]
        d = 0.5 * (px * px + py * py - R * R) / (px * c1 + py * s1)
        h = h - torch.where(d.abs() < 1e-3 * R, d, 0.0)
    return h, (X >= 0.0) & (h > 0.0)


def sinc(u):
    """sin(u)/u and its derivative."""
    small = u.abs() < 0.05
    v, u2 = torch.where(small, 1.0, u), u * u
    s = torch.sin(v) / v
    series = 1 - u2 / 6 * (1 - u2 / 20 * (1 - u2 / 42 * (1 - u2 / 72)))
    ds = -u / 3 * (1 - u2 / 10 * (1 - u2 / 28 * (1 - u2 / 54 * (1 - u2 / 88))))
    return torch.where(small, series, s), torch.where(small, ds, (torch.cos(v) - s) / v)


def helix(x, y, cph, sph, kappa, h):
    """x', y', cos phi', sin phi' after a transverse path h, and the factors
    that its derivatives need."""
    u = 0.5 * kappa * h
    s, ds = sinc(u)
    cu, su = torch.cos(u), torch.sin(u)
    cm, sm = cph * cu - sph * su, sph * cu + cph * su
    dx, dy = h * s * cm, h * s * sm
    return x + dx, y + dy, cm * cu - sm * su, sm * cu + cm * su, dx, dy, s, ds, cm, sm


def matrix(rows):
    return torch.stack([torch.stack(r, -1) for r in rows], -2)


def fit64(mode, par, cov, q, hits, nlayer, gate=None):
    """The fit of the tracks (columns of par (6, n), cov (21, n), q (n,)), all
    of one mode, in 64 bits.  hits(l): list of (position 3, covariance 6), the
    candidates of layer l; without a gate there is one and it is taken."""
    p = list(par.double())
    q = q.double()
    packed = {pr: cov[k].double() for k, pr in enumerate(PAIRS)}
    C = matrix([[packed[max(i, j), min(i, j)] for j in range(6)] for i in range(6)])
    chi2 = torch.zeros_like(q)
    alive = torch.ones_like(q, dtype=torch.bool)
    one, zero = torch.ones_like(q), torch.zeros_like(q)
    for l in range(nlayer):
        S = float(surfaces(mode, nlayer)[l])
        x, y, z, w, phi, th = p
        kappa, dk = -q * KA * B_FIELD * w, -q * KA * B_FIELD
        cph, sph, tan = torch.cos(phi), torch.sin(phi), torch.tan(th)
        if mode == P2Z:
            h = (S - z) * tan
            ok = h > 0
        else:
            with torch.no_grad():
                h, ok = path_length(x, y, phi, kappa, torch.full_like(x, S))
            px, py, c1, s1 = helix(x, y, cph, sph, kappa, h)[:4]
            # a Newton step that only carries the derivative of h
            h = h - 0.5 * (px * px + py * py - S * S) / (px * c1 + py * s1).detach()
        px, py, c1, s1, dx, dy, s, ds, cm, sm = helix(x, y, cph, sph, kappa, h)
        hh = 0.5 * h * h * dk
        xw, yw = hh * (ds * cm - s * sm), hh * (ds * sm + s * cm)
        A = matrix([[one, zero, zero, xw, -dy, zero], [zero, one, zero, yw, dx, zero],
                    [zero, zero, one, zero, zero, -h / torch.sin(th) ** 2],
                    [zero, zero, zero, one, zero, zero], [zero, zero, zero, h * dk, one, zero],
                    [zero, zero, zero, zero, zero, one]])
        v = torch.stack([c1, s1, 1.0 / tan, zero, kappa, zero], -1)
        if mode == P2Z:
            g = torch.stack([zero, zero, -tan, zero, zero, (S - z) / torch.cos(th) ** 2], -1)
        else:
            g = -(px[:, None] * A[:, 0] + py[:, None] * A[:, 1]) / (px * c1 + py * s1)[:, None]
        J = A + v[:, :, None] * g[:, None, :]
        Cp = J @ C @ J.transpose(1, 2)
        pp = torch.stack([px, py, z + h / tan if mode == P2R else torch.full_like(z, S), w,
                          phi + kappa * h, th], -1)
        best, take = None, None
        for c, (m, V) in enumerate(hits(l)):
            m, V = [k.double() for k in m], [k.double() for k in V]
            if mode == P2Z:
                H = matrix([[one, zero, zero], [zero, one, zero]])
            else:
                r = torch.sqrt(m[0] * m[0] + m[1] * m[1])
                H = matrix([[-m[1] / r, m[0] / r, zero], [zero, zero, one]])
            V = matrix([[V[0], V[1], V[3]], [V[1], V[2], V[4]], [V[3], V[4], V[5]]])
            res = (H @ (torch.stack(m, -1) - pp[:, :3])[:, :, None])[:, :, 0]
            a = Cp[:, :, :3] @ H.transpose(1, 2)
            Sm = H @ a[:, :3] + H @ V @ H.transpose(1, 2)
            det = Sm[:, 0, 0] * Sm[:, 1, 1] - Sm[:, 0, 1] * Sm[:, 1, 0]
            Si = matrix([[Sm[:, 1, 1], -Sm[:, 0, 1]], [-Sm[:, 1, 0], Sm[:, 0, 0]]]) / det[:, None, None]
            x2 = (res * (Si @ res[:, :, None])[:, :, 0]).sum(-1)
            K = a @ Si
            this = (x2, pp + (K @ res[:, :, None])[:, :, 0], Cp - K @ Sm @ K.transpose(1, 2))
            if gate is None:
                best, take = this, alive & ok
            else:
                better = (x2 < gate) if best is None else (x2 < best[0])
                if best is None:
                    best, take = (torch.full_like(x2, gate), pp, Cp), torch.zeros_like(alive)
                best = tuple(torch.where(better.view(-1, *[1] * (b.dim() - 1)), t, b)
                             for t, b in zip(this, best))
                take = take | better
        alive = alive & ok
        chi2 = chi2 + torch.where(alive & take, best[0], 0.0)
        pn, Cn = best[1], best[2]
        flip = pn[:, 3] < 0
        sign = torch.ones_like(pn)
        sign[:, 3] = torch.where(flip, -1.0, 1.0)
        phi = pn[:, 4]
        if gate is None:
            wrapped = phi - 2.0 * math.pi * torch.ceil(((phi - math.pi) / (2.0 * math.pi)).detach())
        else:  # a layer without a hit leaves the azimuth as it is
            wrapped = torch.where(take, phi - 2.0 * math.pi * torch.ceil((phi - math.pi) / (2.0 * math.pi)), phi)
        pn = torch.cat([pn[:, :4], wrapped[:, None], pn[:, 5:]], 1) * sign
        Cn = Cn * sign[:, :, None] * sign[:, None, :]
        p = [torch.where(alive, pn[:, k], p[k]) for k in range(6)]
        C = torch.where(alive[:, None, None], Cn, C)
        q = torch.where(alive & flip, -q, q)
    return torch.stack(p), torch.stack([C[:, i, j] for i, j in PAIRS]), chi2


def fit64_events(case, md, nt, a, grad=False):
    """fit64 over the case's tracks, a mode and a chunk at a time."""
    mode = np.repeat(md, nt)
    n, nl = mode.shape[0], case["nlayer"]
    dev = a["par"].device
    new = lambda *shape: torch.zeros(shape + (n,), dtype=torch.float64, device=dev)  # noqa: E731
    res = {"par": new(6), "cov": new(21), "chi2": new()}
    if grad:
        res.update(g_hpos=new(nl, 3), g_par=new(6), g_cov=new(21))
    for m in (P2R, P2Z):
        every = torch.from_numpy(np.nonzero(mode == m)[0]).to(dev)
        for idx in every.split(20000 if grad else 200000):
            if not len(idx):
                continue
            par, cov, q = (a[k][..., idx].double() for k in ("par", "cov", "q"))
            if case["entry"] == "find":
                hits = lambda l: [(a["cpos"][l, c][:, idx], a["ccov"][l, c][:, idx])  # noqa: E731
                                  for c in range(case["ncand"])]
            else:
                hp, hc = a["hpos"][..., idx].double(), a["hcov"][..., idx].double()
                hits = lambda l: [(hp[l], hc[l])]  # noqa: E731
            if grad:
                leaves = [t.detach().requires_grad_(True) for t in (hp, par, cov)]
                hp, par, cov = leaves
            p, c, x2 = fit64(m, par, cov, q, hits, nl, GATE if case["entry"] == "find" else None)
            for k, t in zip(("par", "cov", "chi2"), (p, c, x2)):
                res[k][..., idx] = t.detach()
            if grad:
                for k, t in zip(("g_hpos", "g_par", "g_cov"), torch.autograd.grad(x2.sum(), leaves)):
                    res[k][..., idx] = t
    return res


def splitmix64(x):
    mask = (1 << 64) - 1
    x = (x + 0x9e3779b97f4a7c15) & mask
    z = x
    z = ((z ^ (z >> 30)) * 0xbf58476d1ce4e5b9) & mask
    z = ((z ^ (z >> 27)) * 0x94d049bb133111eb) & mask
    return x, z ^ (z >> 31)


def train64(x, y, params, batch, epochs, seed, lr=2e-3, lr_final=1e-4):
    """Adam on the network's mean squared error in 64 bits, without rounding
    to BF16: (parameters, mean loss of each epoch); the batches that
    fit_mlp_train takes."""
    n = x.shape[0]
    X, Y = x.double(), y.double()
    P = torch.from_numpy(params).to(x.device).double()
    parts = [math.prod(s) for s in MLP_SHAPES]
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    steps, t, losses = n // batch, 0, []
    for _ in range(epochs):
        seed, r = splitmix64(seed)
        first, loss = r % n, torch.zeros((), dtype=torch.float64, device=x.device)
        for k in range(steps):
            rate = lr_final + 0.5 * (lr - lr_final) * (1 + math.cos(math.pi * t / max(1, steps * epochs - 1)))
            lo = (first + k * batch) % n
            xb, yb = X[lo:lo + batch], Y[lo:lo + batch]
            if lo + batch > n:
                xb, yb = torch.cat([xb, X[:lo + batch - n]]), torch.cat([yb, Y[:lo + batch - n]])
            W1, b1, W2, b2, W3, b3 = (w.view(s) for w, s in zip(P.split(parts), MLP_SHAPES))
            z1 = torch.addmm(b1, xb, W1.T)
            a1 = z1.clamp(min=0)
            z2 = torch.addmm(b2, a1, W2.T)
            a2 = z2.clamp(min=0)
            e = a2 @ W3[0] + b3 - yb
            loss += (e * e).sum()
            dy = 2.0 / batch * e
            dz2 = dy[:, None] * W3 * (z2 > 0)
            dz1 = dz2 @ W2 * (z1 > 0)
            G = torch.cat([(dz1.T @ xb).view(-1), dz1.sum(0), (dz2.T @ a1).view(-1), dz2.sum(0),
                           dy @ a2, dy.sum()[None]])
            t += 1
            M = 0.9 * M + 0.1 * G
            V = 0.999 * V + 0.001 * G * G
            P = P - rate * (M / (1 - 0.9 ** t)) / (torch.sqrt(V / (1 - 0.999 ** t)) + 1e-8)
        losses.append(loss / (batch * steps))
    return P, torch.stack(losses)


def exact(case, seed):
    if case["entry"] == "train":
        x, y = train_inputs(case["n"], seed)
        p, loss = train64(x, y, start_params(seed + 1), case["batch"], case["epochs"], 7)
        return {"params": p, "loss": loss}
    nt, md, a = track_inputs(case, seed)
    n = int(nt.sum())
    res = fit64_events(case, md, nt, a, grad=case["entry"] == "adjoint")
    if case["entry"] == "plan" and case["layout"] == fit.FIT_LAYOUT_AOSOA32:
        for k in ("par", "cov"):
            r = res[k].shape[0]
            res[k] = res[k][:, :n // 32 * 32].reshape(r, -1, 32).transpose(0, 1).contiguous()
    return res
