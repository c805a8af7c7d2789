"""Performance cases of the radiation-deposit library: what a user's program has it compute.

Each case is one pass through the public entry points on inputs that live on the GPU: zero the
detector, deposit trajectories (in one call, in streamed stretches behind a particle push, or many
problems in one batch), then read the fields, take spectra, or run the adjoint.  Trajectories and
detectors are those of paper_2302_14812_gb300.workloads (undulator ensembles on a spherical cap, the
helix and the K = 10 line detector of the paper's examples, circular orbits, oscillators, the
plasma-mirror surface on a plane), evaluated with PyTorch on the device from the seed.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs and detectors
  run(state)           one pass
  work(case)           bytes and flops a pass cannot do without
  exact(case, seed)    the same outputs in 64-bit PyTorch
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W

_F64 = {"dtype": torch.float64, "device": "cuda"}


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _deposit(name, motion, n_part, n_steps, rows, cols, n_bins, precision="mixed", far=False, interp="held"):
    return {"name": name, "path": "deposit", "motion": motion, "n_part": n_part, "n_steps": n_steps, "rows": rows,
            "cols": cols, "n_bins": n_bins, "precision": precision, "far": far, "interp": interp}


def listed():
    return [
        # one electron on a circular orbit seen by a 64-cell arc: a textbook check, an interactive
        # parameter scan -- the smallest call, bound by launches and latency
        _deposit("arc_one_electron", "circular", 1, 2000, 1, 64, 1024),
        # one electron on the helix of Section 3.3, a 64 x 64 image with 8192 narrow bins: little
        # arithmetic, much detector memory
        _deposit("helix_image", "helix", 1, 400, 64, 64, 8192),
        # Section 4 benchmark: one K = 10 electron, a line of 512 cells x 131072 bins, and the power
        # spectra of E that are compared with the synchrotron formulas
        {"name": "line_spectrum", "path": "spectrum", "motion": "wiggler", "n_part": 1, "n_steps": 38000, "rows": 1,
         "cols": 512, "n_bins": 131072, "precision": "mixed", "far": False, "interp": "held"},
        # a modest undulator run with sizes that are multiples of nothing
        _deposit("cap_ragged", "undulator", 37, 3001, 61, 53, 1021),
        # the benchmark's ensemble at full size
        _deposit("cap_full", "undulator", 1000, 4000, 128, 128, 2048),
        # a slice of the plasma-mirror surface on a plane with a time origin for every cell
        _deposit("mirror_plane", "mirror", 40, 5000, 72, 96, 2400),
        # second-order interpolation in time, taken where the particle code's step is coarse
        _deposit("cap_linear", "undulator", 100, 1500, 100, 100, 1500, interp="linear"),
        # the plain FP64 path, as a reference for a mixed run
        _deposit("cap_fp64", "undulator", 24, 1200, 64, 64, 1024, precision="fp64"),
        # run-time coupling: every 25 Boris steps the new samples are deposited at once
        {"name": "push_and_stream", "path": "stream", "motion": "gyration", "n_part": 256, "n_steps": 400, "rows": 30,
         "cols": 40, "n_bins": 1500, "stretch": 25, "precision": "mixed", "far": False, "interp": "held"},
        # many uneven problems in one batched call (a scan over set-ups)
        {"name": "batch_uneven", "path": "batch", "n_problems": 24, "scale": 0.0005, "sizes": 4},
        # a training step: forward, misfit against a measured field, gradients for FP32 corrections to
        # the trajectories
        {"name": "fit_step", "path": "fit", "motion": "undulator", "n_part": 48, "n_steps": 1500, "rows": 64,
         "cols": 64, "n_bins": 1024, "precision": "mixed", "far": False, "interp": "held"},
        # gradients to 1e-6 in FP64 (the compensated adjoint), for given seeds
        {"name": "adjoint_compensated", "path": "adjoint", "motion": "undulator", "n_part": 12, "n_steps": 1000,
         "rows": 48, "cols": 64, "n_bins": 768, "precision": "mixed", "far": False, "interp": "held"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# most (particle, interval, cell) triples of a drawn case, or (particle, cell, bin) triples where its steps
# pass several bins, and most detector bins
_DRAW_TRIPLES = {"deposit": 1.5e10, "deposit_fp64": 4e8, "spectrum": 2e8, "stream": 2e9, "fit": 5e8, "adjoint": 5e7}
_DRAW_BINS = 2.0e7


def draw(rng: random.Random):
    path = rng.choice(["deposit"] * 5 + ["spectrum", "stream", "batch", "fit", "adjoint"])
    if path == "batch":
        return {"path": "batch", "n_problems": rng.randint(3, 24),
                "scale": math.exp(rng.uniform(math.log(1e-4), math.log(1e-3))), "sizes": rng.randrange(1 << 20)}
    c = {"path": path, "precision": "mixed", "far": False, "interp": "held"}
    if path == "deposit":
        c["motion"] = rng.choice(["circular", "helix", "undulator", "undulator", "mirror"])
        c["precision"] = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        c["interp"] = rng.choice(["held", "held", "held", "linear", "previous", "quadratic"])
        c["far"] = c["motion"] in ("circular", "undulator") and rng.random() < 0.25
    elif path == "spectrum":
        c["motion"] = "wiggler"
    elif path == "stream":
        c["motion"] = "gyration"
    else:
        c["motion"] = "undulator"
    one = c["motion"] in ("helix", "wiggler")           # single-electron examples
    budget = _DRAW_TRIPLES["deposit_fp64" if c["precision"] == "fp64" else path]
    while True:
        c["n_part"] = 1 if one else _log_int(rng, 1, 1200)
        c["n_steps"] = _log_int(rng, 200, 800) if c["motion"] == "helix" else _log_int(rng, 300, 8000)
        if c["motion"] == "circular" and not c["far"] and rng.random() < 0.5:
            c["rows"], c["cols"] = 1, _log_int(rng, 16, 600)
        elif c["motion"] == "wiggler":
            c["n_steps"], c["rows"], c["cols"] = _log_int(rng, 8000, 40000), 1, _log_int(rng, 32, 600)
        else:
            c["rows"], c["cols"] = _log_int(rng, 8, 128), _log_int(rng, 8, 128)
        if path == "spectrum":
            c["n_bins"] = 1 << rng.randint(10, 17)
        elif c["motion"] == "helix":
            c["n_bins"] = _log_int(rng, 2000, 9000)
        else:
            c["n_bins"] = _log_int(rng, 300, 4096)
        cells = c["rows"] * c["cols"]
        if c["n_part"] * max(c["n_steps"], c["n_bins"]) * cells <= budget and cells * c["n_bins"] <= 4 * _DRAW_BINS:
            break
    if path == "stream":
        c["stretch"] = _log_int(rng, 5, 120)
    return c


# ------------------------------------------------------------------------------------------------
# trajectories (FP64, on the device) and detectors
# ------------------------------------------------------------------------------------------------
def _charges(n, g):
    """Macro-particle charges around -1."""
    return -(0.5 + torch.rand(n, generator=g, **_F64))


def _integrate(beta, x0, dt, n_steps):
    """x_k = x0 + int beta dt by 8-node Gauss-Legendre quadrature of every step; beta(t, rows) -> [rows][m][3]."""
    nodes, weights = (torch.tensor(v, **_F64) for v in np.polynomial.legendre.leggauss(8))
    t = (dt * (torch.arange(n_steps, **_F64)[:, None] + 0.5 * (1.0 + nodes[None, :]))).reshape(-1)
    x = torch.empty((x0.shape[0], n_steps + 1, 3), **_F64)
    x[:, 0] = x0
    for p in range(0, x0.shape[0], 256):
        s = slice(p, min(x0.shape[0], p + 256))
        inc = 0.5 * dt * torch.einsum("psnc,n->psc", beta(t, s).reshape(s.stop - p, n_steps, 8, 3), weights)
        x[s, 1:] = x0[s, None, :] + torch.cumsum(inc, dim=1)
    return x


def _undulator(n_part, n_steps, gamma, K, n_periods, g, lam=1.0, sigma=1e-3):
    """Planar undulator along +z, wiggling in y, random phases and transverse offsets."""
    bz_bar, w = W.undulator_params(gamma, K, lam)
    dt = n_periods * lam / bz_bar / n_steps
    phi = 2.0 * math.pi * torch.rand(n_part, generator=g, **_F64)
    x0 = torch.zeros((n_part, 3), **_F64)
    x0[:, :2] = sigma * torch.randn((n_part, 2), generator=g, **_F64)

    def beta(t, s):
        by = (K / gamma) * torch.sin(w * t[None, :] + phi[s, None])
        return torch.stack([torch.zeros_like(by), by, torch.sqrt(1.0 - 1.0 / gamma ** 2 - by * by)], dim=-1)

    x = _integrate(beta, x0, dt, n_steps)
    t = dt * torch.arange(n_steps + 1, **_F64)
    return x, gamma * beta(t, slice(0, n_part)), dt


def _circular(n_part, n_steps, gamma, n_orbits, g):
    """Unit circle in the x-y plane, random phases."""
    w = math.sqrt(1.0 - 1.0 / gamma ** 2)
    dt = n_orbits * 2.0 * math.pi / w / n_steps
    ph = w * dt * torch.arange(n_steps + 1, **_F64)[None, :]
    ph = ph + 2.0 * math.pi * torch.rand((n_part, 1), generator=g, **_F64)
    z = torch.zeros_like(ph)
    x = torch.stack([torch.cos(ph), torch.sin(ph), z], dim=-1)
    return x, gamma * w * torch.stack([-torch.sin(ph), torch.cos(ph), z], dim=-1), dt


def _oscillators(n_part, n_steps, g):
    """Linear relativistic oscillators along x, random amplitudes and phases, 6 periods."""
    a = 0.1 + 1.9 * torch.rand((n_part, 1), generator=g, **_F64)
    phi = 2.0 * math.pi * torch.rand((n_part, 1), generator=g, **_F64)
    dt = 12.0 * math.pi / n_steps

    def mom(t, s):
        ux = a[s] * torch.sin(t[None, :] + phi[s])
        return torch.stack([ux, torch.zeros_like(ux), torch.zeros_like(ux)], dim=-1)

    def beta(t, s):
        uu = mom(t, s)
        return uu / torch.sqrt(1.0 + (uu * uu).sum(-1, keepdim=True))

    x = _integrate(beta, 1e-2 * torch.randn((n_part, 3), generator=g, **_F64), dt, n_steps)
    return x, mom(dt * torch.arange(n_steps + 1, **_F64), slice(0, n_part)), dt


def _helix(n_steps, g):
    """Section 3.3: gamma 57.3, K 0.8, unit frequency, dt = 0.1, along +x; the phase is random."""
    gamma, K, dt = 57.3, 0.8, 0.1
    bp = K / gamma
    bx = math.sqrt(1.0 - 1.0 / gamma ** 2 - bp ** 2)
    t = dt * torch.arange(n_steps + 1, **_F64)
    ph = t + 2.0 * math.pi * torch.rand(1, generator=g, **_F64)
    x = torch.stack([bx * t, bp * torch.cos(ph), bp * torch.sin(ph)], dim=-1)
    u = gamma * torch.stack([torch.full_like(t, bx), -bp * torch.sin(ph), bp * torch.cos(ph)], dim=-1)
    return x[None].contiguous(), u[None].contiguous(), dt


def _cap(rows, cols, radius, half, axis):
    """rows x cols cells of a spherical detector spanning +-half rad around coordinate `axis`."""
    a = torch.sin(-half + (torch.arange(rows, **_F64) + 0.5) * (2.0 * half / rows))[:, None].expand(rows, cols)
    b = torch.sin(-half + (torch.arange(cols, **_F64) + 0.5) * (2.0 * half / cols))[None, :].expand(rows, cols)
    p = torch.empty((rows, cols, 3), **_F64)
    others = [i for i in range(3) if i != axis]
    p[..., others[0]], p[..., others[1]], p[..., axis] = a, b, torch.sqrt(1.0 - a * a - b * b)
    return (radius * p).reshape(-1, 3)


def _first_arrival(pos, x, dt):
    """Earliest arrival of the (single) particle's samples at every cell."""
    t = dt * torch.arange(x.shape[1], **_F64)
    return torch.cat([(t[None] + torch.linalg.vector_norm(p[:, None] - x[0][None], dim=2)).amin(1)
                      for p in pos.split(64)])


def _setup(c, seed):
    """(x, u, q, t0, dt), (pos, pix_t0, t_min, dt_det, n_bins) of a case."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n, S, nb = c["n_part"], c["n_steps"], c["n_bins"]
    q, t0v = None, None
    if c["motion"] == "undulator":
        # gamma 20, K 1, 10 periods, a cap of +-1.5/gamma at 1e4, the window holds every arrival
        gamma, K, half, dist = 20.0, 1.0, 0.075, 1e4
        x, u, dt = _undulator(n, S, gamma, K, 10.0, g)
        q = _charges(n, g)
        bz, w = W.undulator_params(gamma, K)
        pos = _cap(c["rows"], c["cols"], dist, half, 2)
        t_min, dt_det = W.axial_window(dist, S * dt, bz, math.asin(math.sqrt(2.0) * math.sin(half)),
                                       K / (gamma * w) + 6e-3, nb)
    elif c["motion"] == "wiggler":
        # gamma 50, K 10, 5 periods of 2 pi / 0.1, a line of cells over 0.1 rad at 1e5; the bin width
        # scales with the number of bins, so that the window stays the benchmark's
        lam, dist = 20.0 * math.pi, 1e5
        x, u, dt = _undulator(n, S, 50.0, 10.0, 5.0, g, lam, 0.0)
        x[:, :, :2] -= x[:, :1, :2]
        th = torch.linspace(-0.05, 0.05, c["cols"], **_F64)
        pos = torch.stack([dist * torch.sin(th), torch.zeros_like(th), dist * torch.cos(th)], dim=1)
        dt_det = 2.98e-5 * 131072 / nb
        t_min, t0v = dist, _first_arrival(pos, x, dt) - 0.01 - dist
    elif c["motion"] == "helix":
        dist = 1e6
        x, u, dt = _helix(S, g)
        pos = _cap(c["rows"], c["cols"], dist, 0.05, 0)
        dt_det = 1.33e-5 * 8192 / nb
        t_min, t0v = dist, _first_arrival(pos, x, dt) - 20.0 * dt_det - dist
    elif c["motion"] == "circular":
        gamma, dist = 5.0, 1e3
        x, u, dt = _circular(n, S, gamma, S / 100.0, g)
        span = S * dt + 2.0
        if c["rows"] == 1:
            # an arc in the orbit plane, neighbouring cells 2 dt of the orbit apart
            w = math.sqrt(1.0 - 1.0 / gamma ** 2)
            ph = 2.0 * dt * w * torch.arange(c["cols"], **_F64)
            pos = dist * torch.stack([torch.cos(ph), torch.sin(ph), torch.zeros_like(ph)], dim=1)
        else:
            pos = _cap(c["rows"], c["cols"], dist, 0.6, 2)
        dt_det = 1.04 * span / nb
        t_min = dist - 1.0 - 0.02 * span
    elif c["motion"] == "mirror":
        x, u, q, (_, dt) = W.plasma_mirror_surface_torch(slice(0, n), n_part=n, n_steps=S, seed=int(seed) % (1 << 31))
        lam0 = 2.0 * math.pi
        s = [(-6.4 * lam0 + (torch.arange(m, **_F64) + 0.5) * (12.8 * lam0 / m)) for m in (c["rows"], c["cols"])]
        yy, zz = torch.meshgrid(s[0], s[1], indexing="ij")
        pos = torch.stack([torch.full_like(yy, -6.4 * lam0), yy, zz], dim=-1).reshape(-1, 3)
        reach = 3.0 * math.sqrt(2.0) * lam0 + 0.1 * lam0 + 5.0
        span = S * dt + 2.0 * reach
        t_min, t0v, dt_det = 0.0, torch.linalg.vector_norm(pos, dim=1) - reach, span / nb
    elif c["motion"] == "gyration":
        # charges turning about a uniform field (Boris steps), all around them a far cap
        dist, dt = 200.0, 0.05
        u0 = torch.stack([torch.rand(n, generator=g, **_F64) - 0.5, 1.0 + 2.0 * torch.rand(n, generator=g, **_F64),
                          0.5 * torch.rand(n, generator=g, **_F64)], dim=1)
        x = 0.1 * torch.randn((n, 3), generator=g, **_F64)
        u, q = u0, _charges(n, g)
        pos = _cap(c["rows"], c["cols"], dist, 0.5, 2)
        reach = 5.0 + 0.25 * S * dt
        t_min, dt_det = dist - reach, (S * dt + 2.0 * reach) / nb
    else:
        raise ValueError(c["motion"])
    if q is None:
        q = torch.full((n,), -1.0, **_F64)
    return (x.contiguous(), u.contiguous(), q, 0.0, dt), (pos.contiguous(), t0v, t_min, dt_det, nb)


def _flags(c):
    f = (rd.RD_FAR | rd.RD_FARFIELD) if c["far"] else (rd.RD_NEAR | rd.RD_FAR)
    return f | {"held": 0, "linear": rd.RD_LINEAR, "previous": rd.RD_HOLD_PREV,
                "quadratic": rd.RD_QUADRATIC}[c["interp"]]


def _batch_setups(c, seed):
    """The uneven problems of a batch: kinds and sizes from the case, phases and amplitudes from the seed."""
    sizes = random.Random(c["sizes"])
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    out = []
    for i in range(c["n_problems"]):
        n = max(1, int(round(math.exp(sizes.uniform(math.log(100.0), math.log(5e4))) * c["scale"])))
        S, side = sizes.randint(500, 8000), sizes.choice([32, 64, 128])
        nb, a, b = 16 * side, sizes.random(), sizes.random()
        kind = ("undulator", "circular", "oscillator")[i % 3]
        if kind == "undulator":
            gamma, K, half = 5.0 + 25.0 * a, 0.3 + 1.7 * b, 1.5 / (5.0 + 25.0 * a)
            x, u, dt = _undulator(n, S, gamma, K, 5.0, g)
            bz, w = W.undulator_params(gamma, K)
            pos = _cap(side, side, 1e3, half, 2)
            t_min, dt_det = W.axial_window(1e3, S * dt, bz, math.asin(math.sqrt(2.0) * math.sin(half)),
                                           K / (gamma * w) + 6e-3, nb)
        elif kind == "circular":
            x, u, dt = _circular(n, S, 2.0 + 6.0 * a, 4.0, g)
            pos, span = _cap(side, side, 1e3, 0.6, 2), S * dt + 2.0
            t_min, dt_det = 1e3 - 1.0 - 0.02 * span, 1.04 * span / nb
        else:
            x, u, dt = _oscillators(n, S, g)
            pos, span = _cap(side, side, 1e3, 0.6, 1), S * dt + 6.0
            t_min, dt_det = 1e3 - 3.0 - 0.02 * span, 1.04 * span / nb
        out.append(((x.contiguous(), u.contiguous(), _charges(n, g), 0.0, dt), (pos, None, t_min, dt_det, nb)))
    return out


def _detector(geo, precision="mixed", flags=rd.RD_NEAR | rd.RD_FAR):
    pos, t0v, t_min, dt_det, nb = geo
    return rd.RadiationDetector(pos, t_min, dt_det, nb, t0v, precision, flags)


_GYRO_B, _GYRO_QM = (0.0, 0.0, 1.5), -1.0


def _corrections(shape, seed):
    """FP32 corrections to the positions and momenta (what a fit adjusts), small against a bin."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    return [1e-9 * torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) for _ in range(2)]


def _target(c, geo, seed):
    """A measured field to fit: a smooth oscillating burst in every cell, of the size of the electrons' own."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 78)
    n_pix, nb = geo[0].shape[0], geo[4]
    b = torch.arange(nb, **_F64)[None, :]
    ph = 2.0 * math.pi * torch.rand((n_pix, 1), generator=g, **_F64)
    E = torch.zeros((n_pix, nb, 3), **_F64)
    E[..., 1] = 0.2 * c["n_part"] ** 0.5 * torch.sin(2.0 * math.pi * 10.0 * b / nb + ph)
    E[..., 0] = 0.1 * E[..., 1]
    return E


def _seeds(n_pix, nb, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 79)
    return [torch.randn((n_pix, nb, 3), generator=g, **_F64) for _ in range(2)]


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    if c["path"] == "batch":
        setups = _batch_setups(c, seed)
        return {"case": c, "dets": [_detector(geo) for _, geo in setups], "trajs": [tr for tr, _ in setups]}
    tr, geo = _setup(c, seed)
    s = {"case": c, "tr": tr, "det": _detector(geo, c["precision"], _flags(c))}
    if c["path"] == "fit":
        s["dx"], s["du"] = [d.requires_grad_() for d in _corrections(tr[0].shape, seed)]
        s["target"] = _target(c, geo, seed)
    elif c["path"] == "adjoint":
        s["seeds"] = _seeds(geo[0].shape[0], geo[4], seed)
        s["det"].set_adjoint_mode("compensated")
    elif c["path"] == "stream":
        # the particle code's state arrays
        s["x"], s["u"] = torch.empty_like(tr[0]), torch.empty_like(tr[1])
    return s


def run(state):
    c = state["case"]
    if c["path"] == "batch":
        for d in state["dets"]:
            d.zero()
        rd.deposit_batch(state["dets"], state["trajs"])
        return [d.read("float32", "cuda") for d in state["dets"]]
    det, (x, u, q, t0, dt) = state["det"], state["tr"]
    if c["path"] == "fit":
        state["dx"].grad = state["du"].grad = None
        E, _ = rd.DepositFunction.apply(det, x + state["dx"], u + state["du"], q, t0, dt)
        (0.5 * (E - state["target"]).square().sum()).backward()
        return [state["dx"].grad, state["du"].grad]
    if c["path"] == "adjoint":
        return det.adjoint(x, u, q, t0, dt, *state["seeds"])
    det.zero()
    if c["path"] == "stream":
        det.stream_reset()
        state["x"].copy_(x)
        state["u"].copy_(u)
        done = 0
        # the initial state is sample 0 of the stream; then every stretch as the push finishes it
        det.deposit_stream(x[:, None], u[:, None], q, t0, dt)
        while done < c["n_steps"]:
            m = min(c["stretch"], c["n_steps"] - done)
            xo, uo = rd.rd_push_boris(state["x"], state["u"], m, dt, _GYRO_B, _GYRO_QM)
            det.deposit_stream(xo, uo, q, t0 + (done + 1) * dt, dt)
            done += m
        return det.read("float32", "cuda")
    det.deposit(x, u, q, t0, dt)
    if c["path"] == "spectrum":
        return det.power_spectrum("E")
    return det.read("float64" if c["precision"] == "fp64" else "float32", "cuda")


def work(case):
    c = case
    if c["path"] == "batch":
        sizes, triples, nbytes = random.Random(c["sizes"]), 0, 0
        for _ in range(c["n_problems"]):
            n = max(1, int(round(math.exp(sizes.uniform(math.log(100.0), math.log(5e4))) * c["scale"])))
            S, side = sizes.randint(500, 8000), sizes.choice([32, 64, 128])
            sizes.random(), sizes.random()
            triples += n * S * side * side
            nbytes += 48 * n * (S + 1) + 24 * side * side * 16 * side
        return {"bytes": nbytes, "flops": 75 * triples}
    cells = c["rows"] * c["cols"]
    triples = c["n_part"] * c["n_steps"] * cells
    samples = c["n_part"] * (c["n_steps"] + 1)
    # per triple: the mixed field, arrival increment and held deposit are 75 flops, the plain FP64 form
    # 70, each interpolated field some more; the adjoint recomputes the field and runs its derivative
    flops = {"held": 75, "linear": 95, "previous": 75, "quadratic": 130}[c["interp"]] if c["precision"] == "mixed" else 70
    fields = 24 * cells * c["n_bins"] * (2 if c["precision"] == "fp64" else 1)
    if c["path"] == "spectrum":
        nk = c["n_bins"] // 2 + 1
        return {"bytes": 48 * samples + 4 * cells * nk,
                "flops": 75 * triples + 2 * cells * 5 * c["n_bins"] * math.log2(c["n_bins"])}
    if c["path"] == "fit":
        return {"bytes": 48 * samples * 2 + 24 * samples + 24 * cells * c["n_bins"], "flops": (75 + 230) * triples}
    if c["path"] == "adjoint":
        return {"bytes": 96 * samples + 48 * cells * c["n_bins"], "flops": 1700 * triples}
    return {"bytes": 48 * samples + fields, "flops": flops * triples}


# ------------------------------------------------------------------------------------------------
# the same outputs in 64-bit PyTorch
# ------------------------------------------------------------------------------------------------
_CHUNK = 1 << 23            # (cell, interval) pairs evaluated at once


def _samples(x, u, dt):
    """Per-sample quantities of one particle: x, beta, betadot (backward difference), gamma^-2 for k = 0..S."""
    g2 = 1.0 + (u * u).sum(-1, keepdim=True)
    beta = u / torch.sqrt(g2)
    bd = torch.zeros_like(beta)
    bd[1:] = (beta[1:] - beta[:-1]) / dt
    return beta, bd, 1.0 / g2


def _field_and_arrival(x, beta, bd, ig2, q, pos, T0, t0, dt, dt_det, far):
    """Fields (E, B) of samples 1..S and arrival times (bins) of samples 0..S at the cells pos."""
    t = t0 + dt * torch.arange(x.shape[0], **_F64)
    if far:
        R = torch.sqrt((pos * pos).sum(-1))[:, None]
        n = (pos / R)[:, None, :].expand(-1, x.shape[0], -1)
        a = ((t[None] + R) - (x[None] * n).sum(-1) - T0[:, None]) * (1.0 / dt_det)
    else:
        d = pos[:, None, :] - x[None]
        R = torch.sqrt((d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2])
        n = d / R[..., None]
        a = ((t[None] + R) - T0[:, None]) * (1.0 / dt_det)
        R = R[:, 1:]
    n, b, bd = n[:, 1:], beta[None, 1:], bd[None, 1:]
    nb = n - b
    kap = 0.5 * (ig2[None, 1:, 0] + (nb * nb).sum(-1))
    c1 = (n * bd).sum(-1)
    if not far:
        c1 = c1 + ig2[None, 1:, 0] / R
    E = (q / (kap ** 3 * R))[..., None] * (nb * c1[..., None] - kap[..., None] * bd)
    return torch.cat([E, torch.linalg.cross(n, E, dim=-1)], dim=-1), a


def _overlaps(a, n_bins):
    """(cell, interval, bin, start, end) of every overlap of an arrival interval with a bin of the window."""
    lo, hi = torch.floor(a[:, :-1]), torch.floor(a[:, 1:])
    m = hi - lo
    for i in range(int(m.max().item()) + 1):
        b = lo + i
        cell, k = torch.nonzero((m >= i) & (b >= 0) & (b < n_bins), as_tuple=True)
        if len(cell) == 0:
            continue
        b = b[cell, k]
        yield cell, k, b.long(), torch.maximum(a[cell, k], b), torch.minimum(a[cell, k + 1], b + 1.0)


def _weighted(F, a, cell, k, s, e, interp):
    """Integral over [s, e] of the interpolated field of interval k (0-based: samples k and k + 1)."""
    F1 = F[cell, k]
    if interp == "held":
        return F1 * (e - s)[:, None]
    F0 = F[cell, (k - 1).clamp(min=0)]                  # the first interval holds its own field
    if interp == "previous":
        return F0 * (e - s)[:, None]
    a0 = a[cell, k]
    L = a[cell, k + 1] - a0
    s0, s1 = s - a0, e - a0
    out = F0 * (s1 - s0)[:, None] + (F1 - F0) * ((s1 - s0) * (s1 + s0) / (2.0 * L))[:, None]
    if interp == "quadratic":
        has = (k >= 2).to(torch.float64)
        h = a0 - a[cell, (k - 1).clamp(min=0)]
        h = torch.where(k >= 2, h, torch.ones_like(h))
        Fpp = F[cell, (k - 2).clamp(min=0)]
        D2 = ((F1 - F0) / L[:, None] - (F0 - Fpp) / h[:, None]) / (L + h)[:, None]
        cub = (s1 ** 3 - s0 ** 3) / 3.0 - L * (s1 ** 2 - s0 ** 2) / 2.0
        out = out + D2 * (has * cub)[:, None]
    return out


def _deposit64(tr, geo, far=False, interp="held"):
    """E and B, [n_pix][n_bins][3] each."""
    x, u, q, t0, dt = tr
    pos, t0v, t_min, dt_det, nb = geo
    T0 = t_min + (t0v if t0v is not None else torch.zeros(pos.shape[0], **_F64))
    out = torch.zeros((pos.shape[0] * nb, 6), **_F64)
    step = max(1, _CHUNK // x.shape[1])
    for p in range(x.shape[0]):
        beta, bd, ig2 = _samples(x[p], u[p], dt)
        for j in range(0, pos.shape[0], step):
            F, a = _field_and_arrival(x[p], beta, bd, ig2, q[p], pos[j:j + step], T0[j:j + step], t0, dt, dt_det, far)
            for cell, k, b, s, e in _overlaps(a, nb):
                out.index_add_(0, (j + cell) * nb + b, _weighted(F, a, cell, k, s, e, interp))
    out = out.reshape(pos.shape[0], nb, 6)
    return out[..., :3].contiguous(), out[..., 3:].contiguous()


def _adjoint64(tr, geo, gE, gB):
    """d/dx and d/du of sum(E gE) + sum(B gB) for the held field, by PyTorch's reverse mode."""
    x, u, q, t0, dt = tr
    pos, t0v, t_min, dt_det, nb = geo
    T0 = t_min + (t0v if t0v is not None else torch.zeros(pos.shape[0], **_F64))
    g = torch.cat([gE, gB], dim=-1).reshape(-1, 6)
    gx, gu = torch.zeros_like(x), torch.zeros_like(u)
    step = max(1, _CHUNK // 2 // x.shape[1])
    for p in range(x.shape[0]):
        for j in range(0, pos.shape[0], step):
            xp, up = x[p].detach().requires_grad_(), u[p].detach().requires_grad_()
            beta = up / torch.sqrt(1.0 + (up * up).sum(-1, keepdim=True))
            ig2 = 1.0 / (1.0 + (up * up).sum(-1, keepdim=True))
            bd = torch.cat([torch.zeros_like(beta[:1]), (beta[1:] - beta[:-1]) / dt])
            F, a = _field_and_arrival(xp, beta, bd, ig2, q[p], pos[j:j + step], T0[j:j + step], t0, dt, dt_det, False)
            loss = 0.0
            for cell, k, b, s, e in _overlaps(a.detach(), nb):
                lo, hi = a[cell, k], a[cell, k + 1]
                w = torch.where(e < hi.detach(), e, hi) - torch.where(s > lo.detach(), s, lo)
                loss = loss + (w * (F[cell, k] * g[(j + cell) * nb + b]).sum(-1)).sum()
            if isinstance(loss, float):
                continue
            dx, du = torch.autograd.grad(loss, (xp, up))
            gx[p] += dx
            gu[p] += du
    return gx, gu


def _boris64(x, u, n_steps, dt):
    """Samples 0..n_steps of the Boris push in the uniform field."""
    B = torch.tensor(_GYRO_B, **_F64)
    g = torch.sqrt(1.0 + (u * u).sum(1, keepdim=True))
    t = (0.5 * _GYRO_QM * dt / g) * B
    s = 2.0 * t / (1.0 + (t * t).sum(1, keepdim=True))
    X, U = [x], [u]
    for _ in range(n_steps):
        v = u + torch.linalg.cross(u, t)
        u = u + torch.linalg.cross(v, s)
        x = x + (dt / g) * u
        X.append(x)
        U.append(u)
    return torch.stack(X, dim=1), torch.stack(U, dim=1)


def exact(case, seed):
    c = case
    if c["path"] == "batch":
        if work(c)["flops"] / 75 > 1.5e9:
            return None
        return [_deposit64(tr, geo) for tr, geo in _batch_setups(c, seed)]
    triples = c["n_part"] * c["n_steps"] * c["rows"] * c["cols"]
    if triples > (4e8 if c["path"] in ("fit", "adjoint") else 2e9):
        return None
    tr, geo = _setup(c, seed)
    x, u, q, t0, dt = tr
    if c["path"] == "stream":
        X, U = _boris64(x, u, c["n_steps"], dt)
        return _deposit64((X, U, q, t0, dt), geo)
    if c["path"] == "fit":
        dx, du = _corrections(x.shape, seed)
        tr = (x + dx, u + du, q, t0, dt)
        E, _ = _deposit64(tr, geo)
        return list(_adjoint64(tr, geo, E - _target(c, geo, seed), torch.zeros_like(E)))
    if c["path"] == "adjoint":
        return _adjoint64(tr, geo, *_seeds(geo[0].shape[0], geo[4], seed))
    E, B = _deposit64(tr, geo, c["far"], c["interp"])
    if c["path"] == "spectrum":
        P = torch.zeros((E.shape[0], geo[4] // 2 + 1), **_F64)
        for i in range(3):
            P += torch.fft.rfft(E[..., i], dim=1).abs().square()
        return geo[3] ** 2 * P
    return E, B
