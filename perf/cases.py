"""What the performance of this library is measured on: its public entry points, as a
simulation program calls them, over the sizes and options such programs use.

Kinds of work
  step      Handle.step, FP32 integrand: whole Euler steps with the moments of each, from the
            20^3 homogeneous gluon box (launch latency) to 16^3 x 20^3 phase-space cells
  batch     Batch.step: an ensemble of ragged homogeneous boxes in one launch
  collide64 Handle.collision_term in FP64 (the binding's default precision)
  learned   Handle.step with the learned proposal, its parameters given
  drift     Handle.drift: free streaming, with or without the force term
  moments   Handle.moments and Handle.energy_source: the diagnostics of a state
  train     Handle.proposal_train: Adam steps on recorded samples
  infer     Handle.proposal_infer and the per-anchor parameters it gives

The states are those of a run some steps after its start: the closed forms of the
benchmark's workloads (a step in |p|, a spatial bump, exponential tails in every cell) times
one per cent of noise drawn from the seed.  Time steps are 0.0005 and 0.001 fm/c, in the range of
the runs of the paper (5e-5 to 0.01 fm/c).
"""
import math
import random

import numpy as np
import torch

from paper_1912_04457_gb300 import bz

SCALE = 2.0 ** 40
HBARC = 0.1973269804
DEG = (16.0, 6.0, 6.0, 6.0, 6.0, 6.0, 6.0)
ALL, GLUON = 0x7F, 0x01


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _grid(kind, nx, np_, mask, **more):
    c = {"kind": kind, "nx0": nx[0], "nx1": nx[1], "nx2": nx[2], "np0": np_[0], "np1": np_[1], "np2": np_[2],
         "L": 2.0, "mask": mask, "alpha": 0.3, "mass_mode": 0}
    c.update(more)
    return c


def listed():
    one = (1, 1, 1)
    return [
        # the smallest production run: ten steps of a homogeneous gluon box, where launches count
        _grid("step", one, (20, 20, 20), GLUON, name="step_gluon_20", N=64, nsteps=10, dt=0.001, force=False),
        # quark-gluon matter in one cell: 70 (species, term) pairs
        _grid("step", one, (32, 32, 32), ALL, name="step_qgp_32", L=3.0, N=1024, nsteps=1, dt=0.001, force=False),
        # the largest: space-time evolution of a gluon bump
        _grid("step", (16, 16, 16), (20, 20, 20), GLUON, name="step_bump_16x20", N=256, nsteps=1, dt=0.0005,
              force=False),
        # ragged grids on both sides, four species, the force term, a sample count that is no multiple of 32
        _grid("step", (5, 3, 7), (10, 9, 12), 0x17, name="step_ragged_force", N=45, nsteps=4, dt=0.001, force=True),
        # an ensemble of ragged boxes
        {"kind": "batch", "name": "batch_10", "nboxes": 10, "mix": 5, "dt": 0.001, "nsteps": 1},
        # the plain FP64 method, gluons and seven species
        _grid("collide64", one, (20, 20, 20), GLUON, name="collide64_gluon_20", N=64, dt=0.01, sampler=0),
        _grid("collide64", one, (12, 13, 10), ALL, name="collide64_qgp_ragged", N=100, dt=0.01, sampler=0),
        # learned proposals on seven species
        _grid("learned", one, (16, 16, 16), ALL, name="learned_qgp_16", N=256, dt=0.001),
        # free streaming and diagnostics of the largest state
        _grid("drift", (16, 16, 16), (20, 20, 20), GLUON, name="drift_bump_16x20", dt=0.005, force=False),
        _grid("moments", (16, 16, 16), (20, 20, 20), GLUON, name="moments_bump_16x20", dt=0.005),
        # the proposal network: training steps, and its parameters for every anchor
        _grid("train", one, (32, 32, 32), ALL, name="train_16384", records=400000, steps=20, batch=16384, lr=1e-3),
        _grid("infer", one, (16, 16, 16), ALL, name="infer_qgp_16"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _np(rng, lo, hi):
    """Momentum cells per axis: cubes of a run, or ragged; not odd along all three axes."""
    n = _log_int(rng, lo, hi)
    v = [n, n, n] if rng.random() < 0.5 else [max(lo, min(hi, n + rng.randint(-3, 3))) for _ in range(3)]
    if all(k & 1 for k in v):
        v[rng.randrange(3)] += 1
    return tuple(v)


def _mask(rng):
    return rng.choice([GLUON, GLUON, ALL, ALL, 0x13, 0x0F, 0x17])


def _terms(mask):
    """Terms of each active species' equation."""
    return [len(_equation(d, mask)) for d in range(7) if mask >> d & 1]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "collide64", "learned", "drift", "moments", "train", "infer"])
    if kind == "batch":
        return {"kind": "batch", "nboxes": _log_int(rng, 2, 12), "mix": rng.randrange(1000), "dt": 0.001,
                "nsteps": rng.randint(1, 2)}
    mask, L = _mask(rng), rng.choice([2.0, 2.0, 3.0, 2.5])
    one, np_ = (1, 1, 1), _np(rng, 8, 32)
    cells = bin(mask).count("1") * int(np.prod(np_))
    alpha = round(rng.uniform(0.2, 0.4), 3)
    if kind in ("step", "drift", "moments"):
        nx = one
        if kind == "drift" or rng.random() < 0.5:
            top = max(2.0, (3.2e7 / cells) ** (1 / 3))
            n = math.exp(rng.uniform(math.log(2.0), math.log(min(16.0, top))))
            nx = tuple(max(1, min(16, int(n) + rng.choice([0, 0, 1, -1]))) for _ in range(3))
        cells *= int(np.prod(nx))
        c = _grid(kind, nx, np_, mask, L=L, alpha=alpha, dt=rng.choice([0.0005, 0.001]))
        if kind != "moments":
            c["force"] = rng.random() < 0.3
        if kind == "step":
            c["nsteps"] = rng.choice([1, 2, 3, 5, 10])
            # term evaluations of a call stay below those of a quarter of the largest listed case
            per = c["nsteps"] * int(np.prod(nx)) * int(np.prod(np_)) * sum(_terms(mask))
            c["N"] = _log_int(rng, 8, max(9, min(1024, int(2.0e9 / per))))
            c["mass_mode"] = 1 if rng.random() < 0.15 else 0
        return c
    if kind == "collide64":
        per = int(np.prod(np_)) * sum(_terms(mask))
        return _grid(kind, one, np_, mask, L=L, alpha=alpha, N=_log_int(rng, 16, max(17, min(512, int(2.5e7 / per)))),
                     dt=0.01, sampler=1 if rng.random() < 0.2 else 0)
    if kind == "learned":
        per = int(np.prod(np_)) * sum(_terms(mask))
        return _grid(kind, one, np_, mask, L=L, alpha=alpha, N=_log_int(rng, 16, max(17, min(1024, int(4.0e8 / per)))),
                     dt=0.001)
    if kind == "train":
        return _grid(kind, one, np_, mask, L=L, alpha=alpha, records=_log_int(rng, 5000, 1000000),
                     steps=_log_int(rng, 1, 50), batch=_log_int(rng, 500, 32768), lr=1e-3)
    return _grid(kind, one, np_, mask, L=L, alpha=alpha)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _species(mask):
    return [s for s in range(7) if mask >> s & 1]


def _momenta(np_, L):
    axes = [-L + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * (2.0 * L / n) for n in np_]
    return torch.stack([g.reshape(-1) for g in torch.meshgrid(*axes, indexing="ij")])


def _state(nx, np_, L, mask, seed, dx=0.2, f0=0.5, qs=1.0):
    """int64 state N_s f 2^40, [slot][x][p]."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    p = (_momenta(np_, L) ** 2).sum(0).sqrt()
    axes = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5 - n / 2.0) * dx for n in nx]
    r2 = sum(g.reshape(-1) ** 2 for g in torch.meshgrid(*axes, indexing="ij"))
    bump = 1.0 + 0.3 * torch.exp(-r2 / (2.0 * 0.8 ** 2))
    out = []
    for s in _species(mask):
        f = torch.exp(-p / 0.4) * (0.02 if s == 0 else 0.05) + (f0 * (p < qs) if s == 0 else 0.0)
        f = bump[:, None] * f[None, :]
        f *= 1.0 + 0.01 * (2.0 * torch.rand(f.shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0)
        out.append(torch.round(f * (DEG[s] * SCALE)).to(torch.int64))
    return torch.stack(out).reshape(-1).contiguous()


def _shape(case):
    return ((case["nx0"], case["nx1"], case["nx2"]), (case["np0"], case["np1"], case["np2"]))


def _handle(case, seed):
    nx, np_ = _shape(case)
    return bz.Handle(nx=nx, dx=0.2, np_=np_, L=case["L"], seed=1000 + seed, species_mask=case["mask"],
                     alpha_s=case["alpha"], mass_mode=case["mass_mode"])


def _boxes(case):
    """The boxes of an ensemble: grids, species, couplings, initial states and sample counts from `mix`."""
    rng = random.Random(case["mix"])
    boxes = []
    for i in range(case["nboxes"]):
        n = rng.choice([12, 12, 16, 16, 20, 24])
        np_ = (n, n, n) if rng.random() < 0.7 else (n, n + rng.choice([-2, -1, 1, 3]), n)
        boxes.append({"np_": np_, "L": 2.0, "species_mask": ALL if rng.random() < 0.5 else GLUON,
                      "nsamples": rng.randint(256, 640), "alpha_s": rng.uniform(0.2, 0.4), "mass_mode": 0,
                      "box_id": i, "Qs": rng.uniform(0.8, 1.5), "f0": rng.uniform(0.1, 1.0)})
    return boxes


def _proposal(ncell, seed):
    """Per-anchor proposal parameters in the range a trained network gives."""
    rng = np.random.default_rng(seed + 101)
    prm = np.zeros((ncell, 8), dtype=np.float32)
    prm[:, 0:3] = rng.uniform(-0.4, 0.4, (ncell, 3))
    prm[:, 3] = rng.uniform(0.15, 0.5, ncell)
    prm[:, 4] = rng.uniform(0.15, 0.5, ncell)
    prm[:, 5] = rng.uniform(0.1, 0.4, ncell)
    return prm


def _network(seed):
    """Weights of the 9 -> 128 -> 128 -> 6 network, flat (W1[16][128], b1, W2[128][128], b2, W3[128][8], b3)."""
    rng = np.random.default_rng(seed + 11)
    W1, W3 = np.zeros((16, 128)), np.zeros((128, 8))
    W1[:9] = rng.uniform(-1, 1, (9, 128)) * math.sqrt(6.0 / 137)
    W2 = rng.uniform(-1, 1, (128, 128)) * math.sqrt(6.0 / 256)
    W3[:, :6] = rng.uniform(-1, 1, (128, 6)) * math.sqrt(6.0 / 134)
    b = [rng.uniform(-0.1, 0.1, 128), rng.uniform(-0.1, 0.1, 128), np.zeros(8)]
    b[2][:6] = rng.uniform(-0.1, 0.1, 6)
    return np.concatenate([W1.ravel(), b[0], W2.ravel(), b[1], W3.ravel(), b[2]]).astype(np.float32)


def _records(case, seed):
    """Training records (anchor, w, y[5]) in anchor order, as the recorder leaves them: float32 view [n][8]."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 104729 + 3)
    nx, np_ = _shape(case)
    n = case["records"]
    ncell = bin(case["mask"]).count("1") * int(np.prod(np_))
    a = torch.randint(0, ncell, (n,), generator=gen, device="cuda").sort().values
    w = torch.exp(2.0 * torch.randn(n, generator=gen, device="cuda"))
    y = (0.45 * torch.randn(n, 5, generator=gen, device="cuda")).clamp_(-0.999, 0.999)
    rec = torch.empty(n, 8, dtype=torch.float32, device="cuda")
    rec[:, 0:2] = a.view(torch.float32).reshape(n, 2)
    rec[:, 2] = w
    rec[:, 3:8] = y
    return rec


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed}
    if kind == "batch":
        boxes = [dict(b, seed=1000 + seed) for b in _boxes(case)]
        s["state0"] = torch.cat([_state((1, 1, 1), b["np_"], b["L"], b["species_mask"], 100 * seed + i, f0=b["f0"],
                                        qs=b["Qs"]) for i, b in enumerate(boxes)])
        s["batch"] = bz.Batch(boxes)
        s["state"] = torch.empty_like(s["state0"])
        s["moments"] = torch.empty(case["nsteps"] * s["batch"].nslots_total * 5, dtype=torch.float64, device="cuda")
        return s
    nx, np_ = _shape(case)
    h = s["h"] = _handle(case, seed)
    if kind in ("step", "drift", "moments", "collide64", "learned"):
        s["state0"] = _state(nx, np_, case["L"], case["mask"], seed)
    if kind == "step":
        h.set_force_term(case["force"])
        s["state"] = torch.empty_like(s["state0"])
        s["moments"] = torch.empty(case["nsteps"] * h.nxc * h.nslots * 5, dtype=torch.float64, device="cuda")
    elif kind == "drift":
        h.set_force_term(case["force"])
        s["out"] = torch.empty_like(s["state0"])
    elif kind == "moments":
        s["moments"] = torch.empty(h.nxc * h.nslots * 5, dtype=torch.float64, device="cuda")
        s["source"] = torch.empty(h.nxc * h.nslots * 3, dtype=torch.float64, device="cuda")
    elif kind == "collide64":
        s["A"] = torch.empty_like(s["state0"])
    elif kind == "learned":
        h.set_anchor_params(_proposal(h.ncell, seed))
        h.set_step_sampler(bz.SAMPLER_LEARNED)
        s["state"] = torch.empty_like(s["state0"])
    elif kind == "train":
        s["params"] = _network(seed)
        s["records"] = _records(case, seed).view(torch.uint8).reshape(-1)
        h.set_proposal_params(s["params"])
    elif kind == "infer":
        h.set_proposal_params(_network(seed))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        s["state"].copy_(s["state0"])
        s["h"].step(s["state"], case["dt"], case["nsteps"], case["N"], bz.PREC_F32, step0=0, moments_out=s["moments"])
        # the FP32 integrand's new state, as the particle numbers it stands for
        return {"state": s["state"].double(), "moments": s["moments"]}
    if kind == "batch":
        s["state"].copy_(s["state0"])
        s["batch"].step(s["state"], case["dt"], case["nsteps"], step0=0, moments_out=s["moments"])
        return {"state": s["state"].double(), "moments": s["moments"]}
    if kind == "collide64":
        s["h"].collision_term(s["state0"], s["A"], case["N"], 3, case["dt"], bz.PREC_F64, case["sampler"])
        return s["A"]
    if kind == "learned":
        s["state"].copy_(s["state0"])
        s["h"].step(s["state"], case["dt"], 1, case["N"], bz.PREC_F32, step0=3)
        return s["state"].double()
    if kind == "drift":
        s["h"].drift(s["state0"], s["out"], case["dt"])
        return s["out"]
    if kind == "moments":
        s["h"].moments(s["state0"], s["moments"])
        s["h"].energy_source(s["state0"], case["dt"], out=s["source"])
        return {"moments": s["moments"], "source": s["source"]}
    if kind == "train":
        losses = s["h"].proposal_train(s["records"], case["records"], case["steps"], case["batch"], case["lr"])
        return {"losses": losses, "params": s["h"].proposal_params()}
    s["h"].proposal_infer()
    return s["h"].anchor_params()


# ---------------------------------------------------------------------------
# Work and tolerances
# ---------------------------------------------------------------------------
def _collision_flops(np_, nxc, mask, N):
    """60 operations a sample, 29 a term, 81 an accepted root of which there are 0.36 a term."""
    per = int(np.prod(np_)) * nxc * N
    return per * sum(60 + t * (29 + 0.36 * 81) for t in _terms(mask))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = _boxes(case)
        cells = sum(bin(x["species_mask"]).count("1") * int(np.prod(x["np_"])) for x in b)
        slots = sum(bin(x["species_mask"]).count("1") for x in b)
        return {"bytes": case["nsteps"] * (16 * cells + 40 * slots),
                "flops": case["nsteps"] * sum(_collision_flops(x["np_"], 1, x["species_mask"], x["nsamples"]) for x in b)}
    nx, np_ = _shape(case)
    nxc, slots = int(np.prod(nx)), bin(case["mask"]).count("1")
    cells = slots * nxc * int(np.prod(np_))
    if kind == "step":
        return {"bytes": case["nsteps"] * (16 * cells + 40 * slots * nxc),
                "flops": case["nsteps"] * (_collision_flops(np_, nxc, case["mask"], case["N"]) + 40 * cells)}
    if kind in ("collide64", "learned"):
        return {"bytes": 16 * cells + (32 * cells if kind == "learned" else 0),
                "flops": _collision_flops(np_, nxc, case["mask"], case["N"])}
    if kind == "drift":
        return {"bytes": 16 * cells, "flops": 30 * cells}
    if kind == "moments":
        return {"bytes": 8 * cells + 64 * slots * nxc, "flops": 20 * cells}
    layers = 2 * (9 * 128 + 128 * 128 + 128 * 6)
    if kind == "train":
        return {"bytes": case["steps"] * case["batch"] * 32 + 8 * 19720, "flops": 3 * layers * case["steps"] * case["batch"]}
    return {"bytes": 32 * cells + 4 * 19720, "flops": layers * cells}


def tolerance(case):
    # FP64 deposits, integer fluxes and exact integer sums: the same whole numbers, the same bytes
    return {"collide64": "exact", "drift": "exact", "moments": "exact",
            # FP32 integrand: about four times the largest distance from 64 bits seen (1.8e-4), which a single root's
            # large 1/sqrt(H) can bring into a few cells; the learned sampler draws such roots with small weights
            "step": {"rel": 7e-4, "max": 5e-2}, "batch": {"rel": 7e-4, "max": 5e-2}, "learned": {"rel": 1e-5, "max": 2e-3},
            # BF16 operands, FP32 accumulation
            "train": {"rel": 1e-2, "max": 0.4}, "infer": {"rel": 1e-2, "max": 0.1}}[case["kind"]]


# ---------------------------------------------------------------------------
# The same results in 64-bit torch, from the equations
# ---------------------------------------------------------------------------
def _equation(d, mask):
    """Terms (k1, k2, k3, p = d; symmetry factor; |M|^2 row) of species d's equation with all four legs active."""
    if d == 0:
        t = [(0, 0, 0, 0.5, "gg")]
        for q in (1, 2, 3):
            t += [(q, 0, q, 1.0, "qg"), (q + 3, 0, q + 3, 1.0, "qg"), (q, q + 3, 0, 1.0, "qqbgg")]
    else:
        bar = d + 3 if d < 4 else d - 3
        t = [(d, d, d, 0.5, "qq"), (bar, d, bar, 1.0, "qqb"), (0, 0, bar, 0.5, "qqbgg"), (0, d, 0, 1.0, "qg")]
        for o in (1, 2, 3):
            if o in (d, bar):
                continue
            a, b = (o, o + 3) if d < 4 else (o + 3, o)
            t += [(a, d, a, 1.0, "qqp"), (b, d, b, 1.0, "qqp"), (a, b, bar, 1.0, "qqb2")]
    return [x for x in t if all(mask >> leg & 1 for leg in (x[0], x[1], x[2], d))]


def _msq(row, s, t, u, mg2, alpha):
    g4, dF, CA, CF, dA = (4 * math.pi * alpha) ** 2, 3.0, 3.0, 4.0 / 3.0, 8.0
    A1, A2 = 8 * g4 * dF * dF * CF * CF / dA, 16 * g4 * dF * CF * (CF - CA / 2)
    A3, A4, A5 = 8 * g4 * dF * CF * CF, 8 * g4 * dF * CF * CA, 16 * g4 * dA * CA * CA
    T, U = t - mg2, u - mg2
    if row == "qqp":
        return A1 * (s * s + u * u) / T ** 2
    if row == "qq":
        return A1 * ((s * s + u * u) / T ** 2 + (s * s + t * t) / U ** 2) + A2 * s * s / (T * U)
    if row == "qqb":
        return A1 * ((s * s + u * u) / T ** 2 + (u * u + t * t) / s ** 2) + A2 * u * u / (T * s)
    if row == "qqb2":
        return A1 * (t * t + u * u) / s ** 2
    if row == "qqbgg":
        return A3 * (u / T + t / U) - A4 * (t * t + u * u) / s ** 2
    if row == "qg":
        return A4 * (s * s + u * u) / T ** 2 - A3 * (u / s + s / U)
    return A5 * (3 - s * u / T ** 2 - s * t / U ** 2 - t * u / s ** 2)


def _philox(c0, c1, c2, c3, k0, k1):
    c = [c0 & 0xFFFFFFFF, c1, c2, c3]
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # int64 products modulo 2^64 keep the bits
        c = [(b >> 32 & 0xFFFFFFFF) ^ c[1] ^ k0, b & 0xFFFFFFFF, (a >> 32 & 0xFFFFFFFF) ^ c[3] ^ k1, a & 0xFFFFFFFF]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _mass_slot(s):
    return 0 if s == 0 else 1 + (s - 1) % 3


def _masses(n, p2, meas, mask, alpha, prev):
    """[x][4] thermal masses of n = N_s f 2^40 [slot][x][p]; prev: the previous ones, or None for E = |p|."""
    sp = _species(mask)
    zero = torch.zeros(n.shape[1:], dtype=torch.float64, device="cuda")

    def q(s):
        return n[sp.index(s)] / SCALE if s in sp else zero

    def r(i):
        return 0.5 / (p2[None, :] + (0.0 if prev is None else prev[:, i:i + 1])).sqrt()

    g2, CF = 4 * math.pi * alpha, 4.0 / 3.0
    quarks = [(q(i) + q(i + 3)) * r(i) for i in (1, 2, 3)]
    gl = q(0) * r(0)
    out = [2 * g2 / 8.0 * meas * (9 * gl + 4 * sum(quarks)).sum(1) / 3]
    out += [2 * CF * g2 * meas * (3 * gl + 4 * x).sum(1) / 24 for x in quarks]
    return torch.stack(out, 1)


def _drift(n, nx, np_, L, m2, mask, dt, dx, force):
    sp = _species(mask)
    p = _momenta(np_, L)
    v = n.reshape(len(sp), *nx, -1)
    out = v.clone()
    for i, s in enumerate(sp):
        m = m2[:, _mass_slot(s)].reshape(*nx)
        E = ((p ** 2).sum(0) + m[..., None]).sqrt()
        for d in range(3):
            if nx[d] == 1:
                continue
            flux = v[i] * (p[d] / E).abs() * (dt / dx)
            out[i] += torch.where(p[d] > 0, torch.roll(flux, 1, d), torch.roll(flux, -1, d)) - flux
            if force:
                g = (torch.roll(m, -1, d) - torch.roll(m, 1, d)) / (4 * dx)
                f = (v[i] * (-g[..., None] / E) * (dt / (2 * L / np_[d]))).reshape(*nx, *np_)
                full = out[i].view(*nx, *np_)
                lo = [slice(None)] * 6
                hi = [slice(None)] * 6
                lo[3 + d], hi[3 + d] = slice(0, np_[d] - 1), slice(1, None)
                face = f[tuple(lo)].clamp(min=0) + f[tuple(hi)].clamp(max=0)  # through the faces inside the box
                full[tuple(lo)] -= face
                full[tuple(hi)] += face
    return out.reshape(len(sp), -1, v.shape[-1])


def _collision(n, nxc, np_, L, mask, m2, massless, alpha, N, step, dt, key, prop=None, chunk=1 << 21):
    """Increment of n over dt (no rounding to whole numbers), from the 23-bit uniforms of the FP32 path."""
    sp = _species(mask)
    npc = int(np.prod(np_))
    f = (n / SCALE / torch.tensor([DEG[s] for s in sp], dtype=torch.float64, device="cuda")[:, None, None]).reshape(-1)
    A = torch.zeros_like(f)
    dp = [2 * L / k for k in np_]
    K = (2 * L) ** 5 * dt / (4.0 * N) / HBARC * SCALE
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    u23 = lambda w: ((w >> 9).double() + 0.5) / 8388608.0  # noqa: E731
    cell = lambda k, d: ((k + L) / dp[d]).floor().long().clamp(0, np_[d] - 1)  # noqa: E731
    inside = lambda k: (k >= -L) & (k < L)  # noqa: E731
    lin = lambda x, y, z: (cell(x, 0) * np_[1] + cell(y, 1)) * np_[2] + cell(z, 2)  # noqa: E731
    per = max(1, chunk // N)
    for slot, d in enumerate(sp):
        terms = _equation(d, mask)
        for a0 in range(0, nxc * npc, per):
            a = torch.arange(a0, min(nxc * npc, a0 + per), device="cuda").repeat_interleave(N)
            smp = torch.arange(N, device="cuda").repeat(len(a) // N)
            x, j = a // npc, a % npc
            c3 = torch.full_like(a, step << 3 | d)
            r0, r1 = _philox(2 * smp, j, x, c3, k0, k1), _philox(2 * smp + 1, j, x, c3, k0, k1)
            jv = (j // (np_[1] * np_[2]), j // np_[2] % np_[1], j % np_[2])
            p = [-L + (jv[i] + 0.5) * dp[i] + dp[i] * (u23(r0[i]) - 0.5) for i in range(3)]
            uv = [u23(w) for w in (r0[3], r1[0], r1[1], r1[2], r1[3])]
            wf = 1.0
            if prop is None:
                k = [-L + 2 * L * u for u in uv]
            else:
                r2 = _philox(0x80000000 | smp, j, x, c3, k0, k1)
                prm = prop[slot * nxc * npc + a]
                uni = u23(r2[0]) < prm[:, 5]
                tail = lambda z: 1 / ((2 + z * z).sqrt() * ((2 + z * z).sqrt() + z.abs()))  # noqa: E731
                k, G = [], 1.0
                for i in range(5):
                    mu = torch.zeros_like(uv[0]) if i < 2 else prm[:, i - 2]
                    sg = prm[:, 4] if i < 2 else prm[:, 3]
                    Fa, cFb = tail((-1 - mu) / sg), tail((1 - mu) / sg)
                    D = 1 - cFb - Fa
                    vv, cv = Fa + uv[i] * D, cFb + (1 - uv[i]) * D
                    t2 = 2 * vv * cv
                    y = torch.where(uni, 2 * uv[i] - 1, (mu + sg * (vv - cv) / t2.sqrt()).clamp(-1, 0.99999994))
                    G = G * torch.where(uni, (2 + ((y - mu) / sg) ** 2) ** -1.5, t2 * t2.sqrt()) / (sg * D)
                    k.append(L * y)
                wf = 1 / (32 * (prm[:, 5] / 32 + (1 - prm[:, 5]) * G))
            b = [p[0] + k[2] - k[0], p[1] + k[3] - k[1]]
            keep = (inside(b[0]) & inside(b[1])).nonzero().reshape(-1)
            p, k, b = ([v[keep] for v in w] for w in (p, k, b))
            x, j = x[keep], j[keep]
            wf = wf if prop is None else wf[keep]
            m = m2[x]
            md = torch.zeros_like(m) if massless else m
            Pz = p[2] + k[4]
            PP = (p[0] + k[2]) ** 2 + (p[1] + k[3]) ** 2 + Pz ** 2
            l3 = lin(k[2], k[3], k[4])
            for la, lb, lc, sym, row in terms:
                ma, mb, mc, me = (md[:, _mass_slot(s)] for s in (la, lb, lc, d))
                Ep = (p[0] ** 2 + p[1] ** 2 + p[2] ** 2 + me).sqrt()
                E3 = (k[2] ** 2 + k[3] ** 2 + k[4] ** 2 + mc).sqrt()
                E = Ep + E3
                a2, b2 = k[0] ** 2 + k[1] ** 2 + ma, b[0] ** 2 + b[1] ** 2 + mb
                D = E * E - Pz * Pz
                kap = (E * E + a2 - b2 - Pz * Pz) / 2
                H = kap * kap - a2 * D
                sq = E * H.clamp(min=0).sqrt()
                Q = torch.where(kap * Pz >= 0, kap * Pz + sq, kap * Pz - sq)
                for z in (Q / D, (E * E * a2 - kap * kap) / Q):
                    e1 = (kap + Pz * z) / E
                    E1, dz = (a2 + z * z).sqrt(), Pz - z
                    E2 = (b2 + dz * dz).sqrt()
                    s = E * E - PP
                    t = ma + mc - 2 * (E1 * E3 - (k[0] * k[2] + k[1] * k[3] + z * k[4]))
                    u = ma + me - 2 * (E1 * Ep - (k[0] * p[0] + k[1] * p[1] + z * p[2]))
                    mg2 = m[:, 0]
                    i = ((H > 0) & (D > 0) & (e1 > 0) & (e1 < E) & inside(z) & inside(dz) & (s > 0) & (t < mg2)
                         & (u < mg2)).nonzero().reshape(-1)
                    if not len(i):
                        continue
                    M = _msq(row, s[i], t[i], u[i], mg2[i], alpha)
                    base = x[i] * npc
                    cells = [sp.index(la) * nxc * npc + base + lin(k[0][i], k[1][i], z[i]),
                             sp.index(lb) * nxc * npc + base + lin(b[0][i], b[1][i], dz[i]),
                             sp.index(lc) * nxc * npc + base + l3[i], slot * nxc * npc + base + j[i]]
                    F = [f[c] for c in cells]
                    st = [1 + v if leg == 0 else 1 - v for v, leg in zip(F, (la, lb, lc, d))]
                    W = F[0] * F[1] * st[2] * st[3] - st[0] * st[1] * F[2] * F[3]
                    J = (z[i] / E1[i] - dz[i] / E2[i]).abs()
                    w = sym * W * M / (J * (2 * math.pi) ** 5 * 16 * E1[i] * E2[i] * E3[i] * Ep[i]) * K
                    w = w if prop is None else w * wf[i]
                    for c, sign in zip(cells, (-1, -1, 1, 1)):
                        A.index_add_(0, c, sign * w)
    return A.reshape(n.shape)


def _moments(n, np_, L, m2, mask):
    sp = _species(mask)
    p = _momenta(np_, L)
    pref = (2 * L) ** 3 / int(np.prod(np_)) / (2 * math.pi) ** 3 / SCALE
    out = []
    for i, s in enumerate(sp):
        E = ((p ** 2).sum(0) + m2[:, _mass_slot(s), None]).sqrt()
        out.append(torch.stack([n[i].sum(1), (n[i] * E).sum(1)] + [n[i] @ p[d] for d in range(3)], 1) * pref)
    return torch.stack(out, 1)  # [x][slot][5]


def _run64(state0, nx, np_, L, mask, alpha, massless, N, nsteps, dt, force, key):
    n = state0.double().reshape(bin(mask).count("1"), int(np.prod(nx)), int(np.prod(np_)))
    p2 = (_momenta(np_, L) ** 2).sum(0)
    meas = (2 * L) ** 3 / int(np.prod(np_)) / (2 * math.pi) ** 3
    m2, moments = None, []
    for k in range(nsteps):
        m2 = _masses(n, p2, meas, mask, alpha, None if massless else m2)
        disp = torch.zeros_like(m2) if massless else m2
        inc = _collision(n, int(np.prod(nx)), np_, L, mask, m2, massless, alpha, N, k, dt, key)
        n = _drift(n, nx, np_, L, disp, mask, dt, 0.2, force and not massless) + inc
        moments.append(_moments(n, np_, L, disp, mask))
    return n.reshape(-1), torch.stack(moments).reshape(-1)


def _features(a, np_, L, mask):
    npc = int(np.prod(np_))
    sp = torch.tensor(_species(mask), device="cuda")
    d = sp[a // npc]
    p = (_momenta(np_, L) / L).t()[a % npc]
    pp = (p ** 2).sum(1, keepdim=True)
    one = torch.ones_like(pp)
    kinds = [((d >= lo) & (d <= hi)).double()[:, None] for lo, hi in ((0, 0), (1, 3), (4, 6))]
    return torch.cat([p, pp.sqrt(), pp] + kinds + [one], 1)


def _net(theta, X):
    W1, b1 = theta[:2048].reshape(16, 128)[:9], theta[2048:2176]
    W2, b2 = theta[2176:18560].reshape(128, 128), theta[18560:18688]
    W3, b3 = theta[18688:19712].reshape(128, 8), theta[19712:]
    silu = torch.nn.functional.silu
    o = silu(silu(X @ W1 + b1) @ W2 + b2) @ W3 + b3
    return torch.cat([torch.tanh(o[:, :3]), 0.02 + 0.5 * torch.sigmoid(o[:, 3:5]),
                      0.1 + 0.9 * torch.sigmoid(o[:, 5:6])], 1)


def _logq(prm, y):
    G = 1.0
    for i in range(5):
        mu, s = (torch.zeros_like(prm[:, 0]), prm[:, 4]) if i < 2 else (prm[:, i - 2], prm[:, 3])
        F = lambda z: 0.5 + z / (2 * (2 + z * z).sqrt())  # noqa: E731
        G = G * (2 + ((y[:, i] - mu) / s) ** 2) ** -1.5 / (s * (F((1 - mu) / s) - F((-1 - mu) / s)))
    return torch.log(prm[:, 5] / 32 + (1 - prm[:, 5]) * G)


def _signed(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _splitmix_mod(key, count, n):
    """SplitMix64(key + r) mod n for r = 0 .. count - 1 (unsigned)."""
    with np.errstate(over="ignore"):
        z = np.arange(count, dtype=np.uint64) + np.uint64(key & ((1 << 64) - 1)) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z % np.uint64(n)).astype(np.int64)).cuda()


def _train64(case, seed):
    rec = _records(case, seed)
    a = rec[:, 0:2].contiguous().view(torch.int64).reshape(-1)
    w, y = rec[:, 2].double(), rec[:, 3:8].double()
    theta = torch.from_numpy(_network(seed)).cuda().double()
    X = _features(a, _shape(case)[1], case["L"], case["mask"])
    wbar = w.mean()
    m, v, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    for k in range(case["steps"]):
        i = _splitmix_mod(((k + 1) << 32) * 0x9E3779B97F4A7C15, case["batch"], case["records"])
        th = theta.clone().requires_grad_(True)
        loss = -(w[i] * _logq(_net(th, X[i]), y[i])).sum() / (wbar * case["batch"])
        g, = torch.autograd.grad(loss, th)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        theta = theta - case["lr"] * (m / (1 - 0.9 ** (k + 1))) / ((v / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
        losses.append(float(loss))
    return {"losses": np.array(losses), "params": theta}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("collide64", "drift"):
        return None  # whole numbers
    if kind == "batch":
        boxes = _boxes(case)
        if case["nsteps"] * sum(_collision_flops(b["np_"], 1, b["species_mask"], b["nsamples"]) for b in boxes) > 6e10:
            return None
        states, moments = [], []
        for i, b in enumerate(boxes):
            st = _state((1, 1, 1), b["np_"], b["L"], b["species_mask"], 100 * seed + i, f0=b["f0"], qs=b["Qs"])
            n, mom = _run64(st, (1, 1, 1), b["np_"], b["L"], b["species_mask"], b["alpha_s"], False, b["nsamples"],
                            case["nsteps"], case["dt"], False, (1000 + seed) ^ b["box_id"])
            states.append(n)
            moments.append(mom.reshape(case["nsteps"], -1))
        return {"state": torch.cat(states), "moments": torch.cat(moments, 1).reshape(-1)}
    nx, np_ = _shape(case)
    L, mask, alpha, massless = case["L"], case["mask"], case["alpha"], case["mass_mode"] == 1
    if kind == "train":
        return _train64(case, seed) if case["steps"] * case["batch"] < 4e6 else None
    if kind == "infer":
        a = torch.arange(bin(mask).count("1") * int(np.prod(np_)), device="cuda")
        theta = torch.from_numpy(_network(seed)).cuda().double()
        prm = _net(theta, _features(a, np_, L, mask))
        return torch.cat([prm, torch.zeros_like(prm[:, :2])], 1)
    state0 = _state(nx, np_, L, mask, seed)
    slots, nxc, npc = bin(mask).count("1"), int(np.prod(nx)), int(np.prod(np_))
    if kind == "step":
        if case["nsteps"] * _collision_flops(np_, nxc, mask, case["N"]) > 6e10:
            return None
        n, mom = _run64(state0, nx, np_, L, mask, alpha, massless, case["N"], case["nsteps"], case["dt"],
                        case["force"], 1000 + seed)
        return {"state": n, "moments": mom}
    n = state0.double().reshape(slots, nxc, npc)
    p2 = (_momenta(np_, L) ** 2).sum(0)
    m2 = _masses(n, p2, (2 * L) ** 3 / npc / (2 * math.pi) ** 3, mask, alpha, None)
    if kind == "learned":
        if _collision_flops(np_, nxc, mask, case["N"]) > 6e10:
            return None
        prop = torch.from_numpy(_proposal(state0.numel(), seed)).cuda().double()
        inc = _collision(n, nxc, np_, L, mask, m2, massless, alpha, case["N"], 3, case["dt"], 1000 + seed, prop)
        return (n + inc).reshape(-1)
    src = []
    for i, s in enumerate(_species(mask)):
        m = m2[:, _mass_slot(s)]
        I = (n[i] / (p2[None, :] + m[:, None]).sqrt()).sum(1) * (2 * L) ** 3 / npc / (2 * math.pi) ** 3 / SCALE
        src.append(torch.stack([I, torch.zeros_like(I), -0.25 * m * I], 1))
    return {"moments": _moments(n, np_, L, m2, mask).reshape(-1), "source": torch.stack(src, 1).reshape(-1)}
