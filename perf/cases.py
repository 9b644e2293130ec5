"""What this library is used for, as calls that can be timed and checked.

A case names a workload by plain values; ``prepare`` makes its inputs from a
seed and the simulator handle a user's program keeps, ``run`` is one pass
through the public entry points, ``exact`` is the same result in FP64 from the
definitions (plain torch, none of the library's arithmetic).

Kinds of case:
  simulate   V for every (LST, channel): ``Simulator.simulate``
  pairs      V for explicit (LST, frequency) pairs: ``Simulator.simulate_pairs``
  unique     one value per redundant baseline group: ``Simulator.simulate_unique``
  update     a forward model in a fitting loop: new fluxes, then V on the host
  learned    ``Simulator.simulate`` with the learned beam in place of per-antenna grids
  gradient   loss and gradient of the learned beam's network on given samples
  train      Adam steps of the learned beam on samples of the gridded beams
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_09763_gb300 import Simulator, synth

C_LIGHT = 299792458.0
DEG = math.pi / 180.0
MINUTE = 2 * math.pi / 1440.0     # one sidereal minute of LST
NU_REF = 150e6
LAT = -30.7 * DEG
DEV = "cuda"

# number of feeds and sky axes of each beam model
_BEAMS = {"gaussian": (1, 1), "scalar": (1, 1), "two": (1, 1), "jones": (2, 2), "stokes": (2, 2)}


def _sim(name, n_ant, n_src, n_t, n_nu, beam="scalar", prec="fp16x3", layout="hex", kind="simulate", lo=100.0,
         hi=200.0, channels="even"):
    return {"name": name, "kind": kind, "n_ant": n_ant, "n_src": n_src, "n_t": n_t, "n_nu": n_nu, "beam": beam,
            "prec": prec, "layout": layout, "lo": lo, "hi": hi, "channels": channels}


def listed():
    return [
        # ten antennas, a thousand sources, an analytic beam, four times: a unit test or a notebook;
        # latency and launches
        _sim("tiny", 10, 1000, 4, 1, beam="gaussian", layout="random", lo=150.0, hi=150.0),
        # one snapshot of a small compact array over 16 channels, the size of a validation run
        _sim("snapshot", 64, 8192, 1, 16),
        # a mid-sized irregular array with two kinds of antenna (bilinear beams), ragged counts, unevenly
        # spaced channels after flagging, a short track of times
        _sim("ragged", 131, 30_001, 5, 7, beam="two", layout="random", channels="odd"),
        # the array the library is made for: 350 antennas x 1e5 point sources x 64 channels, four times
        # of an observation
        _sim("hera", 350, 100_000, 4, 64),
        # the same array in FP32, for users who want no split precision
        _sim("hera_fp32", 350, 100_000, 1, 8, prec="fp32"),
        # random (LST, frequency) pairs over a day: spot checks and sparse schedules, uneven live counts
        _sim("uneven", 350, 100_000, 48, 1, kind="pairs", lo=50.0, hi=250.0),
        # a redundant array that stores one value per group of baselines
        _sim("unique", 350, 100_000, 2, 64, kind="unique"),
        # a diffuse, fully polarised sky of 196,608 pixels with 2 x 2 Jones beams
        _sim("diffuse", 350, 196_608, 2, 4, beam="stokes", lo=140.0, hi=160.0),
        # a fitting loop: new fluxes every pass, V back on the host
        _sim("update", 350, 100_000, 1, 16, kind="update"),
        # one beam per antenna held as a network
        {"name": "learned", "kind": "learned", "n_ant": 350, "n_src": 20_000, "n_t": 1, "n_nu": 2},
        # the network's gradient on given samples (an optimiser of the user's own)
        {"name": "gradient", "kind": "gradient", "n_ant": 64, "batch": 16_384},
        # training of the network on 350 beams, as the quality runs do it
        {"name": "train", "kind": "train", "n_ant": 350, "batch": 16_384, "steps": 40},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["simulate"] * 6 + ["pairs", "pairs", "unique", "unique", "update", "learned", "gradient", "train"])
    if kind == "learned":
        return {"kind": kind, "n_ant": _log(rng, 12, 350), "n_src": _log(rng, 1000, 20_000), "n_t": 1,
                "n_nu": rng.randint(1, 2)}
    if kind == "gradient":
        return {"kind": kind, "n_ant": _log(rng, 4, 64), "batch": 8 * _log(rng, 16, 2048)}
    if kind == "train":
        return {"kind": kind, "n_ant": _log(rng, 12, 350), "batch": 8 * _log(rng, 512, 2048), "steps": rng.randint(16, 40)}
    beam = rng.choice(["scalar"] * 5 + ["gaussian", "two", "jones", "stokes"]) if kind == "simulate" else "scalar"
    prec = "fp32" if kind in ("simulate", "pairs") and rng.random() < 0.2 else "fp16x3"
    layout = "hex" if kind == "unique" or rng.random() < 0.6 else "random"
    n_ant, n_src = _log(rng, 8, 350), _log(rng, 500, 150_000)
    feeds, axes = _BEAMS[beam]
    # at most the work of the 350-antenna case above (its FP32 one for FP32)
    most = 256 * 350 ** 2 * 1e5 if prec == "fp16x3" else 16 * 350 ** 2 * 1e5
    count = max(1, min(256, int(most / (max(feeds * n_ant, 64) ** 2 * axes * n_src))))
    count = max(1, _log(rng, 1, count))
    n_t = max(1, min(count, _log(rng, 1, 12)))
    n_nu = max(1, count // n_t)
    if kind == "pairs":
        n_t, n_nu = max(1, min(count, 96)), 1
    lo = rng.uniform(102.0, 140.0)
    return {"kind": kind, "n_ant": n_ant, "n_src": n_src, "n_t": n_t, "n_nu": n_nu, "beam": beam, "prec": prec,
            "layout": layout, "lo": lo, "hi": rng.uniform(lo + 5.0, 198.0),
            "channels": rng.choice(["even", "even", "odd"])}


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _u(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _sky(case, seed):
    """Positions, fluxes and spectral indices; Stokes Q, U, V where the sky is polarised."""
    g, n = _gen(seed, 1), case["n_src"]
    if case.get("beam") == "stokes" and n % 12 == 0 and math.isqrt(n // 12) ** 2 * 12 == n:
        theta, phi = synth.healpix_ring_pix2ang(math.isqrt(n // 12))   # pixel centres of a diffuse sky
        ra, dec = torch.tensor(phi, device=DEV), torch.tensor(np.pi / 2 - theta, device=DEV)
    else:
        ra, dec = 2 * math.pi * _u(g, n), torch.asin(2 * _u(g, n) - 1)
        if case["kind"] == "pairs":   # part of the catalogue clustered: live counts that vary over the day
            m = n // 2
            ra[:m] = torch.remainder(math.pi / 2 + 0.3 * torch.randn(m, generator=g, device=DEV, dtype=torch.float64), 2 * math.pi)
            dec[:m] = LAT + 0.2 * (2 * _u(g, m) - 1)
    if case.get("beam") == "stokes":
        # smooth log-normal brightness: a sum of plane waves with a falling spectrum
        s = torch.stack([torch.cos(dec) * torch.cos(ra), torch.cos(dec) * torch.sin(ra), torch.sin(dec)])
        f = [torch.zeros_like(ra) for _ in range(3)]
        for k in range(24):
            for h in range(3):
                d = torch.randn(3, generator=g, device=DEV, dtype=torch.float64)
                f[h] += torch.cos((k + 1) * (d / d.norm()) @ s + 2 * math.pi * _u(g, 1)) * (k + 1) ** -0.8
        f = [(x - x.mean()) / x.std() for x in f]
        flux = torch.exp(f[0] - 0.5)
        flux *= 1e3 / flux.sum()
        chi = f[1] * 1.5
        quv = torch.stack([0.2 * flux * torch.cos(2 * chi), 0.2 * flux * torch.sin(2 * chi),
                           0.01 * flux * f[2].clamp(-1, 1)])
        return ra, dec, flux, torch.full_like(ra, -2.5), quv
    a, b = 0.01 ** -0.6, 100.0 ** -0.6      # dN/dS ~ S^-1.6 on [0.01, 100] Jy
    flux = (a + _u(g, n) * (b - a)) ** (-1 / 0.6)
    alpha = -0.8 + 0.2 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    return ra, dec, flux, alpha, None


def _array(case, seed):
    n = case["n_ant"]
    if case.get("layout", "hex") == "hex":
        return synth.hex_array(n, 14.6)
    g = _gen(seed, 2)
    side = 50.0 if n <= 16 else 14.6 * math.sqrt(n) * 1.2
    enu = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    enu[:, :2] = side * (_u(g, n, 2) - 0.5)
    enu[:, 2] = 2.0 * (_u(g, n) - 0.5)
    return enu.cpu().numpy()


def _axes(nu, n_za, n_az):
    za = torch.arange(n_za, device=DEV, dtype=torch.float64) * (math.pi / 2 / (n_za - 1))
    az = torch.arange(n_az, device=DEV, dtype=torch.float64) * (2 * math.pi / n_az)
    return torch.meshgrid(nu, za, az, indexing="ij")


def _ripple(za, az, x, g):
    """Smooth seeded ripple within [-1, 1], regular at the zenith."""
    r = torch.zeros(torch.broadcast_shapes(za.shape, az.shape, x.shape), device=DEV, dtype=torch.float64)
    p = _u(g, 4, 6).tolist()
    for m in range(4):
        r += (0.5 * p[m][0] - 0.25) * torch.sin(za) ** m * torch.cos(m * az + 6.28 * p[m][1]) * \
            torch.cos((0.5 + 2.5 * p[m][2]) * za) * torch.cos((0.5 + 3.5 * p[m][3]) * x + 6.28 * p[m][4])
    return r


def _dipole(za, az):
    j = torch.zeros((2, 2) + tuple(za.shape), device=DEV, dtype=torch.float64)
    j[0, 0], j[0, 1] = torch.cos(za) * torch.sin(az), torch.cos(az)
    j[1, 0], j[1, 1] = torch.cos(za) * torch.cos(az), -torch.sin(az)
    return j


def _beam(case, seed):
    """("gaussian", fwhm) or ("grid", values, nu0, dnu, dza, daz)."""
    g, kind = _gen(seed, 3), case.get("beam", "network")
    if kind == "gaussian":
        return ("gaussian", (8.0 + 4.0 * float(_u(g, 1))) * DEG)
    if kind == "network":      # one dipole per antenna with displaced feeds, coarse grids
        n_za, n_az, nu0, dnu, n_nu = 31, 72, 143e6, 1.75e6, 9
        nu, za, az = _axes(nu0 + dnu * torch.arange(n_nu, device=DEV, dtype=torch.float64), n_za, n_az)
        env = torch.exp(-4 * math.log(2) * za ** 2 / (30 * DEG * NU_REF / nu) ** 2)
        base = _dipole(za, az) * env
        s = torch.stack([torch.sin(za) * torch.sin(az), torch.sin(za) * torch.cos(az), torch.cos(za)], -1)
        out = torch.empty((case["n_ant"],) + tuple(base.shape), dtype=torch.complex64, device=DEV)
        for a, d in enumerate(0.04 * (_u(g, case["n_ant"], 3) - 0.5)):
            ph = -2 * math.pi * (nu / C_LIGHT) * (s @ d)
            out[a] = base * torch.polar(torch.ones_like(ph), ph)
        return ("grid", out.cpu().numpy(), nu0, dnu, math.pi / 2 / (n_za - 1), 2 * math.pi / n_az)
    n_za, n_az = (46, 120) if kind == "two" else (91, 360)
    nu0 = math.floor(case["lo"] - 2.0) * 1e6
    n_nu = int(math.ceil(case["hi"] + 2.0) - math.floor(case["lo"] - 2.0)) + 1
    nu, za, az = _axes(nu0 + 1e6 * torch.arange(n_nu, device=DEV, dtype=torch.float64), n_za, n_az)
    x = (nu - NU_REF) / NU_REF
    if kind in ("jones", "stokes"):
        env = torch.exp(-4 * math.log(2) * za ** 2 / (30 * DEG * NU_REF / nu) ** 2) * (1 + 0.05 * _ripple(za, az, x, g))
        ph = 0.1 * _ripple(za, az, x, g)
        v = (_dipole(za, az) * env * torch.polar(torch.ones_like(ph), ph)).to(torch.complex64)[None]
    else:
        v = []
        for width in ((10.0, 13.0) if kind == "two" else (10.0,)):
            env = torch.exp(-4 * math.log(2) * za ** 2 / (width * DEG * NU_REF / nu) ** 2)
            ph = (0.3 if kind == "two" else 0.0) * za ** 2
            v.append(torch.polar(env * (1 + 0.05 * _ripple(za, az, x, g)), ph))
        v = torch.stack(v).to(torch.complex64)[:, None, None]
    return ("grid", v.cpu().numpy(), nu0, 1e6, math.pi / 2 / (n_za - 1), 2 * math.pi / n_az)


def _when(case, seed):
    """LSTs and frequencies (of equal length for pairs)."""
    g = _gen(seed, 4)
    lst0 = 2 * math.pi * float(_u(g, 1))
    if case["kind"] in ("learned", "gradient", "train"):
        return lst0 + np.arange(case.get("n_t", 1)) * MINUTE, 149.3e6 + 1e6 * np.arange(case.get("n_nu", 1))
    lo, hi = case["lo"] * 1e6, case["hi"] * 1e6
    if case["kind"] == "pairs":
        return (2 * math.pi * _u(g, case["n_t"])).cpu().numpy(), (lo + (hi - lo) * _u(g, case["n_t"])).cpu().numpy()
    f = lo + (np.arange(case["n_nu"]) + 0.5) * ((hi - lo) / case["n_nu"])
    if case["channels"] == "odd":
        f = np.sort((lo + (hi - lo) * _u(g, case["n_nu"])).cpu().numpy())
    return lst0 + np.arange(case["n_t"]) * MINUTE, f


def _beam_idx(case):
    if case["kind"] in ("learned", "gradient", "train"):
        return np.arange(case["n_ant"], dtype=np.int32)
    return (np.arange(case["n_ant"]) % 3 == 0).astype(np.int32) if case["beam"] == "two" else None


def _samples(case, seed):
    g, n = _gen(seed, 5), case["batch"]
    beam = torch.randint(0, case["n_ant"], (n,), generator=g, device=DEV).to(torch.int32)
    nu = 145e6 + 9e6 * _u(g, n)
    t = torch.randn(n, 8, generator=g, device=DEV, dtype=torch.float32) * 0.5
    return [x.cpu().numpy() for x in (beam, 2 * math.pi * _u(g, n), math.pi / 2 * _u(g, n), nu, t)]


def prepare(case, seed):
    kind = case["kind"]
    beam = _beam(case, seed)
    s = {"case": case, "sim": Simulator(0, interp="bilinear" if case.get("beam") == "two" else "cubic")}
    sim = s["sim"]
    lsts, freqs = s["lsts"], s["freqs"] = _when(case, seed)
    sim.set_beam(beam)
    sim.set_antennas(_array(case, seed), _beam_idx(case), LAT)
    if kind in ("learned", "gradient", "train"):
        sim.surrogate_create(seed=1 + seed % 1_000_003)
    if kind == "gradient":
        s["samples"] = _samples(case, seed)
        return s
    if kind == "train":
        s["start"], s["seed"] = sim.surrogate_params()[0], 7 + seed % 1_000_003
        return s
    ra, dec, flux, alpha, quv = (None if x is None else x.cpu().numpy() for x in _sky(case, seed))
    s["sky"] = (ra, dec, flux, alpha)
    sim.init_sky(ra, dec, flux, alpha, NU_REF)
    if quv is not None:
        sim.set_sky_polarisation(quv)
    if kind == "learned":
        sim.set_beam_surrogate(True)
    N = sim.n_feed * sim.n_ant
    shape = (lsts.size, freqs.size, N, N)
    if kind == "pairs":
        shape = (lsts.size, N, N)
    elif kind == "unique":
        shape = (lsts.size, freqs.size, sim.set_redundancy(1e-3), sim.n_feed, sim.n_feed)
    if kind == "update":
        s["V"] = torch.empty(shape, dtype=torch.complex64, pin_memory=True)
    else:
        s["V"] = torch.empty(shape, dtype=torch.complex64, device=DEV)
    return s


def run(s):
    case, sim = s["case"], s["sim"]
    kind = case["kind"]
    if kind == "gradient":
        g, loss = sim.surrogate_grad(*s["samples"])
        return {"gradient": g, "loss": loss}
    if kind == "train":
        sim.surrogate_set_params(s["start"])
        first, last = sim.surrogate_train(case["steps"], case["batch"], 1e-3, 1e-4, s["seed"])
        return {"parameters": sim.surrogate_params()[0], "losses": [first, last]}
    prec = case.get("prec", "fp16x3")
    if kind == "pairs":
        return sim.simulate_pairs(s["lsts"], s["freqs"], prec, out=s["V"])
    if kind == "unique":
        return sim.simulate_unique(s["lsts"], s["freqs"], prec, out=s["V"])
    if kind == "update":
        ra, dec, flux, alpha = s["sky"]
        sim.init_sky(ra, dec, flux, alpha, NU_REF)
        return sim.simulate(s["lsts"], s["freqs"], prec, out=s["V"], host=True)
    return sim.simulate(s["lsts"], s["freqs"], prec, out=s["V"])


# -------------------------------------------------------------------- work

_NET = 2 * (144 * 256 + 3 * 256 * 256 + 256 * 8)      # operations of the network at one point


def work(case):
    kind = case["kind"]
    if kind == "gradient":
        n = case["batch"]
        return {"bytes": n * (4 + 3 * 8 + 8 * 4) + 2 * 4 * (_NET / 2), "flops": 3.0 * n * _NET}
    if kind == "train":
        n = case["batch"] * case["steps"]
        # 64 taps of 4 complex components per sample; parameters, moments read and written per step
        return {"bytes": n * 64.0 * 32 + case["steps"] * 24.0 * (_NET / 2), "flops": 3.0 * n * _NET}
    feeds, axes = (2, 2) if kind == "learned" else _BEAMS[case["beam"]]
    N, live = feeds * case["n_ant"], case["n_src"] / 2
    inst = case["n_t"] * case["n_nu"]
    out = N * N
    if kind == "unique":
        out = _groups(synth.hex_array(case["n_ant"], 14.6))[0].size
    # the lower triangle of V = Z Z^H in real operations, or only the stored values of it
    flops = inst * live * axes * (8.0 * out if kind == "unique" else 4.0 * N * N)
    if kind == "learned":
        flops += inst * live * case["n_ant"] * float(_NET)
    return {"bytes": case["n_src"] * (3 * 8 + 8.0) + inst * 8.0 * out, "flops": flops}


# ------------------------------------------------------------------- exact

def _groups(enu):
    """Representatives (a, b) of the redundant groups, a <= b, in lexicographic order."""
    a, b = np.triu_indices(enu.shape[0])
    d = np.rint((enu[a] - enu[b]) / 1e-3).astype(np.int64)
    first = np.where(d[:, 0] != 0, d[:, 0], np.where(d[:, 1] != 0, d[:, 1], d[:, 2]))
    d = np.where((first < 0)[:, None], -d, d)        # a reversed baseline belongs to the same group
    at = np.sort(np.unique(d, axis=0, return_index=True)[1])
    return a[at], b[at]


def _keys(t):
    """Weights of the four nodes about a point at t in [0, 1) (Keys 1981, a = -1/2)."""
    def h(x):
        x = x.abs()
        return torch.where(x <= 1, (1.5 * x - 2.5) * x * x + 1, torch.where(x < 2, ((-0.5 * x + 2.5) * x - 4) * x + 2, 0 * x))
    return torch.stack([h(t + 1), h(t), h(1 - t), h(2 - t)])


def _interpolate(plane, za, az, dza, daz, cubic, sign):
    """Beam components [c, za, az] at points (za, az): reflected at the zenith, periodic in az."""
    nz, na = plane.shape[-2:]
    uz, ua = za / dza, az / daz
    fz, fa = torch.floor(uz), torch.floor(ua)
    wz = _keys(uz - fz) if cubic else torch.stack([1 - (uz - fz), uz - fz])
    wa = _keys(ua - fa) if cubic else torch.stack([1 - (ua - fa), ua - fa])
    z0, a0 = fz.long() - (1 if cubic else 0), fa.long() - (1 if cubic else 0)
    flat = plane.reshape(plane.shape[0], nz * na)
    out = 0
    for i in range(wz.shape[0]):
        row = z0 + i
        below = row < 0
        r = torch.where(below, -row, row).clamp(max=nz - 1)
        w = torch.where(below, sign * wz[i], wz[i])
        for j in range(wa.shape[0]):
            col = torch.remainder(a0 + j + below.long() * (na // 2), na)
            out = out + flat[:, r * na + col] * (w * wa[j])
    return out


def _network(sim, n_ant):
    """The learned beam's parameters as FP64 tensors: (list of [W, b], embedding, B), and where they lie."""
    p, B, lay = sim.surrogate_params()
    p = torch.tensor(p, device=DEV, dtype=torch.float64)
    layers = []
    for l in range(5):
        kin, out = (int(lay[-1]) if l == 0 else 256), (8 if l == 4 else 256)
        w, b = int(lay[2 * l]), int(lay[2 * l + 1])
        layers.append((w, (out, kin), b))
    return p, layers, int(lay[-2]), torch.tensor(B, device=DEV, dtype=torch.float64)


def _forward(net, beam, az, za, nu):
    p, layers, emb, B = net
    mid, half = 143e6 + 4 * 1.75e6, 4 * 1.75e6
    x = torch.stack([az / (2 * math.pi), za / (math.pi / 2), (nu - mid) / half], -1)
    ph = 2 * math.pi * (x @ B.T)
    e = p[emb:].reshape(-1, 16)[beam]
    h = torch.cat([torch.sin(ph), torch.cos(ph), e], -1)
    for l, (w, shape, b) in enumerate(layers):
        W = p[w:w + shape[0] * shape[1]].reshape(shape)[:, :h.shape[-1]]
        h = h @ W.T + p[b:b + shape[0]]
        if l < 4:
            h = torch.relu(h)
    return h


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return None
    if kind == "gradient":
        sim = prepare(case, seed)["sim"]
        net = _network(sim, case["n_ant"])
        p = net[0].requires_grad_(True)
        beam, az, za, nu, t = (torch.tensor(x, device=DEV) for x in _samples(case, seed))
        y = _forward(net, beam.long(), az, za, nu)
        loss = ((y - t.double()) ** 2).mean()
        loss.backward()
        return {"gradient": p.grad.cpu().numpy(), "loss": float(loss)}
    lsts, freqs = _when(case, seed)
    if kind == "pairs":
        inst = list(zip(lsts, freqs))
    else:
        inst = [(t, f) for t in lsts for f in freqs]
    ra, dec, flux, alpha, quv = _sky(case, seed)
    enu = torch.tensor(_array(case, seed), device=DEV)
    idx = _beam_idx(case)
    net = _network(prepare(case, seed)["sim"], case["n_ant"]) if kind == "learned" else None
    beam = None if net else _beam(case, seed)
    grid = torch.tensor(beam[1], device=DEV).to(torch.complex128) if beam and beam[0] == "grid" else None
    feeds, axes = (2, 2) if kind == "learned" else _BEAMS[case["beam"]]
    pairs = _groups(_array(case, seed)) if kind == "unique" else None
    xeq = torch.stack([torch.cos(ra) * torch.cos(dec), torch.sin(ra) * torch.cos(dec), torch.sin(dec)])
    out = []
    for lst, nu in inst:
        sl, cl, sh, ch = math.sin(LAT), math.cos(LAT), math.sin(-lst), math.cos(-lst)
        R = torch.tensor([[sh, ch, 0], [-sl * ch, sl * sh, cl], [cl * ch, -cl * sh, sl]], device=DEV, dtype=torch.float64)
        s = R @ xeq
        up = s[2] > 0
        s = s[:, up]
        az, za = torch.remainder(torch.atan2(s[0], s[1]), 2 * math.pi), torch.atan2(torch.hypot(s[0], s[1]), s[2])
        spec = (nu / NU_REF) ** alpha[up]
        if net:
            A = torch.empty(case["n_ant"], 2, 2, s.shape[1], dtype=torch.complex128, device=DEV)
            for b in range(case["n_ant"]):
                y = _forward(net, torch.full((s.shape[1],), b, device=DEV), az, za, torch.full_like(az, nu))
                A[b] = torch.complex(y[:, 0::2], y[:, 1::2]).T.reshape(2, 2, -1)
        elif grid is None:
            A = torch.exp(-4 * math.log(2) * za ** 2 / beam[1] ** 2).to(torch.complex128)[None, None, None]
        else:
            nb = grid.shape[0]
            u = (nu - beam[2]) / beam[3]
            m = math.floor(u)
            w = _keys(torch.tensor(u - m, dtype=torch.float64, device=DEV))
            plane = (grid[:, :, :, m - 1:m + 3] * w[:, None, None]).sum(3).reshape(nb * feeds * axes, *grid.shape[-2:])
            A = _interpolate(plane, za, az, beam[4], beam[5], case["beam"] != "two", -1.0 if axes == 2 else 1.0)
            A = A.reshape(nb, feeds, axes, -1)
        if quv is None:
            A = A * torch.sqrt(flux[up] * spec)
        else:        # C = M M^H per source, M lower triangular
            I, (Q, U, V) = flux[up], quv[:, up]
            m00 = torch.sqrt(I + Q)
            m10 = torch.complex(U, -V) / m00
            m11 = torch.sqrt((I - Q - m10.abs() ** 2).clamp(min=0))
            A = torch.stack([A[:, :, 0] * m00 + A[:, :, 1] * m10, A[:, :, 1] * m11], 2) * torch.sqrt(spec)
        turns = (nu / C_LIGHT) * (enu @ s)
        ph = torch.polar(torch.ones_like(turns), -2 * math.pi * (turns - torch.round(turns)))
        A = A[torch.tensor(idx, device=DEV).long()] if idx is not None else A
        Z = A.expand(case["n_ant"], feeds, axes, -1) * ph[:, None, None, :]
        Z = Z.reshape(case["n_ant"] * feeds, -1)
        V = Z @ Z.conj().T
        out.append(V if pairs is None else V[torch.tensor(pairs[0], device=DEV), torch.tensor(pairs[1], device=DEV)])
    V = torch.stack(out)
    if kind == "pairs":
        return V
    if kind == "unique":
        return V.reshape(len(lsts), len(freqs), -1, 1, 1)
    return V.reshape(len(lsts), len(freqs), *V.shape[1:])
