"""Channels of one call whose beams see the same few sources with very different
strength (needs a GB300): a beam that narrows with frequency and sources 18 to 26
degrees off the zenith, so that |A| falls by up to ten orders of magnitude over the
band.  Every channel keeps its own accuracy, in both forms of the products (few and
many antennas), one and two axes, one beam and several, evenly and unevenly spaced
channels.

Tolerance: the products add at most 1e-5 of max|V| per instance, as in every mode,
which is held against FP32 mode (the same beam values).  Against the oracle comes what
FP32 directions do on so steep a beam: the zenith angle is good to about 2 ulp and its
place in a grid of half degrees to another, 9e-6 of a step, over which |A| changes by
at most a factor e^1.3: 1.2e-5 of A, 2.4e-5 of V; 4e-5 in all."""
import numpy as np
import pytest

import oracle
from helpers import dipole_jones_grid, oracle_problem, rel_err, sample_pairs, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu
TOL, TOL_ORACLE = 1e-5, 4e-5


def workload(n_ant, za_deg, n_chan, beam="scalar", channels="even", n_beam=1, seed=0):
    w = synth.hera_like(n_ant=n_ant, n_src=len(za_deg), n_chan=n_chan, n_times=1, n_za=181, n_az=120)
    g = np.random.default_rng(seed)
    za, az = np.radians(za_deg), g.uniform(0, 2 * np.pi, len(za_deg))
    e, n, u = np.sin(za) * np.sin(az), np.sin(za) * np.cos(az), np.cos(za)
    sl, cl = np.sin(w.lat), np.cos(w.lat)
    w.dec = np.arcsin(sl * u + cl * n)
    w.ra = w.lsts[0] + np.arctan2(e, cl * u - sl * n)
    w.freqs = np.linspace(100.5e6, 199.5e6, n_chan)
    if channels == "odd":
        w.freqs = np.sort(g.uniform(100.5e6, 199.5e6, n_chan))
    if beam == "jones":
        vals = dipole_jones_grid(98e6 + np.arange(105) * 1e6, 181, 120, np.radians(10.0), 150e6, g)
        w.beam = ("grid", vals, 98e6, 1e6, (np.pi / 2) / 180, 2 * np.pi / 120, "cubic")
    if n_beam > 1:
        vals = np.concatenate([w.beam[1] * np.complex64(1 - 0.2j * b) for b in range(n_beam)])
        w.beam = (w.beam[0], vals) + tuple(w.beam[2:])
        w.beam_idx = (np.arange(n_ant) % n_beam).astype(np.int32)
    return w


@pytest.mark.parametrize("n_ant,za,n_chan,beam,channels,n_beam", [
    (40, [22.0], 64, "scalar", "even", 1),
    (40, [25.0], 64, "scalar", "odd", 1),
    (300, [25.0], 64, "scalar", "even", 1),
    (150, [18.0, 21.0, 26.0], 200, "scalar", "even", 1),
    (150, list(np.linspace(20.0, 26.0, 20)), 200, "scalar", "odd", 2),
    (60, [24.0], 64, "jones", "even", 1),
    (130, [19.0, 23.0, 26.0], 64, "jones", "even", 2),
])
def test_every_channel_keeps_its_accuracy(n_ant, za, n_chan, beam, channels, n_beam):
    w = workload(n_ant, za, n_chan, beam, channels, n_beam, seed=n_ant)
    sim = simulator(w)
    V = sim.simulate(w.lsts, w.freqs, "fp16x3").cpu().numpy()[0]
    V32 = sim.simulate(w.lsts, w.freqs, "fp32").cpu().numpy()[0]
    assert sim.last_live_counts(n_chan)[0] == len(za)
    P = oracle_problem(w)
    pa, pb = sample_pairs(n_ant, 100, seed=2)
    nf = V.shape[-1] // n_ant
    worst = {}
    for ic in range(n_chan):
        vo = oracle.vis(P, w.lsts[0], w.freqs[ic], pairs=(pa, pb))
        err = rel_err(V[ic].reshape(n_ant, nf, n_ant, nf)[pa, :, pb, :], vo), rel_err(V[ic], V32[ic])
        if err[0] > TOL_ORACLE or err[1] > TOL:
            worst[ic] = err
    assert not worst


def test_a_channel_out_of_range_leaves_the_others_alone():
    # a spectrum so steep that the last channels overflow FP32: theirs alone are lost.
    # exp(320 ln(nu / nu_ref)) in FP32 has up to 34.5 x 2 roundings of its argument, 4.2e-6,
    # twice in V: 2e-5 with the mode's own 1e-5
    w = workload(30, [5.0, 9.0], 24, seed=3)
    w.flux_ref = np.full(2, 1.0)
    w.spec_idx = np.array([640.0, 640.0])     # (200 / 150 MHz)^320 > 1e39, (142 / 150)^320 ~ 1e-8
    w.nu_ref = 150e6
    with np.errstate(all="ignore"):
        V = simulator(w).simulate(w.lsts, w.freqs, "fp16x3").cpu().numpy()[0]
    P = oracle_problem(w)
    amp = (w.freqs / 150e6) ** 320.0
    ok = np.flatnonzero((amp > 1e-12) & (amp < 1e15))
    assert ok.size >= 5 and (amp > 4e38).any()
    for ic in ok:
        assert rel_err(V[ic], oracle.vis(P, w.lsts[0], w.freqs[ic])) <= 2e-5, ic
