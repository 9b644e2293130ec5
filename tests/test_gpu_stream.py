"""The streamed schedule (Z built into a ring that stays in L2 and expanded as
it is written, the default FP16x3 path) at the sizes where it can go wrong
(needs a GB300): antenna counts about the 128-row panels (in the real form and
in the three-product one), one antenna, chunks of 64 sources that are partly
filled, channel groups of one, of a few and past a multiple of the recurrence
block, unevenly spaced channels, several launches of a call, source ranges
split over SMs, every feed / axis combination, several beams, and pairs of
very different live counts.

Tolerance: max|V - V_oracle| / max|V_oracle| <= 1e-5, as for every mode.
"""
import numpy as np
import pytest

import oracle
from helpers import dipole_jones_grid, oracle_problem, rel_err, sample_pairs, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5


def workload(n_ant, n_src, n_chan, n_times, layout="random", channels="even", seed=0):
    w = synth.hera_like(n_ant=n_ant, n_src=n_src, n_chan=n_chan, n_times=n_times, n_za=46, n_az=120)
    g = np.random.default_rng(100 + seed)
    if layout == "random":
        w.enu = synth.square_array(n_ant, 40.0 + 8.0 * np.sqrt(n_ant), g)
        w.enu[:, 2] = g.uniform(-2, 2, n_ant)
    if channels == "odd":
        w.freqs = np.sort(g.uniform(101e6, 199e6, n_chan))
    return w


def check(w, V, P, picks, n_pairs=400):
    nf = V.shape[-1] // w.n_ant
    pa, pb = sample_pairs(w.n_ant, n_pairs, seed=2) if w.n_ant > 1 else (np.zeros(1, np.int32), np.zeros(1, np.int32))
    for it, ic in picks:
        Vi = V[it, ic].reshape(w.n_ant, nf, w.n_ant, nf)
        vo = oracle.vis(P, w.lsts[it], w.freqs[ic], pairs=(pa, pb))
        assert rel_err(Vi[pa, :, pb, :], vo) <= TOL, (it, ic)
        # the mirror image is exact and autocorrelations are real
        assert np.array_equal(Vi[pb, :, pa, :], np.conj(np.swapaxes(Vi[pa, :, pb, :], 1, 2)))
        assert np.all(np.diagonal(V[it, ic]).imag == 0)


@pytest.mark.parametrize("n_ant,n_src,n_chan,n_times,channels", [
    (1, 65, 1, 1, "even"),
    (2, 1000, 3, 2, "even"),
    (63, 4097, 8, 1, "even"),       # one recurrence block
    (64, 130, 9, 2, "even"),        # a block and one; two 64-source chunks
    (65, 3000, 21, 1, "even"),      # a group longer than a buffer holds
    (128, 2000, 2, 3, "odd"),       # one 128-row panel of the three-product form
    (129, 5000, 5, 2, "odd"),
    (256, 1500, 17, 1, "even"),
    (257, 700, 3, 1, "even"),
    (350, 3001, 20, 2, "even"),     # the flagship array: waves of 19 instances
])
def test_sizes(n_ant, n_src, n_chan, n_times, channels):
    w = workload(n_ant, n_src, n_chan, n_times, channels=channels, seed=n_ant)
    V = simulator(w).simulate(w.lsts, w.freqs, "fp16x3").cpu().numpy()
    check(w, V, oracle_problem(w), {(0, 0), (n_times - 1, n_chan - 1), (n_times // 2, n_chan // 2)})


@pytest.mark.parametrize("n_feed,n_ax,n_beam", [(1, 1, 2), (1, 2, 1), (2, 1, 1), (2, 2, 1), (2, 2, 3), (1, 2, 2)])
def test_feeds_axes_and_beams(n_feed, n_ax, n_beam):
    n_ant = 90
    w = workload(n_ant, 3500, 5, 2, seed=n_feed * 10 + n_ax)
    g = np.random.default_rng(7)
    J = dipole_jones_grid(98e6 + np.arange(105) * 1e6, 31, 72, 0.5, 150e6, g)[:, :n_feed, :n_ax]
    if n_ax == 1:   # a single axis is a scalar field: smooth and single-valued at the zenith
        J = np.repeat(np.abs(J[:, :1, :1]) * 0 + np.exp(-2.0 * np.linspace(0, np.pi / 2, 31) ** 2)[:, None], n_feed, axis=1)
    vals = np.concatenate([(J * (1.0 - 0.2j * b)).astype(np.complex64) for b in range(n_beam)])
    w.beam = ("grid", vals, 98e6, 1e6, (np.pi / 2) / 30, 2 * np.pi / 72, "cubic")
    w.beam_idx = (np.arange(n_ant) % n_beam).astype(np.int32) if n_beam > 1 else None
    V = simulator(w).simulate(w.lsts, w.freqs, "fp16x3").cpu().numpy()
    check(w, V, oracle_problem(w), {(0, 0), (1, 4)})


@pytest.mark.parametrize("n_ant,max_batch", [(70, 3), (140, 7)])
def test_several_launches_and_repeats_are_bit_equal(n_ant, max_batch):
    # a call of several launches, each with its own waves; the same call again,
    # captured and replayed, gives the same bits
    w = workload(n_ant, 6000, 6, 3)
    sim = simulator(w, max_batch=max_batch)
    a = sim.simulate(w.lsts, w.freqs, "fp16x3").cpu().numpy()
    b = sim.simulate(w.lsts, w.freqs, "fp16x3").cpu().numpy()
    c = simulator(w, max_batch=max_batch, use_graph=False).simulate(w.lsts, w.freqs, "fp16x3", host=True)
    assert np.array_equal(a, b) and np.array_equal(a, c)
    check(w, a, oracle_problem(w), {(0, 0), (2, 5), (1, 3)})


def test_pairs_of_very_different_live_counts():
    # a catalogue clustered on a tenth of the sky: instances with a handful and
    # with almost all of the sources above the horizon share a wave
    w = synth.batched_uneven(n_pairs=23, n_ant=150, n_src=9000, n_za=46, n_az=120)
    ra, dec = synth.vmf_cluster(9000, 40.0, 1.0, w.lat, np.random.default_rng(4))
    w.ra, w.dec = ra, dec
    sim = simulator(w)
    V = sim.simulate_pairs(w.lsts, w.freqs, "fp16x3").cpu().numpy()
    live = sim.last_live_counts(23)
    assert live.min() < 0.1 * live.max()
    P = oracle_problem(w)
    pa, pb = sample_pairs(w.n_ant, 300, seed=9)
    for i in (int(np.argmin(live)), int(np.argmax(live)), 11):
        assert live[i] == oracle.count_live(P, w.lsts[i])
        if live[i] == 0:
            assert not V[i].any()
            continue
        vo = oracle.vis(P, w.lsts[i], w.freqs[i], pairs=(pa, pb))[:, 0, 0]
        # (the last sources at the horizon are seen through a beam of 1e-22: V below
        # the smallest normal FP32 number has no relative precision to hold)
        err = np.abs(V[i][pa, pb].astype(np.complex128) - vo).max()
        assert err <= TOL * np.abs(vo).max() + np.finfo(np.float32).tiny, (i, live[i])
