"""Which calls run the streamed schedule (needs a GB300): seen in the launches of a call,
one k_front, k_cull_scatter, k_wa, k_zherk_prep, k_zherk and k_zherk_final for one
batch of instances, whatever the array, the feeds and the kind of call.  Without this,
every test of its results would also pass on the older schedules that it falls back to."""
import numpy as np
import pytest

from helpers import dipole_jones_grid, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu
ONE_BATCH = 6


def workload(n_ant, n_src=900, n_chan=4, n_times=2, beam="scalar"):
    w = synth.hera_like(n_ant=n_ant, n_src=n_src, n_chan=n_chan, n_times=n_times, n_za=46, n_az=120)
    if beam == "jones":
        vals = dipole_jones_grid(98e6 + np.arange(105) * 1e6, 31, 72, 0.5, 150e6, np.random.default_rng(3))
        w.beam = ("grid", vals, 98e6, 1e6, (np.pi / 2) / 30, 2 * np.pi / 72, "cubic")
    return w


@pytest.mark.parametrize("n_ant,beam", [(1, "scalar"), (9, "scalar"), (64, "scalar"), (65, "scalar"), (128, "scalar"),
                                        (129, "scalar"), (257, "scalar"), (350, "scalar"), (1000, "scalar"),
                                        (70, "jones"), (350, "jones")])
def test_simulate_streams(n_ant, beam):
    w = workload(n_ant, beam=beam)
    sim = simulator(w)
    sim.simulate(w.lsts, w.freqs)
    assert sim.last_launch_count() == ONE_BATCH
    sim.simulate_pairs(w.lsts, w.freqs[:2])
    assert sim.last_launch_count() == ONE_BATCH


@pytest.mark.parametrize("n_ant", [37, 350])
def test_redundant_groups_stream(n_ant):
    w = workload(n_ant)
    sim = simulator(w)
    sim.set_redundancy()
    sim.simulate_unique(w.lsts, w.freqs)
    assert sim.last_launch_count() == ONE_BATCH


@pytest.mark.parametrize("option", [dict(fuse_zbuild=False), dict(overlap_batches=True), dict(herk_tile_n=128),
                                    dict(herk_split=2), dict(herk_flush_kblocks=8)])
def test_an_option_for_another_schedule_gets_it(option):
    w = workload(100, n_times=3)
    sim = simulator(w, **option)
    sim.simulate(w.lsts, w.freqs)
    assert sim.last_launch_count() != ONE_BATCH
