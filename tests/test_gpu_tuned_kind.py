"""What the autotuner found for one kind of call says nothing of another (needs a GB300).
The whole V of 1800 antennas has more products than the streamed schedule takes, so a
tuning of simulate() keeps another one; the redundant groups of the same array, the same
matrix and batch size, still run streamed."""
import numpy as np
import pytest

from helpers import simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


def test_tuning_of_the_whole_v_leaves_redundant_groups_alone():
    import torch
    w = synth.hera_like(n_ant=1800, n_src=600, n_chan=2, n_times=1, n_za=46, n_az=120)
    sim = simulator(w)
    assert 0 < sim.set_redundancy() < 1800 * 1801 // 4
    before = sim.simulate_unique(w.lsts, w.freqs)
    launches = sim.last_launch_count()
    sim.autotune(w.lsts, w.freqs)
    after = sim.simulate_unique(w.lsts, w.freqs)
    assert sim.last_launch_count() == launches
    assert torch.equal(before, after)
    # (and another schedule would show in the count)
    other = simulator(w, fuse_zbuild=False)
    other.set_redundancy()
    other.simulate_unique(w.lsts, w.freqs)
    assert other.last_launch_count() != launches
    assert np.isfinite(torch.view_as_real(after).abs().max().item())
