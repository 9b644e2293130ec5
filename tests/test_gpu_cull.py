"""The horizon cut where it is close (needs a GB300): sources from a hundredth to
1e-15 radians above and below the horizon, where FP32 products cannot decide.
The live counts are those of the oracle, exactly."""
import numpy as np
import pytest

import oracle
from helpers import oracle_problem, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_src", [700, 600_000])   # (above 524,288 the block counts are scanned by a kernel)
def test_sources_about_the_horizon(n_src):
    w = synth.hera_like(n_ant=3, n_src=n_src, n_chan=1, n_times=3, n_za=46, n_az=120)
    g = np.random.default_rng(5)
    lst = w.lsts[1]
    alt = g.choice([-1.0, 1.0], n_src) * 10.0 ** g.uniform(-15, -2, n_src)
    az = g.uniform(0, 2 * np.pi, n_src)
    sl, cl = np.sin(w.lat), np.cos(w.lat)
    e, n, u = np.cos(alt) * np.sin(az), np.cos(alt) * np.cos(az), np.sin(alt)
    w.dec = np.arcsin(np.clip(sl * u + cl * n, -1, 1))
    w.ra = np.mod(lst - np.arctan2(-e, cl * u - sl * n), 2 * np.pi)
    sim = simulator(w)
    sim.simulate(w.lsts, w.freqs)
    P = oracle_problem(w)
    live = sim.last_live_counts(3)
    assert [int(x) for x in live] == [oracle.count_live(P, t) for t in w.lsts]
    assert 0.4 * n_src < live[1] < 0.6 * n_src
