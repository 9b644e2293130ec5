"""FP32 visibilities on the CUDA cores at the sizes where the product tiles can
go wrong (needs a GB300): antenna-feed counts about the 16-, 32- and 128-row
steps in the two-product-per-entry form and in the three-product one, one
antenna, stages of 32 sources that are partly filled, source ranges split over
blocks, and feeds x axes.

Tolerance: max|V - V_oracle| / max|V_oracle| <= 1e-5, as for every mode.
"""
import numpy as np
import pytest

from helpers import oracle_problem, simulator
from paper_2312_09763_gb300 import synth
from test_gpu_stream import check, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ant,n_src,n_chan,n_times", [
    (1, 65, 1, 1),
    (8, 31, 2, 2),
    (17, 1000, 3, 1),
    (49, 20000, 1, 1),      # few products: the sources split over many blocks
    (64, 130, 9, 2),
    (65, 3000, 5, 1),
    (128, 2000, 2, 3),
    (129, 5000, 5, 2),
    (160, 1500, 3, 1),
    (257, 700, 3, 1),
    (350, 12001, 2, 2),
])
def test_sizes(n_ant, n_src, n_chan, n_times):
    w = workload(n_ant, n_src, n_chan, n_times, seed=n_ant)
    sim = simulator(w)
    V = sim.simulate(w.lsts, w.freqs, "fp32").cpu().numpy()
    check(w, V, oracle_problem(w), {(0, 0), (n_times - 1, n_chan - 1)})
    assert np.array_equal(V, sim.simulate(w.lsts, w.freqs, "fp32").cpu().numpy())


@pytest.mark.parametrize("n_ant", [40, 75])
def test_feeds_and_axes(n_ant):
    w = synth.polarised_diffuse(n_ant=n_ant, nside=16, n_chan=3, n_times=1, n_za=31, n_az=72, lmax=40, full_stokes=True)
    V = simulator(w).simulate(w.lsts, w.freqs, "fp32").cpu().numpy()
    check(w, V, oracle_problem(w), {(0, 0), (0, 2)})
