"""V written to page-locked host memory (needs a GB300): a call of many instances is cut
into batches whose copies run beside the next batch, and gives what it gives on the
device.  Tolerance: channel groups are cut elsewhere, so that phases of the channel
recurrence differ by its rounding; both are within 1e-5 of the oracle, and of each
other."""
import numpy as np
import pytest

import oracle
from helpers import oracle_problem, rel_err, sample_pairs, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ant,n_times,n_chan", [(200, 3, 64), (350, 2, 70), (256, 5, 40)])
def test_page_locked_output_comes_in_batches(n_ant, n_times, n_chan):
    import torch
    w = synth.hera_like(n_ant=n_ant, n_src=900, n_chan=n_chan, n_times=n_times, n_za=46, n_az=120)
    sim = simulator(w)
    on_device = sim.simulate(w.lsts, w.freqs)
    one = sim.last_launch_count()
    out = torch.full(on_device.shape, float("nan"), dtype=torch.complex64, pin_memory=True)
    sim.simulate(w.lsts, w.freqs, out=out, host=True)
    # every batch but the first has a launch for its phase table, and four of its own
    batches = -(-n_times * n_chan // 64)
    assert sim.last_launch_count() >= one + 5 * (batches - 1)
    V, D = out.numpy(), on_device.cpu().numpy()
    P = oracle_problem(w)
    pa, pb = sample_pairs(n_ant, 100, seed=1)
    for it in range(n_times):
        for ic in range(n_chan):
            assert rel_err(V[it, ic], D[it, ic]) <= 1e-5, (it, ic)
    for it, ic in ((0, 0), (n_times - 1, n_chan - 1)):
        assert rel_err(V[it, ic][pa, pb], oracle.vis(P, w.lsts[it], w.freqs[ic], pairs=(pa, pb))[:, 0, 0]) <= 1e-5


def test_long_pairs_stay_in_one_batch():
    # pairs are put in waves by their live counts; where the products far outlast the
    # copy, cutting them into batches would only disturb that
    import torch
    w = synth.batched_uneven(n_pairs=80, n_ant=200, n_src=60_000, n_za=46, n_az=120)
    sim = simulator(w)
    on_device = sim.simulate_pairs(w.lsts, w.freqs)
    one = sim.last_launch_count()
    out = torch.empty(on_device.shape, dtype=torch.complex64, pin_memory=True)
    sim.simulate_pairs(w.lsts, w.freqs, out=out, host=True)
    assert sim.last_launch_count() == one
    assert np.array_equal(out.numpy(), on_device.cpu().numpy())
    # short ones are cut as a grid is
    w = synth.batched_uneven(n_pairs=80, n_ant=350, n_src=500, n_za=46, n_az=120)
    sim = simulator(w)
    sim.simulate_pairs(w.lsts, w.freqs, out=torch.empty((80, 350, 350), dtype=torch.complex64, pin_memory=True), host=True)
    assert sim.last_launch_count() >= one + 5
