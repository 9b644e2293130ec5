"""Device memory of FP32 calls (needs a GB300 and some 40 GB of it): Z planes, beam
tables and partial tiles of a batch keep to the 20 GiB that batches are sized for; a
batch that the caller sized takes no more than two FP32 rows per antenna-feed where
three would pass that."""
import numpy as np
import pytest

from helpers import simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu
GIB = 2 ** 30


@pytest.mark.parametrize("max_batch,limit", [
    (0, 20.0 * GIB),
    # 24 instances of 700 rows x 400,128 columns, and 1 GiB of partial tiles
    (24, 24 * 4 * 700 * 400_128 + 1.0 * GIB),
])
def test_fp32_batches_keep_to_their_memory(max_batch, limit):
    import torch
    w = synth.hera_like(n_ant=350, n_src=400_000, n_chan=24, n_times=1, n_za=46, n_az=120)
    sim = simulator(w, max_batch=max_batch)
    out = torch.empty((1, 24, 350, 350), dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.memory_allocated()
    torch.cuda.reset_peak_memory_stats()
    sim.simulate(w.lsts, w.freqs, "fp32", out=out)
    torch.cuda.synchronize()
    used = torch.cuda.max_memory_allocated() - before
    # live tables (36 bytes a source), beam planes and the call's tables beside it
    assert used <= limit + 0.25 * GIB, used / GIB
    assert used > 0.5 * limit
    assert np.isfinite(torch.view_as_real(out).abs().max().item())
    del sim, out
    torch.cuda.empty_cache()
