"""Setting a sky whose tables go up in pieces of 2^20 sources (needs a GB300): V
is additive over the sources, and a refused sky leaves the old one in place."""
import numpy as np
import pytest

from helpers import simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu
PIECE = 1 << 20
TOL = 1e-5   # max|V - exact| / max|exact| of every mode


@pytest.mark.parametrize("n_src", [PIECE, PIECE + 3])
def test_skies_in_pieces(n_src):
    w = synth.hera_like(n_ant=4, n_src=n_src, n_chan=1, n_times=1, n_za=46, n_az=120)
    sim = simulator(w)

    def vis(a, b):
        sim.init_sky(w.ra[a:b], w.dec[a:b], w.flux_ref[a:b], w.spec_idx[a:b], w.nu_ref)
        return sim.simulate(w.lsts, w.freqs).cpu().numpy()

    parts = [vis(0, 5000), vis(5000, n_src)]
    whole = vis(0, n_src)
    bound = TOL * sum(np.abs(v).max() for v in [whole] + parts)
    assert np.abs(whole - parts[0] - parts[1]).max() <= bound
    flux = w.flux_ref.copy()
    flux[[n_src - 1, n_src - 2]] = np.nan
    with pytest.raises(Exception, match=rf"flux_ref\[{n_src - 2}\]"):
        sim.init_sky(w.ra, w.dec, flux, w.spec_idx, w.nu_ref)
    assert np.array_equal(sim.simulate(w.lsts, w.freqs).cpu().numpy(), whole)
