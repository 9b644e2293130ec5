"""Set-up calls right behind a simulation that is still running on a stream of the
caller's (needs a GB300): antennas, beams, polarisation, redundancy and network
parameters replace what the running kernels read only once those are through."""
import numpy as np
import pytest

from helpers import dipole_jones_grid, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


def workload(beam="scalar", n_src=60_000):
    w = synth.hera_like(n_ant=200, n_src=n_src, n_chan=16, n_times=3, n_za=46, n_az=120)
    if beam == "jones":
        g = np.random.default_rng(1)
        vals = dipole_jones_grid(98e6 + np.arange(105) * 1e6, 31, 72, 0.5, 150e6, g)
        w.beam = ("grid", vals, 98e6, 1e6, (np.pi / 2) / 30, 2 * np.pi / 72, "cubic")
        w.stokes_quv = np.stack([0.3 * w.flux_ref, -0.2 * w.flux_ref, 0.1 * w.flux_ref])
    return w


def other_beam(w):
    b = w.beam
    return (b[0], (b[1] * np.complex64(0.3 - 0.8j)).astype(np.complex64)) + tuple(b[2:])


CHANGES = {
    "antennas": lambda sim, w: sim.set_antennas(w.enu * 1.7, w.beam_idx, w.lat),
    "beam": lambda sim, w: sim.set_beam(other_beam(w)),
    "polarisation": lambda sim, w: sim.set_sky_polarisation(-w.stokes_quv),
    "sky": lambda sim, w: sim.init_sky(w.ra, -w.dec, w.flux_ref[::-1].copy(), w.spec_idx, w.nu_ref),
}


@pytest.mark.parametrize("change", list(CHANGES))
def test_a_running_call_keeps_what_it_was_given(change):
    import torch
    w = workload("jones" if change == "polarisation" else "scalar")
    sim = simulator(w)
    want = sim.simulate(w.lsts, w.freqs)
    torch.cuda.synchronize()
    out = torch.empty_like(want)
    st = torch.cuda.Stream()
    sim.simulate(w.lsts, w.freqs, out=out, stream=st)   # (a few milliseconds; nothing waits for it here)
    CHANGES[change](sim, w)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    after = sim.simulate(w.lsts, w.freqs)
    assert not torch.equal(after, want)


def test_redundancy_behind_a_running_call():
    import torch
    w = workload()
    sim = simulator(w)
    sim.set_redundancy()
    want = sim.simulate_unique(w.lsts, w.freqs)
    torch.cuda.synchronize()
    out = torch.empty_like(want)
    sim.simulate_unique(w.lsts, w.freqs, out=out, stream=torch.cuda.Stream())
    # the same groups in other places: the array turned round
    sim.set_antennas(w.enu[::-1].copy(), w.beam_idx, w.lat)
    sim.set_redundancy()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def test_network_parameters_behind_a_running_call():
    import torch
    w = workload()
    w.freqs = w.freqs[:4]
    sim = simulator(w)
    sim.surrogate_create()
    sim.set_beam_surrogate(True)
    want = sim.simulate(w.lsts, w.freqs)
    torch.cuda.synchronize()
    out = torch.empty_like(want)
    sim.simulate(w.lsts, w.freqs, out=out, stream=torch.cuda.Stream())
    p = sim.surrogate_params()[0]
    sim.surrogate_set_params((1.5 * p).astype(np.float32))
    torch.cuda.synchronize()
    assert torch.equal(out, want)
