"""Calls of one context on different streams, one behind the other without a
synchronisation between (needs a GB300): they share the context's buffers, so each
starts where the one before has ended, and gives what it gives alone."""
import numpy as np
import pytest

from helpers import simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,use_graph", [("fp16x3", True), ("fp16x3", False), ("fp32", True)])
def test_calls_on_two_streams_do_not_mix(prec, use_graph):
    import torch
    w = synth.hera_like(n_ant=200, n_src=40_000, n_chan=8, n_times=6, n_za=46, n_az=120)
    sim = simulator(w, use_graph=use_graph)
    halves = [w.lsts[:3], w.lsts[3:]]
    alone = []
    for t in halves:
        alone.append(sim.simulate(t, w.freqs, prec))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.empty_like(v) for v in alone]
    torch.cuda.synchronize()
    for _ in range(3):
        for t, out, st in zip(halves, outs, streams):
            sim.simulate(t, w.freqs, prec, out=out, stream=st)
    torch.cuda.synchronize()
    sim.check_device_status()
    for out, v in zip(outs, alone):
        assert torch.equal(out, v)


def test_host_output_behind_device_output():
    import torch
    w = synth.batched_uneven(n_pairs=60, n_ant=200, n_src=60_000, n_za=46, n_az=120)
    sim = simulator(w)
    want = sim.simulate_pairs(w.lsts, w.freqs)
    torch.cuda.synchronize()
    on_device = sim.simulate_pairs(w.lsts, w.freqs)              # on torch's stream
    on_host = sim.simulate_pairs(w.lsts, w.freqs, host=True)     # on the context's own
    torch.cuda.synchronize()
    assert torch.equal(on_device, want)
    assert np.array_equal(on_host, want.cpu().numpy())
