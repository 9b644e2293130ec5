"""Calls on a stream of a green context, which owns a part of the GPU's SMs (needs a
GB300).  The streamed schedule needs one block resident on every SM of the device; such
calls keep the schedules that do not, and give the same visibilities.  Tolerance:
max|V - V_oracle| / max|V_oracle| <= 1e-5, as for every mode."""
import ctypes

import numpy as np
import pytest

import oracle
from helpers import oracle_problem, rel_err, simulator
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture
def green_stream():
    import torch
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    whole, part = (ctypes.c_byte * 144)(), (ctypes.c_byte * 144)()   # CUdevResource
    groups, desc, ctx, st = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    dev = ctypes.c_int()
    ok = cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
    ok = ok and cu.cuDeviceGetDevResource(dev, whole, 1) == 0   # 1: SMs
    ok = ok and cu.cuDevSmResourceSplitByCount(part, ctypes.byref(groups), whole, None, 0, 64) == 0 and groups.value == 1
    ok = ok and cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1) == 0
    ok = ok and cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, dev, 1) == 0
    ok = ok and cu.cuGreenCtxStreamCreate(ctypes.byref(st), ctx, 1, 0) == 0   # 1: non-blocking
    if not ok:
        pytest.skip("no green contexts here")
    yield torch.cuda.ExternalStream(st.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(st)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("prec", ["fp16x3", "fp32"])
def test_simulate_on_part_of_the_sms(green_stream, use_graph, prec):
    import torch
    w = synth.hera_like(n_ant=150, n_src=4000, n_chan=6, n_times=2, n_za=46, n_az=120)
    sim = simulator(w, use_graph=use_graph)
    whole = sim.simulate(w.lsts, w.freqs, prec)
    n_whole = sim.last_launch_count()
    torch.cuda.synchronize()
    out = torch.zeros_like(whole)
    torch.cuda.synchronize()
    for _ in range(2):
        sim.simulate(w.lsts, w.freqs, prec, out=out, stream=green_stream)
    green_stream.synchronize()
    sim.check_device_status(stream=green_stream)
    if prec == "fp16x3":
        assert sim.last_launch_count() != n_whole   # (another schedule)
    P = oracle_problem(w)
    V = out.cpu().numpy()
    for it, ic in ((0, 0), (1, 5)):
        assert rel_err(V[it, ic], oracle.vis(P, w.lsts[it], w.freqs[ic])) <= 1e-5, (it, ic)
    # a new sky waits for the calls on any stream, and the whole device still serves
    sim.init_sky(w.ra, w.dec, w.flux_ref, w.spec_idx, w.nu_ref)
    again = sim.simulate(w.lsts, w.freqs, prec)
    assert sim.last_launch_count() == n_whole
    assert torch.equal(again, whole)
