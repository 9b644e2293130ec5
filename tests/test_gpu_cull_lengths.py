"""The horizon cut of vectors of any length (needs a GB300): above or below the horizon
is the sign of the FP64 Up component, also where FP32 products of the vector would
lose their places (lengths about 1e-40) or overflow."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2312_09763_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1e-300, 1e-43, 1e-41, 1e-39, 1e-30, 1.0, 1e38, 1e200])
def test_static_cull_is_the_sign_of_up_at_any_length(length):
    import torch
    from paper_2312_09763_gb300 import binding
    lib = binding.load_library()
    w = synth.hera_like(n_ant=3, n_src=20_000, n_chan=1, n_times=1, n_za=31, n_az=60)
    lst, n = 1.9, w.n_src
    # half of the sources within 1e-7 .. 1e-2 of the horizon
    g = np.random.default_rng(8)
    alt = np.where(np.arange(n) % 2, g.choice([-1.0, 1.0], n) * 10.0 ** g.uniform(-7, -2, n), np.arcsin(g.uniform(-1, 1, n)))
    az = g.uniform(0, 2 * np.pi, n)
    enu = np.stack([np.cos(alt) * np.sin(az), np.cos(alt) * np.cos(az), np.sin(alt)], 1)
    R = oracle.rotation(lst, w.lat)
    x = length * (enu @ R)
    up = oracle.to_topo(R, x)[:, 2]
    assert 0.4 * n < np.sum(up > 0) < 0.6 * n
    xeq = torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    idx = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    out = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    azza = torch.zeros((n, 2), dtype=torch.float32, device="cuda")
    nl = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = lib.mv_horizon_cull_static(n, ctypes.c_void_p(xeq.data_ptr()), lst, float(w.lat), ctypes.c_void_p(idx.data_ptr()),
                                    ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(azza.data_ptr()),
                                    ctypes.c_void_p(nl.data_ptr()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream or 1))
    assert rc == 0, lib.mv_last_error().decode()
    torch.cuda.synchronize()
    live = np.flatnonzero(up > 0)
    assert int(nl.item()) == live.size
    assert np.array_equal(idx[:live.size].cpu().numpy(), live)
