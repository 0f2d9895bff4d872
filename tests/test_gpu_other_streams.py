"""FP64 handles with digit contractions: their synchronising calls wait for their own stream only."""
import time

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["get_state", "info", "energy"])
def test_call_waits_for_its_own_stream_only(call):
    afq = need_gpu()
    import torch
    M, X, nu, nd, nw = 40, 200, 6, 5, 300   # contractions in digit form
    rng = np.random.default_rng(0)
    L = rng.standard_normal((X, M, M)) / np.sqrt(X * M)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    side, busy = torch.cuda.Stream(), torch.cuda.Event()
    phi = torch.empty(2, nw, M, nu + nd, device="cuda", dtype=torch.float64)
    with torch.cuda.stream(side):
        s = afq.System(np.diag(np.linspace(-2, 3, M)), L + np.swapaxes(L, 1, 2), trial, nu, nd, dt=0.005, n_walkers=nw)
        s.propagate(1)
        run = {"get_state": lambda: afq.afqmc_get_state(s.h, phi), "info": s.info, "energy": s.energy}[call]
        run()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    torch.cuda._sleep(400_000_000)   # the default stream (which copies on the legacy stream wait for): about 0.2 s
    busy.record(torch.cuda.default_stream())
    with torch.cuda.stream(side):
        run()
    waited = busy.query()
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 > 0.05 and not waited
