"""A multi-determinant setup that fits the device only without the digit forms' scratch: it gives the scratch
back and runs on the other kernels.

Bound 1e-11: one step and a local energy, each form rounding its sums to a few 1e-16 of their largest terms."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_gpu_step_small import system

pytestmark = pytest.mark.gpu


def test_setup_gives_the_scratch_back_when_memory_is_short():
    afq = need_gpu()
    import torch
    M, X, nu, nd, nw, ndet = 64, 320, 8, 8, 256, 12
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, nw, 5)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    dets = np.stack([trial + 0.2 * np.concatenate([q[:, k:k + nu], q[:, k:k + nd]], axis=1) for k in range(ndet)])
    x = rng.standard_normal((1, nw, X))

    def run():
        free = torch.cuda.mem_get_info()[0]
        s = afq.System(h1, L, None, nu, nd, dt=0.005, n_walkers=nw, dets=dets, coeffs=1.0 / np.arange(1, ndet + 1))
        used = free - torch.cuda.mem_get_info()[0]
        s.set_walkers(phi, w)
        s.propagate(1, x)
        e, st = s.energy()[0], s.state()
        s.close()
        return used, e, st["phi"], st["w"]

    run()                                        # (kernels loaded)
    used, e0, phi0, w0 = run()
    torch.cuda.empty_cache()
    short = 48 << 20                             # the scratch takes at least 128 MB
    fill = torch.empty(torch.cuda.mem_get_info()[0] - used + short, dtype=torch.uint8, device="cuda")
    try:
        less, e1, phi1, w1 = run()
    finally:
        del fill
        torch.cuda.empty_cache()
    assert less < used - (100 << 20)
    assert np.abs(e1 - e0).max() < 1e-11 * np.abs(e0).max()
    assert np.abs(phi1 - phi0).max() < 1e-11 and np.abs(w1 - w0).max() < 1e-11
