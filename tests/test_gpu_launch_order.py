"""Split-precision steps queued back to back (each kernel's launch overlaps the end of the one before it)
against the same steps with a synchronisation after each: the same kernels on the same data, so the same
bits, at sizes where kernels are short and CTAs of neighbouring kernels fit an SM together; on the default
and on another stream."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw,variant", [(8, 24, 2, 2, 37, 3), (33, 60, 5, 4, 300, 4), (64, 100, 8, 8, 900, 3),
                                                  (130, 70, 4, 3, 64, 4), (40, 90, 9, 8, 200, 2)])
@pytest.mark.parametrize("side", [False, True])
def test_queued_steps_equal_synchronised_steps(M, X, nu, nd, nw, variant, side):
    afq = need_gpu()
    import torch
    rng = np.random.default_rng(M)
    h1 = rng.standard_normal((M, M)) * (0.3 / np.sqrt(M))
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) * (0.4 / np.sqrt(X * M))
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    out = []
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.current_stream()):
        for queued in (True, False):
            s = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, seed=5, precision=afq.BF16X3, autotune=False)
            s.select_kernel(afq.K_TAYLOR, variant)
            if queued:
                s.propagate(12)
            else:
                for _ in range(12):
                    s.propagate(1)
                    torch.cuda.synchronize()
            out.append(s.state())
            s.close()
    for k in ("phi", "w", "logO", "alive"):
        np.testing.assert_array_equal(out[0][k], out[1][k])
