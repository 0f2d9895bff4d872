"""FP32 overlap update of the split path (register-tiled sums, column-wise factors in the solves) against
float64: log det O and Theta (through the mixed energy of the one-body part and the next step's force bias)
after a step of the oracle's walkers; blocks of 1 to 16 at the edges of 4 and 8, one spin only, orbital
counts that are no multiple of four, unequal blocks.

Bound on log O: sums of M FP32 products and an FP32 LU of a matrix near the identity, some M + 10 ns
roundings of 2^-24 per pivot, ns pivots: 2e-4 at the largest size here; the same relative to the energy."""
import numpy as np
import pytest

from gpu_util import logo_close, need_gpu
from oracle import afqmc as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw", [
    (8, 20, 1, 0, 5), (17, 30, 4, 5, 33), (30, 40, 8, 3, 40), (33, 30, 9, 8, 20), (66, 50, 16, 0, 9),
    (64, 40, 13, 12, 31), (101, 60, 16, 15, 12), (128, 40, 16, 16, 17)])
def test_update(M, X, nu, nd, nw):
    afq = need_gpu()
    rng = np.random.default_rng(M * 3 + nu)
    h1 = rng.standard_normal((M, M)) * (0.3 / np.sqrt(M))
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) * (0.4 / np.sqrt(X * M))
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.1 / np.sqrt(M)
    w = rng.uniform(0.5, 1.5, nw)
    x = rng.standard_normal((2, nw, X))
    g = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, precision=afq.BF16X3, autotune=False)
    g.select_kernel(afq.K_TAYLOR, 4 if N <= 32 else 2)
    g.set_walkers(phi, w)
    o = orc.System(h1, L, trial, nu, nd, 0.01)
    wk = orc.Walkers(o, nw, phi, w)
    for t in range(2):
        g.propagate(1, x[t:t + 1])
        orc.propagate(o, wk, x[t])
    st = g.state()
    assert np.array_equal(st["alive"], wk.alive)
    # log O of the GPU's own walkers, so that only the update's rounding is compared
    ref = orc.Walkers(o, nw, st["phi"], wk.w)
    assert logo_close(st["logO"], ref.logO, 2e-4)
    e = g.energy()[0]
    eo = orc.local_energy(o, st["phi"])
    assert np.abs(e - eo).max() < 5e-4 * np.abs(eo).max()
    assert np.abs(st["w"] - wk.w).max() < 4e-3 * np.abs(wk.w).max()
    g.close()
