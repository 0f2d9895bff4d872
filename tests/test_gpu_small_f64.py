"""FP64 kernels for small problems against the oracle: the 16 x 16-tile contraction, the Taylor kernel
for M <= 32 and the LU overlap kernel for spin blocks of at most 16, over one- and two-electron
blocks, one spin only, blocks around 8, 9 and 16, and the block-wide kernel above 16.

Bound 1e-10: one step of well-conditioned walkers (overlap matrices near the identity), each side
rounding sums of at most X terms of order one to a few 1e-16."""
import numpy as np
import pytest

from gpu_util import logo_close, need_gpu
from oracle import afqmc as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw,order", [
    (3, 5, 1, 0, 7, 6), (5, 9, 2, 1, 40, 6), (8, 24, 2, 2, 128, 6), (16, 33, 8, 8, 33, 6), (17, 40, 9, 1, 20, 4),
    (23, 50, 11, 10, 11, 6), (32, 70, 16, 16, 9, 6), (32, 64, 32, 32, 3, 2), (31, 20, 12, 0, 5, 7),
    (33, 40, 17, 3, 6, 6), (41, 35, 16, 15, 4, 6)])
@pytest.mark.parametrize("mode", ["phaseless", "free"])
def test_one_step_and_energy(M, X, nu, nd, nw, order, mode):
    afq = need_gpu()
    rng = np.random.default_rng(M * 11 + nu)
    h1 = rng.standard_normal((M, M)) * 0.3
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) / np.sqrt(X * M)
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.2 / np.sqrt(M)
    w = rng.uniform(0.5, 1.5, nw)
    x = rng.standard_normal((1, nw, X))
    g = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, taylor_order=order, mode=1 if mode == "free" else 0)
    o = orc.System(h1, L, trial, nu, nd, 0.01, taylor_order=order, mode=mode)
    g.set_walkers(phi, w)
    wk = orc.Walkers(o, nw, phi, w)
    assert logo_close(g.state()["logO"], wk.logO, 1e-10)
    g.propagate(1, x)
    orc.propagate(o, wk, x[0])
    st = g.state()
    assert np.array_equal(st["alive"], wk.alive)
    assert np.abs(st["phi"] - wk.phi).max() < 1e-10 * np.abs(wk.phi).max()
    assert np.abs(st["w"] - wk.w).max() < 1e-10 * np.abs(wk.w).max()
    live = wk.alive
    assert logo_close(st["logO"][live], wk.logO[live], 1e-10)
    el = g.energy()[0]
    eo = orc.local_energy(o, wk.phi)
    assert np.abs(el - eo)[live].max() < 1e-10 * np.abs(eo).max()
