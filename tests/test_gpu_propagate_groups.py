"""Tensor-core propagator with the occupied columns in two groups that take turns (M <= 128, more than 8
columns) against the oracle on sampled walkers: one and two K blocks, group sizes at the edges of 8 and
16 columns, unequal groups, one walker and more walkers than CTAs, dead walkers in between, and few terms
(one group: a walker's rounds do not cover the next one's loads).

Bounds as for the other tensor-core propagators: split-BF16 products lose at most 2^-15.4 of sum |A| |T|
per term, 5e-4 of the largest element over a step with |A| near one; weights 2e-3."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import afqmc as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw,order", [
    (16, 20, 5, 4, 311, 6), (64, 33, 8, 8, 7, 2), (65, 40, 9, 8, 310, 6), (127, 30, 16, 15, 160, 6),
    (128, 24, 16, 16, 9, 1), (128, 41, 16, 16, 457, 6), (100, 30, 12, 12, 155, 3), (33, 12, 32, 0, 1, 9),
    (96, 20, 8, 1, 153, 6), (128, 20, 4, 4, 170, 6)])
@pytest.mark.parametrize("mode", ["phaseless", "free"])
def test_column_groups(M, X, nu, nd, nw, order, mode):
    afq = need_gpu()
    rng = np.random.default_rng(M * 7 + nu)
    h1 = rng.standard_normal((M, M)) * (0.3 / np.sqrt(M))
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) * (0.6 / np.sqrt(X * M))
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.1 / np.sqrt(M)
    w = rng.uniform(0.5, 1.5, nw)
    w[nw // 3: nw // 3 + nw // 8] = 0.0   # dead
    x = rng.standard_normal((1, nw, X))
    g = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, taylor_order=order, precision=afq.BF16X3,
                   autotune=False, mode=1 if mode == "free" else 0)
    g.select_kernel(afq.K_TAYLOR, 4)
    assert g.info().tuned_taylor_smem == 4
    g.set_walkers(phi, w)
    g.propagate(1, x)
    st = g.state()
    pick = np.unique(np.array([0, nw // 3 + nw // 8, nw // 2, nw - 2, nw - 1]) % nw)
    o = orc.System(h1, L, trial, nu, nd, 0.01, taylor_order=order, mode=mode)
    wk = orc.Walkers(o, len(pick), phi[pick], w[pick])
    orc.propagate(o, wk, x[0][pick])
    assert np.array_equal(st["alive"][pick], wk.alive)
    assert np.abs(st["phi"][pick] - wk.phi).max() < 5e-4 * np.abs(wk.phi).max()
    assert np.abs(st["w"][pick] - wk.w).max() < 2e-3 * np.abs(wk.w).max()
    dead = np.flatnonzero(w == 0.0)
    np.testing.assert_array_equal(st["phi"][dead], phi[dead])   # dead walkers stay as they are
    assert np.all(np.isfinite(st["phi"]))
    g.close()
