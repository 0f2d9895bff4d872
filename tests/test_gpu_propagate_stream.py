"""Tensor-core propagator for more than 128 orbitals (A streamed) against the oracle on sampled walkers:
two CTAs per SM (few columns) and one CTA with two copies of the term operand; orbital counts at both
edges of a 64-wide K block and of the second row tile, up to N M = 4096, one Taylor term and six, fewer
walkers than CTAs and more.

Bounds as for the M <= 64 tensor-core propagator: split-BF16 products lose at most 2^-15.4 of
sum |A| |T| per term, 5e-4 of the largest element over a step with |A| near one; weights 2e-3."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import afqmc as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw,order", [
    (129, 40, 4, 3, 313, 6), (192, 33, 8, 8, 7, 1), (145, 64, 12, 8, 160, 6), (190, 41, 12, 9, 11, 3), (131, 35, 16, 15, 20, 6),
    (193, 50, 1, 0, 5, 6), (200, 24, 9, 9, 157, 6), (255, 30, 8, 8, 3, 6), (256, 36, 9, 7, 155, 2),
    (240, 20, 9, 8, 9, 6)])
@pytest.mark.parametrize("mode", ["phaseless", "free"])
def test_streamed_propagator(M, X, nu, nd, nw, order, mode):
    afq = need_gpu()
    rng = np.random.default_rng(M * 7 + nu)
    h1 = rng.standard_normal((M, M)) * (0.3 / np.sqrt(M))
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) * (0.6 / np.sqrt(X * M))   # |sum_g x_g L_g| of about 1.7
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.1 / np.sqrt(M)
    w = rng.uniform(0.5, 1.5, nw)
    x = rng.standard_normal((1, nw, X))
    g = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, taylor_order=order, precision=afq.BF16X3,
                   autotune=False, mode=1 if mode == "free" else 0)
    g.select_kernel(afq.K_TAYLOR, 4)
    assert g.info().tuned_taylor_smem == 4
    g.set_walkers(phi, w)
    g.propagate(1, x)
    st = g.state()
    pick = np.unique(np.array([0, nw // 2, nw - 1]))
    o = orc.System(h1, L, trial, nu, nd, 0.01, taylor_order=order, mode=mode)
    wk = orc.Walkers(o, len(pick), phi[pick], w[pick])
    orc.propagate(o, wk, x[0][pick])
    assert np.array_equal(st["alive"][pick], wk.alive)
    assert np.abs(st["phi"][pick] - wk.phi).max() < 5e-4 * np.abs(wk.phi).max()
    assert np.abs(st["w"][pick] - wk.w).max() < 2e-3 * np.abs(wk.w).max()
    assert np.all(np.isfinite(st["phi"]))
    g.close()
