"""Tangent mode with the Taylor series and the local energy in digit form (handles with many walkers)
against the same walkers on a handle of three (FP64-pipe kernels): stacked and joined rows, odd M, one
spin only, several orders.

Bound: derivatives of a run of well-conditioned walkers, each form rounding its products to a few
1e-16; 1e-10 of the largest derivative leaves five orders for the steps' accumulation."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw,steps,order", [
    (40, 200, 6, 5, 300, 3, 6), (33, 90, 5, 4, 1201, 2, 1), (64, 160, 6, 0, 700, 2, 3), (65, 130, 5, 4, 400, 3, 6),
    (98, 200, 9, 8, 160, 2, 5), (130, 150, 4, 4, 300, 2, 6)])
def test_tangent_matches_walker_kernels(M, X, nu, nd, nw, steps, order):
    afq = need_gpu()
    rng = np.random.default_rng(M * 19 + nw)
    h1 = np.diag(np.linspace(-2, 3, M)) + 0.02 * rng.standard_normal((M, M))
    h1 = 0.5 * (h1 + h1.T)
    L = rng.standard_normal((X, M, M)) / np.sqrt(X * M)
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.2 / np.sqrt(M)
    x = rng.standard_normal((steps, nw, X))
    P = rng.standard_normal((M, M))
    P = P + P.T

    def run(n, sel):
        s = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=n, taylor_order=order)
        s.set_walkers(phi[sel])
        s.set_tangent(P)
        s.propagate(steps, np.ascontiguousarray(x[:, sel]))
        em, dm, de = s.energy_tangent()
        el = s.energy()[0]
        return s.tangent_state(), de, el, s.state()

    dw, de, el, st = run(nw, np.arange(nw))
    pick = np.array([0, nw // 2, nw - 1])
    dw3, de3, el3, st3 = run(3, pick)
    live = st3["alive"]
    assert np.array_equal(st["alive"][pick], live)
    assert np.abs(dw[pick] - dw3)[live].max() < 1e-10 * np.abs(dw3).max()
    assert np.abs(de[pick] - de3)[live].max() < 1e-10 * np.abs(de3).max()
    assert np.abs(el[pick] - el3)[live].max() < 1e-11 * np.abs(el3).max()
    assert np.abs(st["phi"][pick] - st3["phi"]).max() < 1e-11
