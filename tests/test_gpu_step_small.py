"""FP64 steps of small systems in one kernel: several steps per call against the oracle and against one
step per call (the same arithmetic, so the same bits), with one electron, one spin, the largest blocks,
more steps than one launch takes, walkers dead at the start, walkers that the phase cut kills on the way
(a long time step) and one whose fields overflow.

Bound 1e-9: up to 20 steps, each within the 1e-10 of the one-step test of the separate kernels, of walkers
whose overlaps stay near the identity."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import afqmc as orc

pytestmark = pytest.mark.gpu


def system(M, X, nu, nd, nw, seed):
    rng = np.random.default_rng(seed)
    h1 = rng.standard_normal((M, M)) * 0.3
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) / np.sqrt(X * M)
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    phi = trial + (rng.standard_normal((nw, M, nu + nd)) + 1j * rng.standard_normal((nw, M, nu + nd))) * 0.2 / np.sqrt(M)
    return h1, L, trial, phi, rng.uniform(0.5, 1.5, nw), rng


@pytest.mark.parametrize("M,X,nu,nd,nw,steps,dt,order", [
    (1, 1, 1, 0, 5, 3, 0.01, 6), (3, 5, 1, 0, 7, 9, 0.01, 6), (8, 24, 2, 2, 128, 20, 0.01, 6),
    (8, 24, 2, 1, 300, 8, 0.3, 6), (16, 7, 8, 8, 9, 5, 0.01, 1), (16, 33, 7, 0, 33, 4, 0.02, 12),
    (13, 40, 3, 5, 17, 11, 0.05, 6)])
@pytest.mark.parametrize("mode", ["phaseless", "free"])
def test_steps(M, X, nu, nd, nw, steps, dt, order, mode):
    afq = need_gpu()
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, nw, M * 13 + nu)
    x = rng.standard_normal((steps, nw, X))
    w[1] = 0.0   # dead at the start
    kw = dict(dt=dt, n_walkers=nw, taylor_order=order, mode=1 if mode == "free" else 0)
    g, g1 = (afq.System(h1, L, trial, nu, nd, **kw) for _ in range(2))
    g.set_walkers(phi, w)
    g1.set_walkers(phi, w)
    g.propagate(steps, x)
    for t in range(steps):
        g1.propagate(1, x[t:t + 1])
    a, b = g.state(), g1.state()
    for k in ("phi", "w", "logO", "alive"):
        np.testing.assert_array_equal(a[k], b[k])
    assert g.info().step == steps
    o = orc.System(h1, L, trial, nu, nd, dt, taylor_order=order, mode=mode)
    wk = orc.Walkers(o, nw, phi, w)
    for t in range(steps):
        orc.propagate(o, wk, x[t])
    live = wk.alive.copy()
    live[1] = False
    assert np.array_equal(a["alive"], wk.alive)
    if dt == 0.3 and mode == "phaseless":
        assert 0 < live.sum() < nw - 1
    assert np.abs(a["phi"] - wk.phi)[live].max() < 1e-9 * np.abs(wk.phi[live]).max()
    assert np.abs(a["w"] - wk.w)[live].max() < 1e-9 * np.abs(wk.w[live]).max()


def test_overflow_kills_one_walker_and_generated_fields_advance():
    afq = need_gpu()
    M, X, nu, nd, nw = 8, 24, 2, 2, 6
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, nw, 3)
    x = rng.standard_normal((5, nw, X))
    x[2, 4] = 1e170
    g = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw)
    g.set_walkers(phi, w)
    g.propagate(5, x)
    st = g.state()
    assert list(st["alive"]) == [True] * 4 + [False, True] and st["w"][4] == 0.0
    # generated fields: five and then three steps are eight steps
    g.set_walkers(phi, w)
    g.propagate(5)
    g.propagate(3)
    a = g.state()
    g.set_walkers(phi, w)
    g.propagate(8)
    b = g.state()
    for k in ("phi", "w", "logO", "alive"):
        np.testing.assert_array_equal(a[k], b[k])
