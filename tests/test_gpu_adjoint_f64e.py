"""Reverse mode with its Taylor reverse and measurement reverse in digit form (csrc/taylor_f64e.cu,
csrc/energy_f64e.cu, taken by handles with many walkers): the gradient contracted with random
symmetric P against the tangent mode's derivative (other kernels for both pieces), for stacked and
joined rows, odd M, one spin, and a walker that is dead from the start.

Bound: 1e-8 relative, as between the two modes elsewhere."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

# (M, X, n_up, n_dn, walkers, steps, order)
SHAPES = [(33, 90, 5, 4, 1201, 4, 6), (64, 160, 6, 0, 700, 2, 3), (65, 130, 5, 4, 400, 3, 6), (98, 200, 9, 8, 160, 4, 5),
          (40, 120, 6, 5, 900, 5, 1)]


@pytest.mark.parametrize("M,X,nu,nd,nw,steps,order", SHAPES)
def test_gradient_contracts_to_the_tangent(M, X, nu, nd, nw, steps, order):
    afq = need_gpu()
    rng = np.random.default_rng(M * 13 + nw)
    h1 = np.diag(np.linspace(-2, 3, M)) + 0.02 * rng.standard_normal((M, M))
    h1 = 0.5 * (h1 + h1.T)
    L = rng.standard_normal((X, M, M)) / np.sqrt(X * M)
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.2 / np.sqrt(M)
    w = rng.uniform(0.5, 1.5, nw)
    w[nw // 3] = 0.0
    x = rng.standard_normal((steps, nw, X))
    s = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, taylor_order=order)
    s.set_walkers(phi, w)
    e, g = s.adjoint_run(steps, x, mgs_every=2, energy_every=steps, checkpoint=2)
    P = rng.standard_normal((M, M))
    P = P + P.T
    s.set_walkers(phi, w)
    s.set_tangent(P)
    for t in range(steps):
        s.propagate(1, x[t:t + 1])
        if (t + 1) % 2 == 0:
            s.orthonormalise()
    em, dm, _ = s.energy_tangent()
    assert abs(em[0] - e) < 1e-10 * abs(e)
    assert abs((g * P).sum() - dm[0]) < 1e-8 * np.abs(g * P).sum()
