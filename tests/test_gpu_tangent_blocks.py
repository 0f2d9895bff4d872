"""Forward-mode energies in digit form for the largest spin blocks, against the oracle's tangent.

Bounds: those of the oracle comparison in test_gpu_tangent.py (1e-9 of an energy, 1e-7 of a derivative)."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import afqmc as orc
from oracle import tangent as otan

pytestmark = pytest.mark.gpu


# around the block sizes at which the exchange sums stage fewer Cholesky vectors at a time
@pytest.mark.parametrize("M,X,nu,nd", [(40, 120, 20, 3), (40, 130, 21, 0), (48, 130, 27, 2), (64, 130, 28, 0),
                                       (40, 160, 30, 1), (64, 130, 32, 0)])
def test_large_blocks_match_the_oracle(M, X, nu, nd):
    afq = need_gpu()
    nw, dt = 6, 0.005
    rng = np.random.default_rng(M + 31 * nu)
    h1 = np.diag(np.linspace(-2, 3, M)) + 0.02 * rng.standard_normal((M, M))
    h1 = 0.5 * (h1 + h1.T)
    L = rng.standard_normal((X, M, M)) / np.sqrt(X * M)
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    P = rng.standard_normal((M, M)) * 0.01
    P = P + P.T
    fields = rng.standard_normal((5, nw, X))
    s = afq.System(h1, L, trial, nu, nd, dt=dt, n_walkers=nw)
    s.set_tangent(P)
    s.propagate(5, fields)
    s.orthonormalise()
    em, dm, _ = s.energy_tangent()
    ref, _, _ = otan.run(orc.System(h1, L, trial, nu, nd, dt), P, nw, 5, fields)
    np.testing.assert_allclose(em[0], ref[-1, 0], rtol=1e-9)
    np.testing.assert_allclose(dm[0], ref[-1, 1], rtol=1e-7, atol=1e-9 * np.abs(ref[:, 1]).max())
