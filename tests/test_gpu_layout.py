"""Walkers in and out of a handle, whose matrices share a CTA when they are small: exact, at both sides of the
rule (128 numbers; two CTAs an SM) and with a last CTA that is not full."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,nu,nd", [(1, 1, 0), (2, 1, 1), (5, 1, 0), (9, 4, 3), (16, 4, 4), (43, 2, 1), (61, 2, 0),
                                     (64, 32, 32)])
@pytest.mark.parametrize("nw", [1, 7, 303, 305, 1999])
def test_state_returns_what_was_set(M, nu, nd, nw):
    afq = need_gpu()
    rng = np.random.default_rng(M + nw)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    L = rng.standard_normal((2, M, M)) * 0.1
    s = afq.System(np.eye(M), L + np.swapaxes(L, 1, 2), trial, nu, nd, dt=0.01, n_walkers=nw)
    phi = rng.standard_normal((nw, M, nu + nd)) + 1j * rng.standard_normal((nw, M, nu + nd))
    s.set_walkers(phi)
    np.testing.assert_array_equal(s.state()["phi"], phi)
