"""The FP32 overlap update's forms (an entry per four lanes, register tiles, tiles with more registers) on both
sides of their rule, and the Cholesky QR's for blocks up to 8 and up to 16.

Bounds: the update's as in test_gpu_overlap_tile.py; the QR's 5e-6, some M + 10 ns FP32 roundings of 2^-24 of
walkers near the identity."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_gpu_overlap_tile import test_update as check_update

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw", [
    (22, 20, 1, 1, 7), (24, 30, 4, 4, 20), (24, 30, 5, 4, 21), (48, 30, 8, 1, 9), (128, 30, 8, 8, 9), (64, 30, 10, 10, 9),
    (64, 30, 11, 9, 9), (66, 30, 9, 16, 8), (128, 30, 13, 12, 9)])
def test_update_forms(M, X, nu, nd, nw):
    check_update(M, X, nu, nd, nw)


@pytest.mark.parametrize("M,nu,nd", [(9, 1, 0), (33, 8, 8), (40, 8, 1), (33, 9, 3), (66, 16, 0), (128, 16, 16)])
def test_cholesky_qr(M, nu, nd):
    afq = need_gpu()
    nw = 40
    rng = np.random.default_rng(M + nu)
    L = rng.standard_normal((4, M, M)) * 0.1
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.2 / np.sqrt(M)
    g = afq.System(np.eye(M), L + np.swapaxes(L, 1, 2), trial, nu, nd, dt=0.01, n_walkers=nw, precision=afq.BF16X3,
                   autotune=False)
    g.select_kernel(afq.K_MGS, 1)
    g.set_walkers(phi)
    g.orthonormalise()
    got = g.state()["phi"]
    for a, b in ((0, nu), (nu, N)):
        if b == a:
            continue
        r = np.linalg.cholesky(np.conj(np.swapaxes(phi[:, :, a:b], 1, 2)) @ phi[:, :, a:b])
        ref = np.swapaxes(np.linalg.solve(np.conj(r), np.swapaxes(phi[:, :, a:b], 1, 2)), 1, 2)
        assert np.abs(got[:, :, a:b] - ref).max() < 5e-6
