"""Split-precision refresh of large populations (its float64 overlap sums as digit contractions):
log <psi_T|phi> against numpy at float64 accuracy, for uneven spins, odd sizes and a last chunk of few
walkers, and the walkers' layout through host and device buffers.

Bound 1e-11: sums of M products of order one and an LU of blocks near the identity in float64."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,nu,nd,nw", [(128, 16, 15, 3000), (101, 13, 9, 4097), (200, 9, 9, 4096), (65, 16, 1, 5003)])
def test_refresh_matches_numpy(M, nu, nd, nw):
    afq = need_gpu()
    import torch
    rng = np.random.default_rng(M + nw)
    X, N = 40, nu + nd
    h1 = np.diag(np.linspace(-2, 3, M))
    L = rng.standard_normal((X, M, M)) * 0.01
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.3 / np.sqrt(M)
    s = afq.System(h1, L, trial, nu, nd, dt=0.005, n_walkers=nw, precision=afq.BF16X3, autotune=False)
    s.set_walkers(phi)
    st = s.state()
    assert np.array_equal(st["phi"], phi)
    ref = np.zeros(nw, complex)
    for a, b in ((0, nu), (nu, N)):
        sign, lad = np.linalg.slogdet(trial[:, a:b].T @ phi[:, :, a:b])
        ref += lad + np.log(sign)
    d = st["logO"] - ref
    d = d.real + 1j * (np.mod(d.imag + np.pi, 2 * np.pi) - np.pi)
    assert np.abs(d).max() < 1e-11
    # the same through device buffers
    pd = torch.from_numpy(np.ascontiguousarray(np.stack([phi.real, phi.imag]))).cuda()
    lo = torch.empty(2, nw, dtype=torch.float64, device="cuda")
    out = torch.empty_like(pd)
    afq.afqmc_set_walkers(s.h, pd)
    afq.afqmc_get_state(s.h, out, lo)
    assert torch.equal(out, pd)
    assert np.array_equal(lo.cpu().numpy(), np.stack([st["logO"].real, st["logO"].imag]))
