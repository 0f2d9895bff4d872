"""FP64 local energies in digit form against extended precision, for few walkers (handles of two that take the
digit form too) and many, at the largest blocks, and forward-mode energies after two steps against the oracle's.

Bounds: the energy's of test_gpu_energy_f64e.py (1e-12 of the largest energy), the derivative's of
test_gpu_tangent_f64e.py (1e-10 of the largest derivative)."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import afqmc as orc
from oracle import tangent as otan

pytestmark = pytest.mark.gpu


def system(M, X, nu, nd, nw, scale):
    rng = np.random.default_rng(M * 7 + nu)
    h1 = np.diag(np.linspace(-2, 3, M)) + 0.02 * rng.standard_normal((M, M))
    h1 = 0.5 * (h1 + h1.T)
    L = rng.standard_normal((X, M, M)) * scale
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    N = nu + nd
    phi = trial + (rng.standard_normal((nw, M, N)) + 1j * rng.standard_normal((nw, M, N))) * 0.2 / np.sqrt(M)
    return h1, L, trial, phi, rng


def energy_extended(h1, L, trial, phi, spins):
    """E_L of one walker with every sum in the widest float numpy has (Theta by two refinements)."""
    ld, cld = np.longdouble, np.clongdouble
    one, rho, ex = cld(0), np.zeros(L.shape[0], cld), cld(0)
    for a, b in spins:
        p, f = trial[:, a:b].astype(ld), phi[:, a:b].astype(cld)
        O = p.T @ f
        inv = np.linalg.inv(O.astype(np.complex128)).astype(cld)
        for _ in range(2):
            inv = inv @ (2 * np.eye(b - a).astype(cld) - O @ inv)
        th = f @ inv
        lt = (L.astype(ld) @ p).transpose(0, 2, 1).reshape(-1, L.shape[1])
        T = (lt @ th.real + 1j * (lt @ th.imag)).reshape(L.shape[0], b - a, b - a)
        one += ((h1.astype(ld) @ p) * th).sum()
        rho += np.trace(T, axis1=1, axis2=2)
        ex += (T * T.transpose(0, 2, 1)).sum()
    return one + ((rho * rho).sum() - ex) / 2


@pytest.mark.parametrize("M,X,nu,nd,nw", [(96, 200, 23, 19, 2), (96, 60, 23, 19, 301), (66, 130, 32, 30, 2),
                                          (66, 60, 32, 30, 97), (40, 120, 12, 5, 64)])
def test_energy(M, X, nu, nd, nw):
    afq = need_gpu()
    assert afq.afqmc_plan_value(0, M, X, nu, nd, nw) == 1
    h1, L, trial, phi, _ = system(M, X, nu, nd, nw, 0.1)
    s = afq.System(h1, L, trial, nu, nd, dt=0.005, n_walkers=nw)
    s.set_walkers(phi)
    el = s.energy()[0]
    pick = sorted({0, nw // 2, nw - 1})
    ref = np.array([energy_extended(h1, L, trial, phi[k], ((0, nu), (nu, nu + nd))) for k in pick])
    assert np.abs(el[pick] - ref).max() < 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("nw", [3, 160])
def test_tangent(nw):
    afq = need_gpu()
    M, X, nu, nd, dt = 98, 200, 9, 8, 0.01
    assert afq.afqmc_plan_value(0, M, X, nu, nd, nw) == 1
    h1, L, trial, phi, rng = system(M, X, nu, nd, nw, 1 / np.sqrt(X * M))
    x = rng.standard_normal((2, nw, X))
    P = rng.standard_normal((M, M))
    P = P + P.T
    s = afq.System(h1, L, trial, nu, nd, dt=dt, n_walkers=nw)
    s.set_walkers(phi)
    s.set_tangent(P)
    s.propagate(2, x)
    _, _, de = s.energy_tangent()
    pick = np.array([0, nw // 2, nw - 1])
    o = orc.System(h1, L, trial, nu, nd, dt)
    ts, wk = otan.TangentSystem(o, P), orc.Walkers(o, 3, phi[pick])
    tw = otan.TangentWalkers(wk)
    for t in range(2):
        otan.propagate(ts, wk, tw, x[t][pick])
    _, ref = otan.local_energy_tangent(ts, wk.phi, tw.dphi)
    assert np.abs(de[pick] - ref).max() < 1e-10 * np.abs(ref).max()
