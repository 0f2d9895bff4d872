"""The FP64 local energy in digit form (csrc/energy_f64e.cu, taken by handles with many walkers)
against the per-walker FP64 kernel (taken by a handle with a few) and the oracle, at uneven spins,
odd sizes and walker counts that do not divide the chunks.

Bound: both forms round each of the X sum_s N_s^2 terms T_ab T_ba to a few 1e-16 of max |T|^2; a
relative 1e-12 of the energy's largest part leaves two orders for their sum and cancellation."""
import numpy as np
import pytest

from gpu_util import need_gpu
from oracle import afqmc as orc

pytestmark = pytest.mark.gpu


# (M, X, n_up, n_dn, walkers): one spin only, one electron in a spin, spins of 17 to 32 (several
# chunks of T), K beyond one block, walkers that leave a short last chunk
SHAPES = [(20, 64, 5, 0, 700), (33, 90, 5, 1, 611), (70, 300, 9, 8, 1101), (64, 320, 8, 7, 2048),
          (96, 200, 23, 19, 301), (66, 130, 32, 30, 97), (130, 257, 4, 4, 1500)]


@pytest.mark.parametrize("M,X,nu,nd,nw", SHAPES)
def test_digit_energy_matches_walker_kernel_and_oracle(M, X, nu, nd, nw):
    afq = need_gpu()
    rng = np.random.default_rng(M * 31 + X)
    h1 = rng.standard_normal((M, M))
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) * 0.1
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    phi = trial + (rng.standard_normal((nw, M, nu + nd)) + 1j * rng.standard_normal((nw, M, nu + nd))) * 0.2 / np.sqrt(M)
    big = afq.System(h1, L, trial, nu, nd, dt=0.005, n_walkers=nw)
    big.set_walkers(phi)
    el, em, ws = big.energy()
    pick = np.unique(np.concatenate([[0, nw - 1], rng.integers(0, nw, 6)]))
    small = afq.System(h1, L, trial, nu, nd, dt=0.005, n_walkers=2)
    osys = orc.System(h1, L, trial, nu, nd, 0.005)
    ref = orc.local_energy(osys, phi[pick])
    scale = np.abs(ref).max()
    assert np.abs(el[pick] - ref).max() < 1e-12 * scale * X
    for k in pick:
        small.set_walkers(phi[[k, k]])
        es = small.energy()[0]
        assert abs(es[0] - el[k]) < 1e-12 * scale
    assert abs(em[0] - el.real.mean()) < 1e-12 * scale
    # a walker that is not finite stays on its own
    bad = phi.copy()
    bad[nw // 2, 0, 0] = np.nan
    big.set_walkers(bad)
    keep = np.arange(nw) != nw // 2
    assert np.array_equal(big.energy()[0][keep], el[keep])
