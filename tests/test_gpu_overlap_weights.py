"""FP64 overlaps with the walkers' weights in the same kernel (few walkers) and in a second one (many): the same
walkers in both, through a refresh and a step, have the same bits; and few walkers take a launch less."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_gpu_step_small import system

pytestmark = pytest.mark.gpu
FEW, MANY = 912, 913   # six walkers' CTAs an SM: up to there they take the weights too


# (M, X, n_up, n_dn): one electron, blocks of 8, 9 to 10 and 16 (the kernel's three forms); M above 16, where a
# step is not one kernel, and sizes whose contractions do not depend on the number of walkers
@pytest.mark.parametrize("M,X,nu,nd", [(17, 6, 1, 0), (18, 5, 8, 3), (20, 4, 10, 9), (18, 4, 16, 11)])
@pytest.mark.parametrize("mode", [0, 1])
def test_one_and_two_kernels_give_the_same_bits(M, X, nu, nd, mode):
    afq = need_gpu()
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, MANY, M * 7 + nu)
    w[5] = 0.0                      # dead
    phi[6, :, 0] = 0.0              # singular
    phi[7, 2, 0] = np.nan
    x = rng.standard_normal((1, MANY, X))
    x[0, 9] = 1e200                 # overflows in the step
    out = []
    for nw in (FEW, MANY):
        g = afq.System(h1, L, trial, nu, nd, dt=0.05, n_walkers=nw, mode=mode)
        g.set_walkers(phi[:nw], w[:nw])
        first = g.state()
        g.propagate(1, np.ascontiguousarray(x[:, :nw]))
        out.append((first, g.state()))
    for a, b in zip(*out):
        assert list(a["alive"][5:8]) == [False] * 3
        for k in ("logO", "w", "alive", "phi"):
            np.testing.assert_array_equal(a[k], b[k][:FEW])


def test_few_determinants_match_many():
    """The records of a multi-determinant trial: 114 walkers of 8 determinants, against 115."""
    afq = need_gpu()
    M, X, nu, nd, ndet = 17, 5, 3, 2, 8
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, 115, 3)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    dets = np.stack([trial + 0.3 * np.concatenate([q[:, k:k + nu], q[:, k:k + nd]], axis=1) for k in range(ndet)])
    out = []
    for nw in (114, 115):
        g = afq.System(h1, L, None, nu, nd, dt=0.05, n_walkers=nw, dets=dets, coeffs=1.0 / np.arange(1, ndet + 1))
        g.set_walkers(phi[:nw], w[:nw])
        g.propagate(1, np.full((1, nw, X), 0.3))
        out.append(g.state())
    for k in ("logO", "w", "alive", "phi"):
        np.testing.assert_array_equal(out[0][k], out[1][k][:114])


def test_few_walkers_take_a_launch_less():
    afq = need_gpu()
    M, X, nu, nd = 18, 8, 2, 2
    h1, L, trial, _, _, _ = system(M, X, nu, nd, 2, 4)
    count = []
    for nw in (FEW, MANY):
        A, B = (afq.System(h1, L, trial[:, :nu + n], nu, n, dt=0.01, n_walkers=nw, seed=3) for n in (nd, nd - 1))
        afq.pair_delta_E(A, B, 5, energy_every=5, mgs_every=5)
        count.append(afq.pair_graph_kernels(A))
    assert count[1] - count[0] == 2 * (5 + 1)   # per system: five steps and the orthonormalisation's refresh
