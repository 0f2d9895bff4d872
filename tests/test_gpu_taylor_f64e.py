"""One FP64 step of a large population (contractions and Taylor terms in digit form,
csrc/gemm_f64e.cu, csrc/taylor_f64e.cu) against the same walkers and fields on a handle of two
walkers (FP64-pipe kernels), at the edges of the row stacking (M <= 64), of the 128-row tiles, odd M
(the joined K is padded) and several Taylor orders.

Bound: the walkers of a step are sums of M to X products of numbers of order one, each form rounding
them to a few 1e-16; 1e-12 leaves three orders for the accumulation over the step."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

# (M, X, n_up, n_dn, walkers, order)
SHAPES = [(24, 70, 3, 2, 4096, 6), (63, 130, 8, 7, 900, 6), (64, 200, 8, 8, 2048, 1), (65, 150, 7, 6, 700, 6),
          (97, 300, 12, 11, 333, 9), (128, 260, 16, 16, 160, 6), (129, 200, 5, 4, 400, 6), (200, 310, 9, 9, 153, 6),
          (255, 120, 8, 8, 80, 3), (66, 110, 31, 30, 200, 2)]


@pytest.mark.parametrize("M,X,nu,nd,nw,order", SHAPES)
@pytest.mark.parametrize("mode", [0, 1])
def test_step_matches_walker_kernels(M, X, nu, nd, nw, order, mode):
    afq = need_gpu()
    if mode == 1 and nw > 1000:
        pytest.skip("one mode is enough at the largest populations")
    rng = np.random.default_rng(M * 17 + order)
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
    x = rng.standard_normal((1, nw, X))
    kw = dict(dt=0.01, taylor_order=order, mode=mode)
    big = afq.System(h1, L, trial, nu, nd, n_walkers=nw, **kw)
    big.set_walkers(phi, w)
    big.propagate(1, x)
    st = big.state()
    small = afq.System(h1, L, trial, nu, nd, n_walkers=2, **kw)
    for k in sorted({0, nw - 1, nw // 3, nw // 2, int(rng.integers(nw))}):
        small.set_walkers(phi[[k, k]], w[[k, k]])
        small.propagate(1, np.ascontiguousarray(x[:, [k, k]]))
        s1 = small.state()
        assert s1["alive"][0] == st["alive"][k]
        assert np.abs(s1["phi"][0] - st["phi"][k]).max() < 1e-12 * np.abs(s1["phi"][0]).max()
        assert abs(s1["w"][0] - st["w"][k]) <= 1e-11 * abs(s1["w"][0])
    # a walker that is not finite touches no other
    bad = phi.copy()
    bad[nw // 2, M // 2, 0] = np.inf
    big.set_walkers(bad, w)
    big.propagate(1, x)
    s2 = big.state()
    keep = np.arange(nw) != nw // 2
    assert np.array_equal(s2["phi"][keep], st["phi"][keep]) and np.array_equal(s2["w"][keep], st["w"][keep])
    assert not s2["alive"][nw // 2]
