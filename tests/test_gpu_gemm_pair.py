"""Split-BF16 contraction by pairs of SMs (256 x 256 tiles over two CTAs) at the edges of its rule, against
numpy float64: an even and an odd number of 128-row tiles (the last pair's second CTA empty), two waves of
pairs where single tiles take three, a single row tile (one CTA per tile), rows and columns that end inside a
tile, one k slice, fewer slices than the ring, K that is no multiple of 64.

Bound as for the other split-BF16 contractions: operands to 2^-17, lo * lo dropped (2^-18), FP32 sums:
|C - C_ref| <= (2^-15 + K 2^-23) (|A| |B|^T)."""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Md,Nd,K", [
    (2560, 4096, 64), (2500, 4352, 130), (1408, 7168, 200), (1301, 7100, 1), (1152, 8704, 100),
    (256, 39000, 72), (130, 38912, 300),
    (768, 8192, 330), (1000, 4096, 200), (100, 78000, 64)])
def test_pair_contraction(Md, Nd, K):
    need_gpu()
    from paper_1703_01545_gb300 import _lib
    lib = _lib.load()
    rng = np.random.default_rng(Md + Nd + K)
    A = rng.standard_normal((Md, K))
    B = rng.standard_normal((Nd, K))
    C = np.empty((Nd, Md))
    assert lib.afqmc_test_gemm(1, Md, Nd, K, A.ctypes.data, B.ctypes.data, 1.0, C.ctypes.data, None) == 0
    bound = (2.0 ** -15 + K * 2.0 ** -23) * (np.abs(B) @ np.abs(A).T)
    assert np.all(np.abs(C - B @ A.T) <= bound)


@pytest.mark.parametrize("M,X,nu,nd,nw", [(33, 40, 5, 4, 4096), (97, 70, 3, 2, 768), (129, 33, 4, 3, 512), (128, 20, 2, 2, 640)])
def test_lower_triangle_output(M, X, nu, nd, nw):
    """The V_HS form (lower-triangle block rows, split, both halves written) through a step of the
    tensor-core propagator that reads it, against the oracle on sampled walkers; odd M, where a row's last
    pair reaches into the padding.  5e-4 of the largest element, as for the propagator itself."""
    afq = need_gpu()
    from oracle import afqmc as orc
    rng = np.random.default_rng(M)
    h1 = rng.standard_normal((M, M)) * (0.3 / np.sqrt(M))
    h1 = h1 + h1.T
    L = rng.standard_normal((X, M, M)) * (0.6 / np.sqrt(X * M))
    L = L + np.swapaxes(L, 1, 2)
    q = np.linalg.qr(rng.standard_normal((M, M)))[0]
    trial = np.concatenate([q[:, :nu], q[:, :nd]], axis=1)
    g = afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw, precision=afq.BF16X3, autotune=False)
    g.select_kernel(afq.K_TAYLOR, 4)
    x = rng.standard_normal((1, nw, X))
    g.propagate(1, x)
    st = g.state()
    pick = np.array([0, 1, nw // 2 + 3, nw - 1])
    o = orc.System(h1, L, trial, nu, nd, 0.01)
    wk = orc.Walkers(o, len(pick))
    orc.propagate(o, wk, x[0][pick])
    assert np.abs(st["phi"][pick] - wk.phi).max() < 5e-4 * np.abs(wk.phi).max()
    assert np.all(np.isfinite(st["phi"]))
    g.close()
