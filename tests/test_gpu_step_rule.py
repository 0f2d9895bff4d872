"""FP64 steps on both sides of the rule for whole steps in one kernel: a call of two steps (that kernel) against
two calls of one (the separate kernels, at these populations), and a pair run of which one system, both or
neither takes it, against the two systems propagated on their own.

Bound 1e-12: two to five steps, each form within a few 1e-15 a step of well-conditioned walkers."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_gpu_step_small import system

pytestmark = pytest.mark.gpu
STEPS_SMALL = 4


def plan(afq, shape, nw, n):
    from paper_1703_01545_gb300 import _lib
    return _lib.load().afqmc_plan_value(STEPS_SMALL, *shape, nw, n)


@pytest.mark.parametrize("M,X,nu,nd,nw", [(8, 24, 2, 2, 2000), (12, 40, 3, 3, 700), (4, 8, 1, 0, 1700)])
def test_calls_of_one_and_of_two_steps_agree(M, X, nu, nd, nw):
    afq = need_gpu()
    assert plan(afq, (M, X, nu, nd), nw, 1) == 0 and plan(afq, (M, X, nu, nd), nw, 2) == 1
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, nw, M)
    x = rng.standard_normal((2, nw, X))
    w[3] = 0.0
    a, b = (afq.System(h1, L, trial, nu, nd, dt=0.01, n_walkers=nw) for _ in range(2))
    a.set_walkers(phi, w)
    b.set_walkers(phi, w)
    a.propagate(2, x)
    b.propagate(1, x[:1])
    b.propagate(1, x[1:])
    sa, sb = a.state(), b.state()
    assert np.array_equal(sa["alive"], sb["alive"]) and a.info().step == b.info().step == 2
    assert np.abs(sa["phi"] - sb["phi"]).max() < 1e-12
    assert np.abs(sa["w"] - sb["w"]).max() < 1e-12


# (M, X, n_up, n_dn) of the primary, walkers, whether A and B take the kernel for five steps
@pytest.mark.parametrize("shape,xb,nw,small", [((12, 40, 3, 3), 40, 300, (1, 1)), ((12, 40, 3, 3), 10, 2400, (0, 1)),
                                               ((12, 40, 3, 3), 40, 4000, (0, 0))])
def test_pair_run_matches_its_systems_on_their_own(shape, xb, nw, small):
    afq = need_gpu()
    M, X, nu, nd = shape
    assert (plan(afq, shape, nw, 5), plan(afq, (M, xb, nu, nd - 1), nw, 5)) == small
    h1, L, trial, phi, w, rng = system(M, X, nu, nd, 2, M)
    kw = dict(dt=0.01, n_walkers=nw, seed=5)
    mk = lambda: (afq.System(h1, L, trial, nu, nd, **kw), afq.System(h1, L[:xb], trial[:, :nu + nd - 1], nu, nd - 1, **kw))
    A, B = mk()
    res = afq.pair_delta_E(A, B, 5, energy_every=5, mgs_every=5)
    for k, (S, P) in enumerate(zip(mk(), (A, B))):
        S.propagate(5)
        S.orthonormalise()
        e = S.energy()[1][0]
        st, sp = S.state(), P.state()
        assert np.abs(st["phi"] - sp["phi"]).max() < 1e-12 and np.abs(st["w"] - sp["w"]).max() < 1e-12
        assert abs(res["E"][0, k, 0] - e) < 1e-12 * abs(e) * X
