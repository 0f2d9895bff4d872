"""Two handles in forward mode: the smaller one, set up later, leaves the larger one's launches valid."""
import numpy as np
import pytest

from gpu_util import need_gpu
from test_gpu_step_small import system

pytestmark = pytest.mark.gpu


def test_a_smaller_handle_does_not_lower_the_limits_of_a_larger_one():
    afq = need_gpu()
    out = []
    for second in (False, True):
        h1, L, trial, phi, w, rng = system(70, 20, 10, 9, 6, 1)
        big = afq.System(h1, L, trial, 10, 9, dt=0.01, n_walkers=6)   # 85 KB of shared memory in forward mode
        big.set_walkers(phi, w)
        big.set_tangent(np.eye(70))
        if second:
            g1, K, tr, _, _, _ = system(4, 5, 1, 1, 6, 2)
            small = afq.System(g1, K, tr, 1, 1, dt=0.01, n_walkers=6)
            small.set_tangent(np.eye(4))
            small.propagate(1)
        big.propagate(1, np.ones((1, 6, 20)))
        big.orthonormalise()
        out.append(big.energy_tangent())
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
