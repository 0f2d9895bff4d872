"""Forward-mode energies in digit form with one and two walkers, whose products and derivatives share a
chunk of a single walker, against the oracle's tangent.

Bounds: those of the oracle comparison in test_gpu_tangent.py (1e-9 of an energy, 1e-7 of a derivative)."""
import numpy as np
import pytest

from gpu_util import need_gpu, system_data
from oracle import afqmc as orc
from oracle import tangent as otan
from synthetic import explicit_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nw", [1, 2, 3])
def test_few_walkers_match_the_oracle(nw):
    afq = need_gpu()
    d = system_data("C5", "A", "moderate")   # M = 96, X = 480, 12/12
    steps, dt = 5, 0.01
    fields = explicit_fields(steps, nw, d["X"], seed=7)
    P = np.random.default_rng(3).standard_normal((d["M"], d["M"])) * 0.01
    P = P + P.T
    s = afq.System(d["h1"], d["L"], d["trial"], d["n_up"], d["n_dn"], dt=dt, n_walkers=nw)
    s.set_tangent(P)
    s.propagate(steps, fields)
    s.orthonormalise()
    em, dm, _ = s.energy_tangent()
    ref, _, tw = otan.run(orc.System(d["h1"], d["L"], d["trial"], d["n_up"], d["n_dn"], dt), P, nw, steps, fields)
    np.testing.assert_allclose(em[0], ref[-1, 0], rtol=1e-9)
    np.testing.assert_allclose(dm[0], ref[-1, 1], rtol=1e-7, atol=1e-9 * np.abs(ref[:, 1]).max())
    np.testing.assert_allclose(s.tangent_state(), tw.dlogw, rtol=1e-7, atol=1e-9 * np.abs(tw.dlogw).max())
