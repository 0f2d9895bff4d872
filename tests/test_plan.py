"""Sizes and choices of the library's rules that need no device (afqmc_plan_value)."""
import pytest

ENERGY_DIGITS, ENERGY_T, TANGENT_T, EXCHANGE_SMEM, STEPS_SMALL = range(5)


@pytest.fixture(scope="module")
def plan():
    from paper_1703_01545_gb300 import _lib
    from paper_1703_01545_gb300.build import build
    build()
    return lambda what, shape, nw, arg=0: _lib.load().afqmc_plan_value(what, *shape, nw, arg)


# one walker's products take 1.1 MB at the first shape, 40 MB and more at the last two
@pytest.mark.parametrize("shape", [(96, 480, 12, 12), (128, 768, 16, 16), (64, 320, 8, 8), (66, 130, 32, 30),
                                   (64, 2500, 32, 1), (64, 3000, 32, 32)])
@pytest.mark.parametrize("nw", [1, 2, 3, 5, 36, 37, 300])
def test_tangent_products_stay_inside_the_energy_scratch(plan, shape, nw):
    held, filled = plan(ENERGY_T, shape, nw), plan(TANGENT_T, shape, nw)
    M, X, nu, nd = shape
    assert held % (2 * X * max(nu, nd) ** 2) == 0 and 0 < filled <= held
    if nw <= 2 and shape in ((96, 480, 12, 12), (128, 768, 16, 16)):
        assert plan(ENERGY_DIGITS, shape, nw) == 1   # a handle this small does take the digit form


@pytest.mark.parametrize("tangent", [0, 1])
def test_exchange_sums_fit_the_shared_memory_of_every_launch(plan, tangent):
    """48 KB need no raised limit, and every spin block up to the largest (32) is dispatched to them."""
    for ns in range(1, 33):
        assert 0 < plan(EXCHANGE_SMEM, (64, 130, ns, 0), 40, tangent) <= 48 * 1024


@pytest.mark.parametrize("shape,nw,steps,small", [
    ((8, 24, 2, 2), 128, 1, 1), ((8, 24, 2, 2), 128, 40, 1), ((8, 24, 2, 2), 1000, 1, 1),
    ((8, 24, 2, 2), 8000, 1, 0), ((8, 24, 2, 2), 40000, 1, 0), ((8, 24, 2, 2), 8000, 2, 1),
    ((8, 24, 2, 2), 40000, 2, 0), ((8, 24, 2, 2), 40000, 5, 1), ((12, 40, 3, 3), 300, 1, 1),
    ((12, 40, 3, 3), 1000, 1, 0), ((12, 40, 3, 3), 1000, 5, 1), ((12, 40, 3, 3), 4000, 8, 0),
    ((17, 40, 3, 3), 64, 5, 0)])
def test_whole_steps_of_small_systems_where_they_were_measured_faster(plan, shape, nw, steps, small):
    assert plan(STEPS_SMALL, shape, nw, steps) == small
