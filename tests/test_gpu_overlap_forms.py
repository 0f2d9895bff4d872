"""The FP32 overlap update's forms (an entry per four lanes, register tiles, tiles with more registers) on both
sides of their rule.

Bounds: as in test_gpu_overlap_tile.py."""
import pytest

from test_gpu_overlap_tile import test_update as check_update

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,X,nu,nd,nw", [
    (22, 20, 1, 1, 7), (24, 30, 4, 4, 20), (24, 30, 5, 4, 21), (48, 30, 8, 1, 9), (128, 30, 8, 8, 9), (64, 30, 10, 10, 9),
    (64, 30, 11, 9, 9), (66, 30, 9, 16, 8), (128, 30, 13, 12, 9)])
def test_update_forms(M, X, nu, nd, nw):
    check_update(M, X, nu, nd, nw)
