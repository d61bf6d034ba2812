"""Finite-difference planes around three blocks per SM (152 SMs, a block a row
here), where the step changes its kernel again, against the oracle as in the
test it calls."""
import pytest

import test_gpu_fd_plane as fd_plane

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["D2Q37", "D2Q49"])
@pytest.mark.parametrize("shape", [(40, 16), (5, 456), (5, 457), (5, 608)])
@pytest.mark.parametrize("bc,n", [(("copy", "copy"), 3), (("periodic", "copy"), 0)])
def test_one_step(orc, kind, shape, bc, n):
    fd_plane.test_one_step(orc, kind, shape, bc, n)
