"""The collisions' reciprocals (collide.cuh) are the IEEE quotient 1/x: the packed
one for every float of its range, both signs, the scalar one for every float,
zeros, denormals, infinities and NaN among them."""
import pytest

pytestmark = pytest.mark.gpu


def test_reciprocals_equal_the_quotient(lbmlib, cuda):
    import torch
    bad = torch.full((2,), 77, dtype=torch.int64, device=cuda)
    lbmlib.lbm_selftest_reciprocal(bad)
    assert bad.tolist() == [0, 0]
