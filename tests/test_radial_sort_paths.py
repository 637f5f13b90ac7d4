"""The paths of the radial sort (one block, buckets, radix passes) answer alike:
what one reports the others report."""
import numpy as np
import pytest
import torch

from paper_1406_4254_gb300 import etics, inputs

pytestmark = pytest.mark.gpu

DTYPES = {"mixed": torch.float32, "fp64": torch.float64}
# one block up to 7168 particles, buckets up to 1867776, radix passes above
ONE_BLOCK, BUCKETS, RADIX = 7168, 1867776, 1867777


def device(pm, precision):
    return torch.tensor(pm, dtype=DTYPES[precision], device="cuda")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n", [1, 5000, ONE_BLOCK, ONE_BLOCK + 1, RADIX])
def test_order_reports_a_nonfinite_particle(n, bad, precision):
    x = device(inputs.hernquist(n, seed=3), precision)
    for at, column in ((0, 0), (n // 2, 2), (n - 1, 3)):   # the mass counts as well
        y = x.clone()
        y[at, column] = bad
        order = etics.radial_order(y)
        assert etics.get_error() == etics.ERR_NONFINITE, (at, column)
        assert int(order[-1]) == at       # such a particle sorts last
        etics.mex_field(y, 2)
        assert etics.get_error() == etics.ERR_NONFINITE, (at, column)
    etics.radial_order(x)
    assert etics.get_error() == 0
