"""Tensor-core FP64 products with infinities, NaN and subnormal entries give what FP64 sums give: signed
infinities, NaN only where a sum has one, subnormal rows not lost."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_special_values(tmp_path):
    out = run_driver(tmp_path, "product_special_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc"))
    lines = out.split("\n")[:-1]
    assert len(lines) == 4
    for line in lines:
        kinds, worst = line.split()
        # both round to about K^(1/2) 2^-53 of the norms at most: 260^(1/2) 2^-53 < 2^-48.9, halved for either side's mean
        assert int(kinds) == 0 and float(worst) <= 4.0, out
