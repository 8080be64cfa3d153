"""The reciprocal and reciprocal root of the dense kernels over the whole exponent range.  rsqrt: the product x y
rounds once (2^-53 of the residual, halved), the result once: 1.5 units of 2^-53; rcp: the result alone, 1 unit;
what the series leaves, 2^-64 and 2^-70, is below 0.01.  Zero, infinities, NaN and negative values as CUDA's."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_against_division_and_root(tmp_path):
    out = run_driver(tmp_path, "reciprocal_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc"))
    (rsqrt, k1), (rcp, k2) = [line.split() for line in out.split("\n")[:2]]
    assert int(k1) == 0 and int(k2) == 0, out
    assert float(rsqrt) <= 1.51 and float(rcp) <= 1.01, out
