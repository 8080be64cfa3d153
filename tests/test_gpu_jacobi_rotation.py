"""A Jacobi rotation of the time basis takes its angle in FP64: one rotation leaves two rows orthogonal to
rounding (64 products of a dot product, and the rounding of the rotated entries)."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_one_rotation_is_enough(tmp_path):
    out = run_driver(tmp_path, "jacobi_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc"))
    assert float(out) <= 1.0, out
