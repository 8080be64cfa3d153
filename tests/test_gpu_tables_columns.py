"""The FP64 field from tables for any number of columns: up to 1 600 columns' coefficients of 16 samples fit a
block's shared memory, more take fewer samples at a time."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_any_number_of_columns(tmp_path):
    cases = [(1, 5), (18, 16), (1600, 16), (1601, 16), (2200, 33), (6401, 4), (12800, 3)]
    out = run_driver(tmp_path, "tables_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc", "k_tables64"),
                     "".join(f"{a} {b}\n" for a, b in cases))
    lines = out.split("\n")[:-1]
    assert len(lines) == len(cases), out
    for line, (n_cols, _) in zip(lines, cases):
        assert float(line) < (n_cols + 8) * 1.2e-16, out          # one rounding per multiply-add at most
