"""Column-pivoted QR of a charge history, for columns that fit a block's shared memory and for longer ones
(more than about 28 000 sources)."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_columns_of_any_length(tmp_path):
    cases = [(40, 40), (2304, 40), (28000, 24), (30000, 24), (60001, 33)]
    out = run_driver(tmp_path, "qr_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc"),
                     "".join(f"{a} {b}\n" for a, b in cases))
    lines = out.split("\n")[:-1]
    assert len(lines) == len(cases)
    for line in lines:
        worst, falls = line.split()
        # Householder steps: the error of a column is at most about n_t steps x a few eps of its norm
        assert float(worst) < 40 * 8 * 2.3e-16 * 2 and int(falls) == 1, out
