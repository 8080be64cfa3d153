"""Memory that a call holds for reuse does not make a later allocation of the same call fail."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_call_memory_gives_back_what_nothing_uses(tmp_path):
    out = run_driver(tmp_path, "memory_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc"))
    assert out.split("\n")[:-1] == ["ok"] * 4, out
