"""Memory that a call holds for reuse does not make a later allocation of the same call fail."""
import pytest

from tests.driver_build import run_driver

pytestmark = pytest.mark.gpu


def test_call_memory_gives_back_what_nothing_uses(tmp_path):
    out = run_driver(tmp_path, "memory_driver", ("k_dense", "k_dgemm_tc", "k_expand_tc"))
    assert out.split("\n")[:-1] == ["ok"] * 4, out


def test_points_with_little_memory_left():
    """Exact point values where the sums of 512 points at a time do not fit: fewer points at a time."""
    import numpy as np
    import torch
    import paper_2605_13987_gb300 as P
    import workloads as W
    w = W.tiny_cell(nx=96, nz=128, n_t=8, m_req=32, radius=2.5 * 55e-6 / 96)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    xyz = np.random.default_rng(2).uniform(0, 1, (600, 3)) * [w.grid.Lx, w.grid.Ly, w.grid.Lz]
    want = s.sample_H(xyz, w.times)
    torch.cuda.empty_cache()
    for left in (90, 45, 30):                          # MB; the sums of 512 points take 101
        hold = torch.empty(torch.cuda.mem_get_info()[0] - (left << 20), dtype=torch.uint8, device="cuda")
        got = s.sample_H(xyz, w.times)
        del hold
        torch.cuda.empty_cache()
        # the same sums, by the tensor cores or, without their workspace, the FP64 units; scaled by other norms
        assert np.linalg.norm(got - want) < 1e-12 * np.linalg.norm(want)
    s.close()
