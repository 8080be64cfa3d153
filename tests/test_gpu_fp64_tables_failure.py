"""The lateral tables of the FP64 field: a build that finds no memory leaves one transform per sample, one whose
wait runs out is reported, and neither leaves tables behind that a later call would take for complete."""
import os
from contextlib import contextmanager

import pytest

import workloads as W
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu


@contextmanager
def fault(name):
    os.environ["WT_FAULT"] = name
    try:
        yield
    finally:
        os.environ.pop("WT_FAULT", None)


@pytest.mark.parametrize("name", ["tables_oom", "tables_timeout"])
def test_failed_tables_are_not_used(name):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=40, radius=0.5 * 55e-6 / 16)
    good = P.Sensor(w.grid, w.columns)
    good.fit()
    good.relax(w.times)
    want = good.extend("fp64")
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    with fault(name):
        if name == "tables_oom":
            H = s.extend("fp64")
            s.sync()
            assert rel_l2(H.cpu().numpy(), want.cpu().numpy()) < 1e-12      # the same charges, two forms that round at 1e-15
            assert not torch.equal(H, want)
        else:
            with pytest.raises(P.WTError, match="WT_ERR_TIMEOUT"):
                s.extend("fp64")
    H = s.extend("fp64")
    s.sync()
    assert torch.equal(H, want)
    good.close()
    s.close()


def test_little_memory_left():
    """Smaller pieces, and one transform per sample, where the device is nearly full."""
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=64, nz=32, n_t=200, m_req=16, radius=0.5 * 55e-6 / 64)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    want = s.extend("fp64")
    s.sync()
    s.close()
    torch.cuda.empty_cache()
    for left in (700 << 20, 180 << 20, 40 << 20):
        s = P.Sensor(w.grid, w.columns)
        s.fit()
        s.relax(w.times)
        s.static_field([1.0, 0.0], "fp64")                 # the per-sample transform's own buffers
        H = torch.empty_like(want)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        hold = torch.empty(max(0, free - left), dtype=torch.uint8, device="cuda")
        s.extend("fp64", out=H)
        s.sync()
        del hold
        torch.cuda.empty_cache()
        assert rel_l2(H.cpu().numpy(), want.cpu().numpy()) < 1e-12
        s.close()
