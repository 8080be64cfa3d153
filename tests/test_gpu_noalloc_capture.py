"""After wt_eq1_noalloc was captured into a graph, the sensor relaxes again, closes, and other sensors work: no
event of the capture is waited for."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks

pytestmark = pytest.mark.gpu


def test_relax_and_close_after_a_capture():
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=12, radius=8e-6)

    def sensor():
        s = P.Sensor(w.grid, w.columns)
        s.fit()
        s.relax(w.times)
        return s

    s = sensor()
    H = s.extend("fp32")
    tr = device_tracks(W.configs.mip_tracks(w.grid, 4, 20, np.random.default_rng(1)), torch)
    out = torch.zeros((4, tr["n_out"]), device="cuda")
    P.wt_eq1_noalloc(s.ctx, H, tr, out)
    torch.cuda.synchronize()
    want = out.clone()
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=st):
        P.wt_eq1_noalloc(s.ctx, H, tr, out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    s.relax(w.times)
    s.close()
    other = sensor()
    assert other.info()["rank"] >= 1
    other.close()
