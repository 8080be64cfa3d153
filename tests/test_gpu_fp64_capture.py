"""An FP64 extension captured into a CUDA graph replays to the same bits after other FP64 calls of the same
sensor (static field, extension, loss), whose buffers are their own."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_t", [3, 12, 30, 70])      # one transform per sample; from tables in one piece
def test_replay_after_other_calls(n_t):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=n_t, radius=0.5 * 55e-6 / 16)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    H = s.extend("fp64")                              # sizes the buffers
    torch.cuda.synchronize()
    want = H.clone()
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.extend("fp64", out=H, stream=st.cuda_stream)
    tr = device_tracks(W.configs.mip_tracks(w.grid, 3, 12, np.random.default_rng(4)), torch)
    E = s.static_field([1.0, 0.0], "fp64")
    other = s.extend("fp64")
    loss = s.loss(tr, "fp64")
    hold = [torch.full((n,), float("nan"), dtype=torch.float64, device="cuda") for n in (1 << 10, 1 << 16, 1 << 20, 1 << 22)]
    H.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(H, want)                       # nothing else wrote the captured call's buffers
    assert torch.equal(other, want)
    # and the other calls go on as before
    assert torch.equal(s.static_field([1.0, 0.0], "fp64"), E) and s.loss(tr, "fp64") == loss
    del hold
    s.close()
