"""Capturing an FP32 extension into a graph computes nothing yet: calls that take the basis fields it would have
left (loss, currents without the field, derivative) compute their own until the graph has run."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks

pytestmark = pytest.mark.gpu


def test_captured_extension_leaves_no_fields():
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=12, radius=8e-6)
    other = 3.0 * w.times
    tr = device_tracks(W.configs.mip_tracks(w.grid, 5, 12, np.random.default_rng(4)), torch)

    def fresh():
        s = P.Sensor(w.grid, w.columns)
        s.fit()
        return s

    ref = fresh()
    ref.relax(other)
    s = fresh()
    s.relax(w.times)
    H = s.extend("fp32")                              # launch shapes, buffers, the first times' basis fields
    torch.cuda.synchronize()
    s.relax(other)
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.extend("fp32", out=H, stream=st.cuda_stream)
    assert s.loss(tr, "fp32") == pytest.approx(ref.loss(tr, "fp32"), rel=1e-5)       # the FP32 path's bound
    i, want = s.eq1_direct(tr), ref.eq1_direct(tr)
    assert torch.linalg.norm(i - want) < 1e-5 * torch.linalg.norm(want)
    g.replay()
    torch.cuda.synchronize()
    Href = ref.extend("fp32")
    torch.cuda.synchronize()
    assert torch.linalg.norm(H - Href) < 1e-5 * torch.linalg.norm(Href)
    s.close()
    ref.close()
