"""Eq. 1 from the rank-r form for tracks of 1 to 20 steps (up to 8 by the staged product, more by the convolution),
against the stored field's form and for calls of different sizes one after the other on one sensor."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks, rel_l2

pytestmark = pytest.mark.gpu


def test_few_steps_and_changing_sizes():
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=12, radius=8e-6)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    H = s.extend("fp32")
    first = {}
    for n_steps, n_out in ((1, 1), (7, 300), (8, 16), (9, 18), (9, 780), (8, 784), (20, 40), (8, 800), (9, 800), (9, 18), (20, 40)):
        t = W.configs.mip_tracks(w.grid, 30, n_steps, np.random.default_rng(n_steps))
        t.n_out = n_out
        tr = device_tracks(t, torch)
        a, b = s.eq1_direct(tr), s.eq1(H, tr)
        # both sum FP32 products of the same FP32 basis fields: 1e-5 of the norm, as between the two forms elsewhere
        assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) < 1e-5
        assert torch.equal(a, first.setdefault((n_steps, n_out), a))
    s.close()
