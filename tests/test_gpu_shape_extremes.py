"""Shaping with time constants for which (dt / tau)^order leaves the FP64 range: many tracks as few, finite and as
the sum over taps gives it."""
import numpy as np
import pytest

import workloads as W
from oracle import electronics as E

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,ratio,gain", [(2, 1e160, 1.0), (4, 1e100, 1.0), (20, 1e-16, 1e290)])
@pytest.mark.parametrize("n_tracks", [3, 9000])
def test_many_tracks_as_few(order, ratio, gain, n_tracks):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=4, radius=8e-6)
    s = P.Sensor(w.grid, w.columns)
    i = np.random.default_rng(order).standard_normal((n_tracks, 64)).astype(np.float32)
    dt = 1e-11
    v = s.shape(torch.tensor(i, device="cuda"), dt, dt / ratio, order, gain=gain)[:3].cpu().numpy()
    s.close()
    # a response that has decayed before the first sample after its start, and is zero at its start, gives nothing
    ref = np.zeros_like(v) if ratio > 1 else E.shape(i[:3], dt, dt / ratio, order, gain=gain)
    assert np.isfinite(v).all()
    # FP32 rounding of the result: 2^-24 of each value
    assert np.linalg.norm(v - ref) <= 1e-7 * np.linalg.norm(ref)
