"""The same derivative call gives the same tangents, bit for bit, on a cell whose symmetry makes modes coincide,
so that the sums over modes take pairs without a gap (at most 256 sources: no sums by atomics elsewhere)."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks
from workloads.configs import OHM_CM, UM, pixel_matrix

pytestmark = pytest.mark.gpu


def test_tangents_repeat():
    import torch
    import paper_2605_13987_gb300 as P
    grid, cols = pixel_matrix(3, 55 * UM, 100 * UM, 24, 32, 5 * UM, 0.3 * OHM_CM, 0.3 * OHM_CM, 14,
                              np.random.default_rng(11))
    assert sum(c.n_sources for c in cols) <= 256
    w = W.Workload("sym3x3", grid, cols, W.FitSpec(), W.log_times(48), seed=11)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    mu = s.modes()
    assert np.sum(np.diff(mu) <= 1e-9 * mu[1:]) >= 10
    tr = device_tracks(W.configs.mip_tracks(w.grid, 20, 30, np.random.default_rng(4)), torch)
    i0, di0, _, _ = s.tangents(tr)
    for _ in range(20):
        i, di, _, _ = s.tangents(tr)
        assert torch.equal(i, i0) and torch.equal(di, di0)
    s.close()
