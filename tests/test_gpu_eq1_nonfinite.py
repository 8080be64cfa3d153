"""A track with a non-finite velocity or position at one step: Eq. 1 is causal, so the outputs before that
step are those of the track without it, bit for bit, and none after it is finite; other tracks keep theirs."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("step", [0, 1, 7, 8, 20, 39])
def test_outputs_before_the_step_stay(value, step):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=12, radius=8e-6)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    t = W.configs.mip_tracks(w.grid, 6, 40, np.random.default_rng(1))
    t.vx[:] += 1.0                                           # no resting step
    clean = s.eq1_direct(device_tracks(t, torch)).cpu().numpy()
    t.vz[2, step] = value
    t.x[4, step] = value
    got = s.eq1_direct(device_tracks(t, torch)).cpu().numpy()
    s.close()
    for k in range(6):
        n = step if k in (2, 4) else clean.shape[1]
        assert np.array_equal(got[k, :n], clean[k, :n])
        assert not np.isfinite(got[k, n:]).any()
