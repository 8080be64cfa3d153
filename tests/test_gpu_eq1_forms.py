"""Eq. 1 on a stored field on both sides of the rules that choose between the one-kernel form, the staged one and
the staged one in the order of cells: equal bits to the allocation-free call, which has the one-kernel form."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,n_t", [(16, 32, 12), (16, 32, 70), (32, 64, 66)])
@pytest.mark.parametrize("n_tracks,n_steps", [(1, 14), (1, 15), (1, 84), (200, 60), (201, 60), (201, 350), (1600, 5),
                                              (2700, 32), (2800, 32), (2000, 400)])
def test_equal_bits(nx, nz, n_t, n_tracks, n_steps):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=nx, nz=nz, n_t=n_t, m_req=16, radius=2.5 * 55e-6 / nx)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    H = s.extend("fp32")
    t = W.configs.mip_tracks(w.grid, n_tracks, n_steps, np.random.default_rng(1))
    t.x[:] = np.random.default_rng(2).uniform(-0.5, 1.5, t.x.shape) * w.grid.Lx
    tr = device_tracks(t, torch)
    a = s.eq1(H, tr)
    b = torch.empty_like(a)
    P.wt_eq1_noalloc(s.ctx, H, tr, b)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    s.close()
