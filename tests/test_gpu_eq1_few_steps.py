"""Eq. 1 on a stored field for tracks of 1 to 40 steps: the form that spreads a step's time samples over the lanes
(few values) and the staged one (the same tracks many times over) give equal bits, and the oracle's currents."""
import numpy as np
import pytest

import workloads as W
from oracle import eq1 as OE
from tests.gpu_common import device_tracks, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=50, radius=8e-6)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    H = s.extend("fp32")
    torch.cuda.synchronize()
    yield torch, P, w, s, H
    s.close()


@pytest.mark.parametrize("n_steps", [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 40])
def test_forms_agree(env, n_steps):
    torch, P, w, s, H = env
    t = W.configs.mip_tracks(w.grid, 3, n_steps, np.random.default_rng(n_steps))
    t.n_out = n_steps + 7
    few = device_tracks(t, torch)
    a = s.eq1(H, few)
    b = torch.empty_like(a)
    P.wt_eq1_noalloc(s.ctx, H, few, b)
    n = 1 + (1 << 20) // (3 * n_steps * 20)
    many = {k: (v.repeat(n, 1) if k in ("x", "y", "z", "vx", "vy", "vz") else v.repeat(n) if k == "q" else v) for k, v in few.items()}
    many["n_tracks"] = 3 * n
    c = s.eq1(H, many)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert torch.equal(c.reshape(n, 3, -1), a.expand(n, 3, a.shape[1]))
    ref = OE.currents(w.grid, w.times, H.double().cpu().numpy(), t, v_w=w.fit.v_w)
    assert rel_l2(a.cpu().numpy(), ref) < 1e-5               # the FP32 path's bound
