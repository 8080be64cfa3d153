"""Edges of kernels that change form with the size: many tangent directions (features), more points
than one chunk (point evaluation), more time samples than one pass of threads (modal tangents)."""
import numpy as np
import pytest

import workloads as W
from oracle import adjoint as A
from tests.gpu_common import device_tracks, rel_l2
from workloads.configs import UM

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2605_13987_gb300 as P
    assert torch.cuda.is_available()
    w = W.tiny_cell(nx=16, nz=32, n_t=12, radius=8 * UM)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    yield torch, P, w, s
    s.close()


@pytest.mark.parametrize("n_dir", [1, 8, 9, 17])
def test_features_take_any_number_of_directions(env, n_dir):
    torch, P, w, s = env
    g = torch.Generator(device="cuda").manual_seed(n_dir)
    x = torch.randn(7, 61, generator=g, device="cuda").cumsum(1).contiguous()
    dx = torch.randn(n_dir, 7, 61, generator=g, device="cuda")
    f, df = s.features(x, 1e-11, dx=dx)
    for d in range(n_dir):
        f1, df1 = s.features(x, 1e-11, dx=dx[d:d + 1].contiguous())
        assert torch.equal(f, f1)
        assert torch.equal(df[d], df1[0])


def test_points_of_several_chunks(env):
    torch, P, w, s = env
    rng = np.random.default_rng(3)
    xyz = rng.uniform(0, 1, (1030, 3)) * [w.grid.Lx, w.grid.Ly, w.grid.Lz]
    t = np.array([2e-12, 3e-10, 5e-9])
    whole = s.sample_H(xyz, t)
    for a, b in ((0, 5), (510, 516), (1020, 1030)):
        part = s.sample_H(xyz[a:b], t)
        # the same sums, scaled by other row norms before they are rounded
        assert rel_l2(whole[:, a:b], part) < 1e-13


@pytest.mark.parametrize("n_t", [12, 300])
def test_gradient_with_many_time_samples(env, n_t):
    torch, P, _, _ = env
    w = W.tiny_cell(nx=16, nz=32, n_t=n_t, radius=8 * UM)
    tr = W.configs.mip_tracks(w.grid, 3, 12, np.random.default_rng(4))
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    try:
        _, g = s.loss_grad(device_tracks(tr, torch))
    finally:
        s.close()
    fd = np.asarray(A.fd_grad(w, tr, rel_step=1e-4))
    r = w.columns[0].radius * np.array([0, 0, 1, 0]) + np.array([1, 1, 0, 1])
    scale = np.max(np.abs(fd * r))
    assert np.max(np.abs(g - fd) * r) < 1e-4 * scale        # the bound of the derivative's other tests
