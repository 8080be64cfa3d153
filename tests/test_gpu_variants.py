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


@pytest.mark.parametrize("order", [0, 1, 2, 3, 4, 5, 20])
@pytest.mark.parametrize("n_tracks,n", [(3, 1), (3, 33), (2, 300), (6000, 33), (2100, 200), (9000, 64)])
def test_shaping_forms(env, order, n_tracks, n):
    """Tap by tap (few tracks) and by recursion (many), in place, and rows with an infinity or a NaN,
    which must reach as far as the taps do and no further."""
    from oracle import electronics as E
    torch, P, w, s = env
    dt, tau = 1e-11, 0.7e-11 if order < 3 else 2.3e-11
    rng = np.random.default_rng(order)
    i = rng.standard_normal((n_tracks, n)).astype(np.float32)
    x = torch.tensor(i, device="cuda")
    v = s.shape(x, dt, tau, order, gain=2.0)
    rows = np.unique(np.concatenate([[0, n_tracks - 1], rng.integers(0, n_tracks, 8)]))
    ref = E.shape(i[rows], dt, tau, order, gain=2.0)
    # FP32 rounding of the result: 2^-24 of each value
    got = v[torch.tensor(rows, device="cuda")].cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-7 * np.linalg.norm(ref)      # one sample of order > 0: zero
    bad = x.clone()
    bad[0, n // 2] = float("inf")
    bad[-1, 0] = float("nan")
    alone = s.shape(bad[[0, n_tracks - 1]].contiguous(), dt, tau, order, gain=2.0)
    many = s.shape(bad, dt, tau, order, gain=2.0)
    assert torch.equal(many[1:-1], v[1:-1])
    assert torch.allclose(many[[0, n_tracks - 1]], alone, rtol=1e-6, atol=0.0, equal_nan=True)
    y = bad.clone()
    s.shape(y, dt, tau, order, gain=2.0, out=y)
    assert torch.equal(torch.nan_to_num(y), torch.nan_to_num(many))


@pytest.mark.parametrize("n_tracks,n_steps", [(2000, 60), (700, 100), (1, 33)])
def test_eq1_on_the_field_staged_and_not(env, n_tracks, n_steps):
    """The staged form (large calls) and the one-kernel form (the allocation-free call) interpolate and
    sum in the same order: equal bits."""
    torch, P, w, s = env
    H = s.extend("fp32")
    tr = device_tracks(W.configs.mip_tracks(w.grid, n_tracks, n_steps, np.random.default_rng(1)), torch)
    a = s.eq1(H, tr)
    b = torch.empty_like(a)
    P.wt_eq1_noalloc(s.ctx, H, tr, b)
    torch.cuda.synchronize()
    assert torch.equal(a, b)


@pytest.mark.parametrize("nx,nz", [(16, 32), (20, 36), (36, 60)])
def test_fp64_field_from_tables_and_per_sample(env, nx, nz):
    """Few time samples take one spectral transform each, more the lateral tables and products."""
    torch, P, _, _ = env
    w = W.tiny_cell(nx=nx, nz=nz, n_t=12, radius=0.5 * 55e-6 / nx * (5 if nx > 20 else 1))
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    try:
        s.relax(w.times[:3])
        few = s.extend("fp64")
        s.relax(w.times)
        many = s.extend("fp64")
        torch.cuda.synchronize()
        for t in range(3):
            # the charges of both relaxations agree to the FP64 path's bound
            assert rel_l2(many[t].cpu().numpy(), few[t].cpu().numpy()) < 1e-10
    finally:
        s.close()


@pytest.mark.parametrize("n_tracks,n_steps", [(5000, 70), (20000, 16)])
def test_eq1_steps_in_cell_order(env, n_tracks, n_steps):
    """Enough steps to be taken in the order of their cells: random cells, resting steps, positions outside
    of the box and on its faces; equal bits to the one-kernel form, which keeps the tracks' order."""
    torch, P, w, s = env
    H = s.extend("fp32")
    t = W.configs.mip_tracks(w.grid, n_tracks, n_steps, np.random.default_rng(2))
    rng = np.random.default_rng(3)
    shape = t.x.shape
    t.x[:] = rng.uniform(-1.0, 2.0, shape) * w.grid.Lx
    t.y[:] = rng.uniform(-1.0, 2.0, shape) * w.grid.Ly
    t.z[:] = np.clip(rng.uniform(-0.2, 1.2, shape), 0.0, 1.0) * w.grid.Lz
    rest = rng.uniform(size=shape) < 0.2
    for v in (t.vx, t.vy, t.vz):
        v[rest] = 0.0
    tr = device_tracks(t, torch)
    a = s.eq1(H, tr)
    b = torch.empty_like(a)
    P.wt_eq1_noalloc(s.ctx, H, tr, b)
    torch.cuda.synchronize()
    assert torch.equal(a, b)


@pytest.mark.parametrize("n_steps,n_out", [(8, 16), (33, 40), (200, 400), (1030, 700), (2100, 750)])
def test_eq1_direct_leaves_out_resting_steps(env, n_steps, n_out):
    """Tracks that rest now and then, at any step, or always, or never, over one list of groups and over
    several: against the stored field's form, which takes every step.  Both sum FP32 products of the same
    FP32 basis fields: 1e-5 of the norm, as between the two forms elsewhere."""
    torch, P, w, s = env
    H = s.extend("fp32")
    t = W.configs.mip_tracks(w.grid, 40, n_steps, np.random.default_rng(4))
    rng = np.random.default_rng(5)
    t.n_out = n_out
    v = 1e5 * (1 + rng.uniform(size=t.x.shape))
    rest = np.repeat(rng.uniform(size=(40, (n_steps + 10) // 11)) < 0.6, 11, axis=1)[:, :n_steps]
    rest[0] = True
    rest[1] = False
    rest[2, 1:] = True
    t.x[:] = rng.uniform(0, 1, t.x.shape) * w.grid.Lx
    t.z[:] = rng.uniform(0, 1, t.x.shape) * w.grid.Lz
    t.vx[:] = np.where(rest, 0.0, v)
    t.vy[:] = np.where(rest, 0.0, -0.5 * v)
    t.vz[:] = 0.0
    tr = device_tracks(t, torch)
    a = s.eq1_direct(tr).cpu().numpy()
    b = s.eq1(H, tr).cpu().numpy()
    assert np.all(a[0] == 0.0)
    assert rel_l2(a, b) < 1e-5


@pytest.mark.parametrize("n_t", [13, 18, 23, 30])
def test_fp64_field_from_tables_by_any_count(env, n_t):
    """Counts of time samples that the combination takes by 4, 8, 12 or 16 with some of a pass left empty."""
    torch, P, _, _ = env
    w = W.tiny_cell(nx=16, nz=32, n_t=n_t, radius=0.5 * 55e-6 / 16)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    try:
        s.relax(w.times)
        many = s.extend("fp64")
        for t in (0, n_t // 2, n_t - 1):
            s.relax(w.times[t:t + 1])
            one = s.extend("fp64")
            torch.cuda.synchronize()
            # the charges of both relaxations agree to the FP64 path's bound
            assert rel_l2(many[t].cpu().numpy(), one[0].cpu().numpy()) < 1e-10
    finally:
        s.close()
