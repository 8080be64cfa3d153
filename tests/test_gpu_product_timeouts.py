"""A wait that runs out in any of the tensor-core products of a call is reported by that call (by wt_sync for an
asynchronous extension): each product of a fit, a relaxation, a point evaluation and a derivative in turn.
The call works again afterwards, and no earlier error is reported twice."""
import os
from contextlib import contextmanager

import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks, rel_l2

pytestmark = pytest.mark.gpu


@contextmanager
def fault(at):
    os.environ["WT_FAULT"], os.environ["WT_FAULT_AT"] = "product_timeout", str(at)
    try:
        yield
    finally:
        os.environ.pop("WT_FAULT", None)
        os.environ.pop("WT_FAULT_AT", None)


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=8, nz=160, n_t=140, m_req=150, thick=300e-6, radius=3e-6)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    yield torch, P, w, s
    s.close()


def _every_product(P, call):
    """How many products the call has: the n-th fails for n = 1, 2, ... until there is none."""
    for n in range(1, 400):
        try:
            with fault(n):
                call()
        except P.WTError as e:
            assert "WT_ERR_TIMEOUT" in str(e), (n, str(e))
            continue
        return n - 1
    raise AssertionError("no end")


def test_fit(env):
    torch, P, w, s = env

    def call():
        x = P.Sensor(w.grid, w.columns)
        try:
            x.fit()
        finally:
            x.close()
    assert _every_product(P, call) >= 5


def test_relax(env):
    torch, P, w, s = env
    want = s.charges()
    assert _every_product(P, lambda: s.relax(w.times)) >= 5
    s.relax(w.times)
    assert rel_l2(s.charges(), want) < 1e-10
    s.sync()


def test_points(env):
    torch, P, w, s = env
    s.relax(w.times)
    xyz = np.random.default_rng(1).uniform(0, 1, (700, 3)) * [w.grid.Lx, w.grid.Ly, w.grid.Lz]
    want = s.sample_H(xyz, w.times[60:70])
    assert _every_product(P, lambda: s.sample_H(xyz, w.times[60:70])) >= 4
    assert np.array_equal(s.sample_H(xyz, w.times[60:70]), want)
    s.sync()


def test_derivative(env):
    torch, P, w, s = env
    s.relax(w.times)
    tr = device_tracks(W.configs.mip_tracks(w.grid, 3, 12, np.random.default_rng(4)), torch)
    i, di, loss, g = s.tangents(tr)
    assert _every_product(P, lambda: s.tangents(tr)) >= 10
    i2, _, _, g2 = s.tangents(tr)
    assert torch.equal(i, i2) and rel_l2(g2, g) < 1e-6
    assert s.loss(tr, "fp32") == pytest.approx(loss, rel=1e-6)


def test_field(env):
    torch, P, w, s = env
    s.relax(w.times)
    H = s.extend("fp64")
    s.sync()
    with fault(2):
        s.extend("fp64")
        with pytest.raises(P.WTError, match="WT_ERR_TIMEOUT"):
            s.sync()
    H2 = s.extend("fp64")
    s.sync()
    assert torch.equal(H, H2)
