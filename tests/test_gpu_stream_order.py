"""An extension on a caller's stream is asynchronous and goes on using the sensor's buffers; the calls made
after it, on the sensor's own stream or on another, wait for it there: every result as with a wait between."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=64, nz=96, n_t=128, m_req=32, radius=2.5 * 55e-6 / 64)
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(w.times)
    s.extend("fp32")                                   # launch shapes chosen
    torch.cuda.synchronize()
    tr = device_tracks(W.configs.mip_tracks(w.grid, 8, 20, np.random.default_rng(4)), torch)
    yield torch, P, w, s, tr
    s.close()


def _calls(s, w, tr):
    other = w.times[: len(w.times) // 2] * 1.7

    def relaxed():
        s.relax(other)
        q = s.charges()
        s.relax(w.times)
        return q

    xyz = np.array([[1e-6, 2e-6, 3e-6], [20e-6, 9e-6, 60e-6]])
    return {"currents": lambda: s.tangents(tr)[0], "loss32": lambda: s.loss(tr, "fp32"),
            "loss64": lambda: s.loss(tr, "fp64"), "points": lambda: s.sample_H(xyz, w.times[5:7]),
            "static": lambda: s.static_field([1.0, 0.0], "fp64"), "direct": lambda: s.eq1_direct(tr),
            "relax": relaxed}


def _same(torch, a, b):
    if isinstance(a, tuple):
        return all(_same(torch, x, y) for x, y in zip(a, b))
    if hasattr(a, "is_cuda"):
        return torch.equal(a, b)
    return np.array_equal(np.asarray(a), np.asarray(b))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", ["currents", "loss32", "loss64", "points", "static", "direct", "relax"])
def test_calls_after_an_extension_wait_for_it(env, precision, name):
    torch, P, w, s, tr = env
    s.relax(w.times)
    want_H = s.extend(precision)
    torch.cuda.synchronize()
    want = _calls(s, w, tr)[name]()
    torch.cuda.synchronize()
    s.relax(w.times)
    H = torch.empty_like(want_H)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(20_000_000)                  # the extension starts some 10 ms after the call returns
        s.extend(precision, out=H, stream=st)
    got = _calls(s, w, tr)[name]()
    torch.cuda.synchronize()
    assert torch.equal(H, want_H)
    assert _same(torch, got, want)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_extensions_on_two_streams(env, precision):
    torch, P, w, s, tr = env
    want = s.extend(precision)
    torch.cuda.synchronize()
    a, b = torch.empty_like(want), torch.empty_like(want)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(20_000_000)
        s.extend(precision, out=a, stream=s1)
    s.extend(precision, out=b, stream=s2)
    both = [torch.empty_like(want)]
    with torch.cuda.stream(s1):
        P.extend_batch([s], precision, both, s1)
    torch.cuda.synchronize()
    assert torch.equal(a, want) and torch.equal(b, want) and torch.equal(both[0], want)
