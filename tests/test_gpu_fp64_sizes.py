"""FP64 fields whose rows (lateral points x time samples of a piece) pass the limits of a launch grid's
second dimension, whole and in several pieces with a short last one, alone, in a batch and under the loss,
against the per-sample transform; and products of as many rows, or of more terms than one pass over the
operands takes."""
import os
import subprocess

import numpy as np
import pytest

import workloads as W
from tests.gpu_common import device_tracks, rel_l2

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# nx, nz, time samples; rows of a piece: 294 912, 262 144, 352 256 (of 256 samples: 86, 86, 84)
SIZES = [(24, 24, 512), (32, 32, 256), (64, 32, 256)]
# both routes round at 1e-15 of the field; the charges of two relaxations differ by their conditioning,
# 1e-12 at the late samples taken here
TOL = 1e-11


def _cell(nx, nz, n_t):
    return W.tiny_cell(nx=nx, nz=nz, n_t=n_t, m_req=16, radius=0.5 * 55e-6 / nx)


def _relaxed(P, w, times):
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    s.relax(times)
    return s


@pytest.mark.parametrize("nx,nz,n_t", SIZES)
def test_field_of_many_rows(nx, nz, n_t):
    import torch
    import paper_2605_13987_gb300 as P
    w = _cell(nx, nz, n_t)
    s = _relaxed(P, w, w.times)
    H = s.extend("fp64")
    s.sync()
    for k in (n_t // 2, n_t - n_t // 6, n_t - 1):
        one = _relaxed(P, w, w.times[k:k + 1])              # few samples: one transform each
        ref = one.extend("fp64")
        torch.cuda.synchronize()
        assert rel_l2(H[k].cpu().numpy(), ref[0].cpu().numpy()) < TOL
        one.close()
    s.close()


def test_batch_and_loss_of_many_rows():
    import torch
    import paper_2605_13987_gb300 as P
    w = _cell(*SIZES[0])
    a, b = _relaxed(P, w, w.times), _relaxed(P, w, w.times)
    H = a.extend("fp64")
    a.sync()
    both = P.extend_batch([a, b], "fp64")
    torch.cuda.synchronize()
    assert torch.equal(both[0], H) and torch.equal(both[1], H)
    tr = device_tracks(W.configs.mip_tracks(w.grid, 5, 12, np.random.default_rng(4)), torch)
    L64, L32 = a.loss(tr, "fp64"), a.loss(tr, "fp32")
    assert abs(L64 - L32) < 1e-5 * L64                      # the FP32 path's bound
    a.close()
    b.close()


@pytest.mark.parametrize("case", ["0 0 262145 3 40 0 0 0", "1 1 600001 9 24 0 0 0", "0 1 300000 20 1025 0 0 0",
                                  "0 0 3 2 4300000 0 0 0", "1 1 2 3 4200001 0 0 0"])
def test_products_of_many_rows_or_terms(tmp_path, case):
    from paper_2605_13987_gb300 import build as b
    exe = str(tmp_path / "driver")
    objs = [os.path.join(b.BUILD, o + ".o") for o in ("k_dense", "k_dgemm_tc", "k_expand_tc")]
    subprocess.run([b.nvcc(), *b.ARCH, "-O2", "-std=c++17", os.path.join(ROOT, "tests", "dgemm_driver.cu"), *objs,
                    "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], input=case + "\n", capture_output=True, text=True, timeout=300, check=True).stdout
    worst, untouched, err = out.split()
    assert int(err) == 0 and int(untouched) == 1 and float(worst) <= 1.0, out      # the driver's own bound
