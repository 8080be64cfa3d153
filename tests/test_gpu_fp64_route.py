"""The two forms of an FP64 field (one transform per sample, or products with the lateral tables) agree, on a
fresh sensor and on one that holds the tables from an earlier call, for the counts of samples that the
combination takes by 4, 8, 12 or 16 with some of a pass left empty."""
import pytest

import workloads as W
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu


def _sensor(P, w):
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    return s


@pytest.mark.parametrize("nx,nz,n_t", [(16, 32, 33), (16, 32, 34), (16, 32, 47), (32, 64, 13), (32, 64, 18), (32, 64, 23)])
def test_forms_agree(nx, nz, n_t):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=nx, nz=nz, n_t=n_t, m_req=16, radius=0.5 * 55e-6 / nx)
    s, fresh = _sensor(P, w), _sensor(P, w)
    s.relax(w.times)
    many = s.extend("fp64")                               # builds the tables
    for t in (0, n_t // 2, n_t - 1):
        for k in (1, 3, 7):
            few = w.times[max(0, min(t, n_t - k)):][:k]
            s.relax(few)
            fresh.relax(few)
            a, b = s.extend("fp64"), fresh.extend("fp64")
            torch.cuda.synchronize()
            # the charges of the relaxations agree to the FP64 path's bound
            assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) < 1e-10
            at = max(0, min(t, n_t - k))
            assert rel_l2(many[at:at + k].cpu().numpy(), b.cpu().numpy()) < 1e-10
    s.close()
    fresh.close()
