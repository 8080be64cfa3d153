"""The form that an FP64 field takes (one transform per sample, or products with the lateral tables) depends on
the call and not on what the sensor computed before: a few samples give the same bits on a fresh sensor and on
one that holds the tables; and both forms agree for every count that the combination takes by 4, 8, 12 or 16."""
import pytest

import workloads as W
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu


def _sensor(P, w):
    s = P.Sensor(w.grid, w.columns)
    s.fit()
    return s


@pytest.mark.parametrize("n_t", [4, 13, 18, 23, 30])
def test_forms_agree_and_do_not_depend_on_the_past(n_t):
    import torch
    import paper_2605_13987_gb300 as P
    w = W.tiny_cell(nx=16, nz=32, n_t=n_t, radius=0.5 * 55e-6 / 16)
    s, fresh = _sensor(P, w), _sensor(P, w)
    s.relax(w.times)
    many = s.extend("fp64")
    for t in (0, n_t // 2, n_t - 1):
        s.relax(w.times[t:t + 1])
        fresh.relax(w.times[t:t + 1])
        a, b = s.extend("fp64"), fresh.extend("fp64")
        torch.cuda.synchronize()
        assert torch.equal(a, b)
        # the charges of both relaxations agree to the FP64 path's bound
        assert rel_l2(many[t].cpu().numpy(), b[0].cpu().numpy()) < 1e-10
    s.close()
    fresh.close()
