"""Resistivities for which the resistive pencil is not finite: the relaxation is refused with an error, whatever
the size of the divide-and-conquer tree, and the sensor goes on working with others."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho", [float("inf"), 1e-290, 1e-315])
@pytest.mark.parametrize("m", [4, 30, 150])
def test_relaxation_is_refused(m, rho):
    import dataclasses
    import paper_2605_13987_gb300 as P
    nz = {4: 8, 30: 32, 150: 160}[m]
    w = W.tiny_cell(nx=8, nz=nz, n_t=24, m_req=m, thick=300e-6, radius=3e-6)
    s = P.Sensor(w.grid, [dataclasses.replace(c, resistivity=rho) for c in w.columns])
    good = P.Sensor(w.grid, w.columns)
    good.fit()
    good.relax(w.times)
    s.fit()
    for _ in range(2):
        with pytest.raises(P.WTError):
            s.relax(w.times)
    for k, c in enumerate(w.columns):
        s.set_resistivity_profile(k, np.full(c.n_sources, c.resistivity))
    s.relax(w.times)
    assert rel_l2(s.charges(), good.charges()) < 1e-10
    s.close()
    good.close()
