"""Fit and relaxation at the sizes where the setup's kernels change form: the eigensolver's leaf (8
rows), its one-block and cooperative tridiagonalisation (96), the reflector blocks of its
back-transformation (128) and the batched merges (256); the factorisation's halves and blocks (64,
128).  The reduced pencil has 2 m - 1 rows, the normal matrix 2 m.  Against the oracle at the FP64
parity bound."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from tests.gpu_common import rel_l2

pytestmark = pytest.mark.gpu

TOL64 = 1e-10


@pytest.mark.parametrize("m", [4, 5, 32, 33, 48, 49, 64, 65, 96, 97, 128, 129, 150, 260])
def test_sizes_around_the_block_edges(m):
    import paper_2605_13987_gb300 as P
    nz = next(n for n in (8, 32, 36, 48, 49, 64, 70, 96, 98, 128, 140, 150, 270) if n >= m)
    w = W.tiny_cell(nx=8, nz=nz, n_t=24, m_req=m, thick=300e-6, radius=3e-6)
    assert w.columns[0].n_sources == m
    sol = O.solve(w)
    sen = P.Sensor(w.grid, w.columns)
    try:
        sen.fit()
        sen.relax(w.times)
        assert rel_l2(sen.capacitance(), sol.fit["Cn"]) < TOL64
        assert rel_l2(sen.modes(), np.sort(sol.rel["mu"])) < TOL64
        assert rel_l2(sen.charges(), sol.q.T) < TOL64
    finally:
        sen.close()
