"""Two-pass z transforms of the lengths beside powers of two and their small multiples, against the FP64
path of the same context, at every line count per block; 144 and 400 lines leave a part of the last
block empty."""
import pytest

import workloads as W
from tests.gpu_common import rel_l2
from workloads.configs import UM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz", [(8, 40), (12, 48), (8, 56), (12, 72), (20, 80), (12, 112), (20, 120), (12, 144),
                                   (8, 160), (12, 192), (20, 240)])
def test_two_pass_lengths_match_fp64(monkeypatch, nx, nz):
    import paper_2605_13987_gb300 as P
    P.load_library()
    w = W.tiny_cell(nx=nx, nz=nz, n_t=9, radius=0.7 * 55 * UM / nx)
    lanes = next(r for r in (32, 16, 8, 4) if nz % r == 0 and nz // r in (1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 15))
    xy = next(r for r in (8, 4) if nx % r == 0)
    s = P.Sensor(w.grid, w.columns)
    try:
        s.fit()
        s.relax(w.times)
        H64 = s.extend("fp64").cpu().numpy()
    finally:
        s.close()
    for lb in (16, 32, 64):
        monkeypatch.setenv("WT_LAUNCH_SHAPES", f"1,{lb},64,8,{nx // xy},{nz // lanes},0,1")
        s = P.Sensor(w.grid, w.columns)
        try:
            s.fit()
            s.relax(w.times)
            H32 = s.extend("fp32").double().cpu().numpy()
            assert s.tuning()["two_pass"] == 1
        finally:
            s.close()
        # FP32 transforms and sums of at most 240 terms, as for the other lengths
        assert rel_l2(H32, H64) < 1e-5, lb
