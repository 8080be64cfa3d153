"""The tensor-core FP64 products (residue arithmetic) against long double sums: every operand
layout, edges of the 128 x 256 x 64 tiles and of the 1024-term accumulator chunks, the lower-only
form, one operand used twice, and rows of zeros, extreme scales, an infinity or a dominant entry.
The bound is derived in dgemm_driver.cu; 1 is the bound itself."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CASES = [(ta, tb, M, N, K, 0, 0, 0) for ta in (0, 1) for tb in (0, 1)
         for M, N, K in ((5, 3, 1), (64, 64, 64), (129, 257, 65), (127, 130, 1025))]
CASES += [(0, 1, 257, 257, 2049, 1, 1, 0), (1, 0, 300, 300, 700, 1, 1, 0), (1, 0, 128, 128, 128, 1, 1, 0),
          (0, 1, 400, 400, 130, 1, 0, 0), (0, 0, 1, 1000, 256, 0, 0, 0), (0, 0, 700, 1, 300, 0, 0, 0),
          (0, 0, 70, 90, 200, 0, 0, 1), (1, 1, 70, 90, 1500, 0, 0, 1), (0, 1, 33, 2100, 32, 0, 0, 0)]


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    from paper_2605_13987_gb300 import build as b
    exe = str(tmp_path_factory.mktemp("dgemm") / "driver")
    objs = [os.path.join(b.BUILD, o + ".o") for o in ("k_dense", "k_dgemm_tc", "k_expand_tc")]
    subprocess.run([b.nvcc(), *b.ARCH, "-O2", "-std=c++17", os.path.join(ROOT, "tests", "dgemm_driver.cu"), *objs,
                    "-o", exe], check=True, capture_output=True)
    text = "".join(" ".join(map(str, c)) + "\n" for c in CASES)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, timeout=300, check=True).stdout
    return out.split("\n")


@pytest.mark.parametrize("k", range(len(CASES)))
def test_products_within_the_rounding_bound(results, k):
    worst, untouched, err = results[k].split()
    assert int(err) == 0 and int(untouched) == 1, (CASES[k], results[k])
    assert float(worst) <= 1.0, (CASES[k], results[k])
