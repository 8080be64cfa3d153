"""Builds and runs a test driver (tests/<name>.cu) linked with objects of the library."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_driver(tmp_path, name, objects, text=""):
    from paper_2605_13987_gb300 import build as b
    exe = str(tmp_path / name)
    objs = [os.path.join(b.BUILD, o + ".o") for o in objects]
    subprocess.run([b.nvcc(), *b.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    os.path.join(ROOT, "tests", name + ".cu"), *objs, "-o", exe], check=True, capture_output=True)
    return subprocess.run([exe], input=text, capture_output=True, text=True, timeout=300, check=True).stdout
