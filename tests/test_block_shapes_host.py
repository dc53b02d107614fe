"""Block shapes of the per-cell and paired kernels on the CPU (tests/host/block_shapes.cpp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_row_is_covered_by_one_grid(tmp_path):
    from paper_2310_14746_gb300 import build
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda", "include")
    out = str(tmp_path / "block_shapes")
    r = subprocess.run(["g++", "-std=c++20", "-O1", "-I" + build.CSRC, "-I" + include, "-o", out,
                        os.path.join(ROOT, "tests", "host", "block_shapes.cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([out], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
