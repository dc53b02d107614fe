"""Launch shapes on the CPU: blocks of the per-cell and paired kernels (tests/host/block_shapes.cpp) and
the plan of two steps per launch (tests/host/step2_plan.cpp)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("name", ["block_shapes", "step2_plan"])
def test_launch_shapes(tmp_path, name):
    from paper_2310_14746_gb300 import build
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda", "include")
    out = str(tmp_path / name)
    r = subprocess.run(["g++", "-std=c++20", "-O1", "-I" + build.CSRC, "-I" + include, "-o", out,
                        os.path.join(ROOT, "tests", "host", name + ".cpp")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([out], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
