"""What the C ABI launches and captures (csrc/api.cu), on the CPU against fakes of the CUDA calls and of
the kernel launches (tests/host/step_calls.cpp)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2310_14746_gb300 import build
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda", "include")
    out = str(tmp_path_factory.mktemp("calls") / "step_calls")
    cmd = ["g++", "-std=c++20", "-O1", "-I" + build.CSRC, "-I" + include, "-o", out, "-x", "c++",
           os.path.join(build.CSRC, "api.cu"), os.path.join(ROOT, "tests", "host", "step_calls.cpp")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.mark.parametrize("case", ["captures", "gradient"])
def test_calls(program, case):
    r = subprocess.run([program, case], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
