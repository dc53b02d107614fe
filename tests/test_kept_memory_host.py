"""The memory kept between objects (csrc/mem.cu) on the CPU, against fake CUDA calls that know the
contexts, the allocations and the frees (tests/host/kept_memory.cpp)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_14746_gb300", "csrc")


def _cuda_include():
    from paper_2310_14746_gb300 import build
    home = os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda"
    return os.path.join(home, "include")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("kept") / "kept_memory")
    cmd = ["g++", "-std=c++20", "-O1", "-I" + CSRC, "-I" + _cuda_include(), "-o", out,
           "-x", "c++", os.path.join(CSRC, "mem.cu"), os.path.join(ROOT, "tests", "host", "kept_memory.cpp"), "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.mark.parametrize("case", ["no_context_ids", "several_contexts", "no_host_memory", "context_facts"])
def test_kept_memory(program, case):
    r = subprocess.run([program, case], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
