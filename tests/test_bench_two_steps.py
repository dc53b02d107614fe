"""CPU checks of bench.py's bookkeeping where a launch advances two steps: the launches of a run, the
sources whose change makes the stored traffic stale, and the stored traffic against the bytes of one pass."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("per_launch,nsteps,launches", [(1, 100, 100), (2, 100, 50), (2, 4, 2), (2, 7, 5), (2, 102, 52), (1000, 2003, 3)])
def test_launches_of_a_run(per_launch, nsteps, launches):
    assert bench.step_launches(per_launch, nsteps) == launches


@pytest.mark.parametrize("nsteps,every,single,pairs", [(9, 4, 9 + 6, 2 + 2 + 1 + 6), (8, 4, 8 + 3, 2 + 4 + 3), (13, 5, 13 + 8, 3 + 3 + 3 + 8),
                                                       (7, 20, 7, 7), (2000, 45, 2000 + 44 * 44, 44 * 23 + 20 + 44 * 44)])
def test_launches_of_a_gradient(nsteps, every, single, pairs):
    assert bench.adjoint_forward_launches(nsteps, every, False) == single
    assert bench.adjoint_forward_launches(nsteps, every, True) == pairs


def test_two_step_sources_and_traffic(monkeypatch):
    kname = "stream_collide_d3q19_f32_two"
    assert {"k_step2.cu", "step2_plan.h", "k_step_pair.cuh", "lattice.cuh"} <= set(bench.TWO_STEP_SOURCES)
    now = bench.kernel_source_hash(kname, two_steps=True)
    assert now != bench.kernel_source_hash(kname)
    for n, e in bench.TWO_STEP_TRAFFIC_BYTES.items():
        # the state read and written once per launch, the porosity read once, and some halo rows twice
        assert 0.9 < e["bytes"] / (156 * n ** 3) < 1.1
    monkeypatch.setitem(bench.TWO_STEP_TRAFFIC_BYTES, 256, {"bytes": 5, "source_hash": now})
    assert bench.kernel_traffic(kname, 256, two_steps=True)[0] == 5
    monkeypatch.setitem(bench.TWO_STEP_TRAFFIC_BYTES, 256, {"bytes": 5, "source_hash": "0" * 16})
    assert bench.kernel_traffic(kname, 256, two_steps=True)[0] is None
    assert bench.kernel_traffic(kname, 64, two_steps=True) == (None, "not captured")
