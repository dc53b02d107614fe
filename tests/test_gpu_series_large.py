"""hlbm_reduce_series on lattices whose steps go two per launch: the records and the state of
separate calls, in no more time than they take."""
import time

import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


def _lattice(n=160):
    lat = hb.Lattice(19, n, n, n)
    lat.set_relaxation(0.7)
    lat.set_force(1e-4)
    lat.set_porosity(inputs.regular_sphere_field(n, period=32, radius_ratio=0.3))
    return lat


@pytest.mark.parametrize("every", [3, 4, 5])
def test_series_equals_separate_calls(every):
    import torch
    a, b = _lattice(), _lattice()
    got = torch.empty((40, 8), dtype=torch.float64, device="cuda")
    want = torch.empty_like(got)
    times = []
    for _ in range(5):
        torch.cuda.synchronize()
        t = [time.perf_counter()]
        a.reduce_series(40, every, got)
        torch.cuda.synchronize()
        t.append(time.perf_counter())
        for k in range(40):
            if k:
                b.step(every)
            b.reduce_series(1, 1, want[k])
        torch.cuda.synchronize()
        t.append(time.perf_counter())
        assert torch.equal(got, want)
        times.append((t[1] - t[0], t[2] - t[1]))
    assert a.steps_taken == b.steps_taken
    np.testing.assert_array_equal(a.moments()[1], b.moments()[1])
    series, separate = (min(t[k] for t in times) for k in (0, 1))
    assert series <= 1.02 * separate  # two such timings are 0.2 % apart
    a.close()
    b.close()
