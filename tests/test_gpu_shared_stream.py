"""Gradients while another host thread, with a lattice of its own, steps (graphs), copies and reduces
on the same stream: both threads get what they get alone."""
import threading

import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (36, 34, 40)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


def _lattice(stream, seed, storage=hb.HLBM_F32, pattern=hb.HLBM_TWO_LATTICE):
    nz, ny, nx = SHAPE
    lat = hb.Lattice(19, nx, ny, nz, storage=storage, pattern=pattern, stream=stream)
    lat.set_relaxation(0.7)
    lat.set_force(1e-4)
    lat.set_porosity(inputs.random_porosity(SHAPE, seed=seed, lo=0.2).astype(np.float32))
    return lat


def _gradients(stream, n, pattern):
    lat = _lattice(stream, 31, pattern=pattern)
    out = [lat.adjoint_flux_grad(20, 6) for _ in range(n)]
    state = lat.get_populations()
    lat.close()
    return out, state


def _steps(stream, n):
    lat = _lattice(stream, 32)
    vp = inputs.random_porosity(SHAPE, seed=33, lo=0.2).astype(np.float32)
    out = []
    for _ in range(n):
        lat.step(27)
        lat.set_porosity(vp)
        out.append(lat.reduce())
    state = lat.get_populations()
    lat.close()
    return out, state


@pytest.mark.parametrize("pattern", [hb.HLBM_TWO_LATTICE, hb.HLBM_AA])
@pytest.mark.parametrize("default_stream", [False, True])
def test_two_threads_on_one_stream(default_stream, pattern):
    import torch
    torch_stream = torch.cuda.Stream()
    stream = 0 if default_stream else torch_stream.cuda_stream
    n = 12
    want_grad, want_steps = _gradients(stream, n, pattern), _steps(stream, 4 * n)
    got, failed = {}, []

    def run(key, fn, *args):
        try:
            got[key] = fn(*args)
        except BaseException as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=run, args=("grad", _gradients, stream, n, pattern)),
               threading.Thread(target=run, args=("steps", _steps, stream, 4 * n))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]
    for (ja, ga), (jb, gb) in zip(want_grad[0], got["grad"][0]):
        assert ja == jb
        np.testing.assert_array_equal(ga, gb)
    np.testing.assert_array_equal(want_grad[1], got["grad"][1])
    assert want_steps[0] == got["steps"][0]
    np.testing.assert_array_equal(want_steps[1], got["steps"][1])
