"""Small lattices of different sizes stepped by several threads at once, each on its own
stream: the launches share kernels, and each gets the shared memory that its size needs."""
import threading

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


@pytest.mark.parametrize("q,shapes", [(19, [(4, 4, 4), (20, 20, 20), (9, 10, 11)]), (9, [(1, 8, 8), (1, 100, 120), (1, 30, 41)])])
def test_threads_with_different_sizes(q, shapes):
    import torch

    def lattice(shape, stream=None):
        nz, ny, nx = shape
        lat = hb.Lattice(q, nx, ny, nz, stream=stream)
        lat.set_relaxation(0.7)
        lat.set_force(1e-4)
        lat.set_porosity(inputs.random_porosity(shape, seed=5, lo=0.2).astype(np.float32))
        return lat

    def states(lat, calls):
        for _ in range(calls):
            lat.step(9)
        return lat.get_populations()

    calls, want = 400, []
    for s in shapes:
        lat = lattice(s)
        want.append(states(lat, calls))
        lat.close()
    failed, go = [], threading.Barrier(len(shapes))
    streams = [torch.cuda.Stream() for _ in shapes]
    lats = [lattice(s, streams[i].cuda_stream) for i, s in enumerate(shapes)]

    def work(i):
        try:
            go.wait(60)
            np.testing.assert_array_equal(states(lats[i], calls), want[i])
        except BaseException as e:  # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for lat in lats:
        lat.close()
    assert not failed, failed[0]
