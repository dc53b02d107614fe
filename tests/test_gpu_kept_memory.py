"""Device memory kept between lattices: what a lattice computes does not depend on the
objects whose memory it inherits (other sizes, streams and threads, large lattices that are
not kept), what is kept is bounded, and release_scratch gives it back."""
import threading

import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(7, 9, 16), (40, 33, 24), (5, 6, 7)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


def _solve(shape, storage=hb.HLBM_F32, stream=None, solid=False):
    nz, ny, nx = shape
    lat = hb.Lattice(19, nx, ny, nz, storage=storage, stream=stream)
    lat.set_relaxation(0.7)
    lat.set_force(1e-4)
    lat.set_porosity(inputs.random_porosity(shape, seed=5, lo=0.2).astype(np.float32))
    if solid:
        lat.set_solid_mask(inputs.random_porosity(shape, seed=6) < 0.1)
        lat.set_solid_mask(None)
    lat.step(11)
    J, grad = lat.adjoint_flux_grad(9, 4)
    stats = lat.reduce()
    f = lat.get_populations()
    lat.close()
    return f, J, grad, stats


def _same(a, b):
    np.testing.assert_array_equal(a[0], b[0])
    assert a[1] == b[1] and a[3] == b[3]
    np.testing.assert_array_equal(a[2], b[2])


def test_results_do_not_depend_on_earlier_objects():
    import torch
    first = [_solve(s) for s in SHAPES]
    streams = [torch.cuda.Stream() for _ in range(2)]
    for k in range(6):
        for s, want in zip(SHAPES, first):
            _same(_solve(s, stream=streams[k % 2].cuda_stream, solid=k % 2 == 1), want)
    failed = []

    def work(seed):
        stream = torch.cuda.Stream()
        for k in range(6):
            j = (seed + k) % len(SHAPES)
            try:
                _same(_solve(SHAPES[j], stream=stream.cuda_stream), first[j])
            except BaseException as e:  # noqa: BLE001
                failed.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed[0]


def test_kept_memory_is_bounded_and_given_back():
    import torch
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    small = hb.Lattice(19, 16, 16, 16)
    small.release_scratch()
    before = free()
    for n in (96, 128, 192):  # 148 MiB (kept), 352 MiB (kept), 1.2 GiB (not from the pool)
        lats = [hb.Lattice(19, n, n, n) for _ in range(5)]
        for lat in lats:
            lat.close()
        assert before - free() <= (1536 + 64) << 20
    small.release_scratch()
    assert before - free() <= 64 << 20
    small.close()
