"""Step graphs (long and short, kernels chained) against single launches: the same bits for runs
that mix both graphs and single steps, start at an odd step, or follow a change of the settings."""
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


def _lattice(q, shape, storage, pattern, walls, stream=None):
    nz, ny, nx = shape
    lat = hb.Lattice(q, nx, ny, nz, storage=storage, pattern=pattern, stream=stream)
    lat.set_relaxation(0.7)
    lat.set_force(1e-4)
    if walls:
        lat.set_boundary(1, hb.HLBM_HALFWAY_BOUNCE_BACK)
    lat.set_porosity(inputs.random_porosity(shape, seed=4, lo=0.2).astype(np.float32))
    lat.set_populations(inputs.random_populations(q, shape, seed=3, amplitude=0.02))
    return lat


CASES = [(19, (20, 21, 22)), (19, (32, 32, 32)), (19, (21, 24, 50)), (9, (1, 130, 140)), (9, (1, 131, 333))]
KINDS = [(hb.HLBM_F32, hb.HLBM_TWO_LATTICE), (hb.HLBM_F16DEV, hb.HLBM_TWO_LATTICE), (hb.HLBM_BF16DEV, hb.HLBM_TWO_LATTICE),
         (hb.HLBM_F64, hb.HLBM_TWO_LATTICE), (hb.HLBM_F32, hb.HLBM_AA)]


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("storage,pattern", KINDS)
@pytest.mark.parametrize("q,shape", CASES)
def test_same_bits_as_single_launches(q, shape, storage, pattern, walls):
    a, b = (_lattice(q, shape, storage, pattern, walls) for _ in range(2))
    for call, n in enumerate((160, 8, 31, 45, 100)):
        if call == 2:
            for lat in (a, b):
                lat.set_relaxation(0.8)
        a.step(n)
        for _ in range(n):
            b.step(1)
        np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()


def test_graph_waits_for_the_work_before_it():
    """A replay right behind the write of a new state, a copy or another replay starts from that state."""
    import torch
    shape = (48, 52, 56)
    a, b = (_lattice(19, shape, hb.HLBM_F32, hb.HLBM_TWO_LATTICE, False) for _ in range(2))
    for seed in range(8):
        f = torch.from_numpy(inputs.random_populations(19, shape, seed=seed, amplitude=0.02)).cuda()
        for lat in (a, b):
            hb.hlbm_set_populations(lat.h, f)
        a.step(16)
        a.step(24)
        for _ in range(40):
            b.step(1)
        np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()
