"""Block shapes of the paired 16-bit kernels: rows of every kind of piece (whole rows, halves,
thirds, short pieces; pieces that end inside a row) against the per-cell kernel, same bits."""
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


@pytest.mark.parametrize("pattern,storage", [(hb.HLBM_TWO_LATTICE, hb.HLBM_F16DEV), (hb.HLBM_TWO_LATTICE, hb.HLBM_BF16DEV),
                                             (hb.HLBM_AA, hb.HLBM_F16DEV)])
@pytest.mark.parametrize("shape", [(21, 5, 96), (9, 13, 80), (7, 11, 204), (5, 9, 222), (25, 8, 42), (3, 7, 352), (2, 5, 1030)])
def test_block_shapes_give_the_per_cell_states(shape, pattern, storage):
    nz, ny, nx = shape
    f0 = inputs.random_populations(19, shape, seed=3, amplitude=0.05)
    vp = inputs.random_porosity(shape, seed=4, lo=0.2).astype(np.float32)
    out = []
    for variant in (hb.HLBM_STEP_AUTO, hb.HLBM_STEP_PER_CELL):
        lat = hb.Lattice(19, nx, ny, nz, storage=storage, pattern=pattern)
        lat.set_step_kernel(variant)
        lat.set_relaxation(0.7)
        lat.set_force(1e-4)
        lat.set_porosity(vp)
        lat.set_populations(f0)
        lat.step(11)
        out.append(lat.get_populations())
        lat.close()
    np.testing.assert_array_equal(out[0], out[1])
