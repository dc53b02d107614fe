"""The resident small-lattice steps against the one-launch-per-step kernels: the same bits,
on lattices of one cell up to the largest that stays resident and one just above, for every
storage, collision form, walls and obstacles, over runs that take several resident launches."""
import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs
from hlbm_testutil import make_lattice

pytestmark = pytest.mark.gpu

SHAPES = [(19, (1, 1, 1)), (19, (1, 2, 3)), (19, (5, 7, 9)), (19, (16, 16, 32)), (19, (17, 16, 31)), (9, (1, 3, 5)),
          (9, (1, 32, 64)), (9, (1, 91, 90)), (9, (1, 128, 128)), (9, (1, 129, 128))]
STORAGE = [hb.HLBM_F32, hb.HLBM_F16DEV, hb.HLBM_BF16DEV]


def _run(q, shape, storage, form, bc, variant, steps, solid=None):
    vp = inputs.random_porosity(shape, seed=82, lo=0.2)
    F = (1e-4, 0.0, 0.0) if form == "shift_fx" else (1e-4, -2e-4, 3e-4 if q == 19 else 0.0)
    lat = make_lattice(q, shape, storage, hb.HLBM_TWO_LATTICE, 0.7, F, bc, varpi=vp,
                       f0=inputs.random_populations(q, shape, seed=81, amplitude=0.05))
    lat.set_step_kernel(variant)
    if form == "drag":
        lat.set_homogenization(hb.HLBM_HOMOG_DRAG)
    if form == "aniso":
        lat.set_porosity_tensor(np.stack([inputs.random_porosity(shape, seed=83 + a, lo=0.2) for a in range(3)]))
    if solid is not None:
        lat.set_solid_mask(solid)
    for n in steps:
        lat.step(n)
    out = lat.get_populations()
    taken = lat.steps_taken
    lat.close()
    return out, taken


@pytest.mark.parametrize("storage", STORAGE)
@pytest.mark.parametrize("form", ["shift_fx", "shift", "drag", "aniso"])
@pytest.mark.parametrize("q,shape", SHAPES)
def test_resident_bits(q, shape, form, storage):
    bc = (0, 1, 0) if form in ("shift", "drag") else (0, 0, 0)
    a, na = _run(q, shape, storage, form, bc, hb.HLBM_STEP_AUTO, (7, 1, 16))
    b, nb = _run(q, shape, storage, form, bc, hb.HLBM_STEP_PER_CELL, (7, 1, 16))
    assert na == nb == 24
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("q,shape,bc", [(19, (6, 9, 12), (0, 0, 0)), (9, (1, 40, 70), (1, 1, 0))])
def test_resident_obstacles_and_long_runs(q, shape, bc):
    solid = (np.random.default_rng(5).random(shape) < 0.2).astype(np.uint8)
    a, na = _run(q, shape, hb.HLBM_F32, "shift", bc, hb.HLBM_STEP_AUTO, (2003,), solid)
    b, nb = _run(q, shape, hb.HLBM_F32, "shift", bc, hb.HLBM_STEP_PER_CELL, (2003,), solid)
    assert na == nb == 2003
    np.testing.assert_array_equal(a, b)
