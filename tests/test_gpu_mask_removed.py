"""Solid cells after the mask is removed, and in a checkpoint: at rest, whatever the lattice's memory
held before and however many steps ran, and the fluid's post-collision state is kept."""
import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs
from hlbm_testutil import make_lattice

pytestmark = pytest.mark.gpu
TAU, F = 0.7, (2e-4, -1e-4, 1e-4)
CASES = [(19, (26, 18, 20)), (19, (7, 9, 11)), (9, (1, 150, 140))]  # the first and last are not resident


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


def _spoil(q, shape, storage, pattern):
    """Leave memory behind that is not a state of any lattice."""
    lat = make_lattice(q, shape, storage, pattern)
    lat.set_populations(np.full((q,) + shape, 1e30 if storage != hb.HLBM_F16DEV else 15.0))
    lat.step(1)
    lat.close()


def _masked(q, shape, storage, pattern, steps):
    _spoil(q, shape, storage, pattern)
    rng = np.random.default_rng(91)
    solid = (rng.random(shape) < 0.25).astype(np.uint8)
    lat = make_lattice(q, shape, storage, pattern, TAU, F, (0, 1, 0), f0=inputs.random_populations(q, shape, seed=92),
                       varpi=inputs.random_porosity(shape, seed=93, lo=0.3))
    lat.set_solid_mask(solid)
    lat.step(steps)
    return lat, solid == 1


@pytest.mark.parametrize("storage", [hb.HLBM_F64, hb.HLBM_F32, hb.HLBM_F16DEV])
@pytest.mark.parametrize("pattern", [hb.HLBM_TWO_LATTICE, hb.HLBM_AA])
@pytest.mark.parametrize("q,shape", CASES)
@pytest.mark.parametrize("steps", [0, 3, 4, 7])
def test_removed_mask_leaves_cells_at_rest(q, shape, storage, pattern, steps):
    lat, solid = _masked(q, shape, storage, pattern, steps)
    f = lat.get_populations()
    lat.set_solid_mask(None)
    g = lat.get_populations()
    np.testing.assert_allclose(g, f, rtol=0, atol=2.3e-16)  # in place, two FP64 roundings of values below 1
    rest = make_lattice(q, shape, storage).get_populations()
    np.testing.assert_array_equal(g[:, solid], rest[:, solid])
    other = make_lattice(q, shape, storage, hb.HLBM_TWO_LATTICE, TAU, F, (0, 1, 0), f0=f,
                         varpi=inputs.random_porosity(shape, seed=93, lo=0.3))
    lat.step(5)
    other.step(5)
    # deviations below 0.5 and a few roundings in each of five steps
    atol = {hb.HLBM_F64: 1e-13, hb.HLBM_F32: 1e-6, hb.HLBM_F16DEV: 2e-3}[storage]
    np.testing.assert_allclose(lat.get_populations(), other.get_populations(), rtol=0, atol=atol)
    lat.close()
    other.close()


@pytest.mark.parametrize("pattern", [hb.HLBM_TWO_LATTICE, hb.HLBM_AA])
@pytest.mark.parametrize("steps", [3, 4])
def test_checkpoint_holds_solid_cells_at_rest(tmp_path, pattern, steps):
    q, shape = CASES[0]
    path = str(tmp_path / "a")
    lat, solid = _masked(q, shape, hb.HLBM_F32, pattern, steps)
    lat.save(path)
    f = lat.get_populations()
    lat.close()
    deviations = np.fromfile(path, np.float32)[-20 * solid.size:-solid.size].reshape((q,) + shape)  # then the porosity
    assert (deviations[:, solid] == 0).all()
    back = make_lattice(q, shape, hb.HLBM_F32, pattern)
    back.set_solid_mask(solid.astype(np.uint8))
    back.load(path)
    np.testing.assert_array_equal(back.get_populations(), f)
    back.step(3)
    back.set_solid_mask(None)
    rest = make_lattice(q, shape, hb.HLBM_F32).get_populations()
    np.testing.assert_array_equal(back.get_populations()[:, solid], rest[:, solid])
    back.close()
