"""Which path hlbm_step takes: the tests that compare paths do compare them, and two steps per launch
give the bits of single steps in every form on shapes with remainders along each axis."""
import pytest

import paper_2310_14746_gb300 as hb
import test_gpu_resident as resident
import test_gpu_two_steps as two

pytestmark = pytest.mark.gpu

# (z, y, x): 24 x 9 tiles with a last tile of 4 columns or of one row, 32 x 7 tiles with one of 28
# columns and of one row, and a last block of fewer planes
ALL_FORMS = [(190, 162, 268), (222, 172, 116), (319, 309, 60), (219, 155, 260)]
FORMS = ["fx", "shift", "drag", "tensor"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("shape", ALL_FORMS)
def test_two_steps_in_every_form(shape, form):
    lat = two._lattice(shape, form, hb.HLBM_STEP_AUTO)
    assert [lat.steps_per_launch(n) for n in (0, 3, 4, 100)] == [1, 1, 2, 2]
    lat.close()
    two.test_same_bits_as_single_steps(shape, form)


def test_per_cell_and_unsuitable_lattices_take_single_steps():
    lat = two._lattice(ALL_FORMS[0], "fx", hb.HLBM_STEP_PER_CELL)
    assert lat.steps_per_launch(100) == 1
    lat.set_step_kernel(hb.HLBM_STEP_AUTO)
    assert lat.steps_per_launch(100) == 2
    lat.set_boundary(1, hb.HLBM_HALFWAY_BOUNCE_BACK)
    assert lat.steps_per_launch(100) == 1
    lat.close()
    for storage, pattern in ((hb.HLBM_F16DEV, hb.HLBM_TWO_LATTICE), (hb.HLBM_F32, hb.HLBM_AA), (hb.HLBM_F64, hb.HLBM_TWO_LATTICE)):
        lat = hb.Lattice(19, 128, 128, 128, storage=storage, pattern=pattern)
        assert lat.steps_per_launch(100) == 1
        lat.close()
    lat = hb.Lattice(19, 128, 128, 128)  # the gradient's test size
    lat.set_force(1e-4)
    assert lat.steps_per_launch(100) == 2
    lat.close()


@pytest.mark.parametrize("q,shape", resident.SHAPES)
def test_resident_path(q, shape):
    nz, ny, nx = shape
    fits = nx * ny * nz <= (16384 if q == 9 else 8192)
    for storage in resident.STORAGE:
        lat = hb.Lattice(q, nx, ny, nz, storage=storage)
        assert [lat.steps_per_launch(n) for n in (5, 7, 2003)] == ([1, 7, 1000] if fits else [1, 1, 1])
        lat.close()
    lat = hb.Lattice(q, nx, ny, nz, storage=hb.HLBM_F64)
    assert lat.steps_per_launch(100) == 1
    lat.close()
