"""Forward sweep of the gradient with two steps per launch where no state in between is kept, and
chained kernels: the gradient, the objective and the final state of single steps of the per-cell
kernel, same bits, for run lengths around the checkpoint interval; default and other streams."""
import numpy as np
import pytest

import paper_2310_14746_gb300 as hb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


def _gradient(shape, variant, storage, nsteps, every, stream):
    import torch
    nz, ny, nx = shape
    g = torch.Generator(device="cuda").manual_seed(11)
    varpi = 0.2 + 0.8 * torch.rand(shape, device="cuda", generator=g)
    grad = torch.empty(shape, dtype=torch.float32, device="cuda")
    f = torch.empty((19,) + shape, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    lat = hb.Lattice(19, nx, ny, nz, storage=storage, stream=stream)
    lat.set_step_kernel(variant)
    lat.set_relaxation(0.7)
    lat.set_force(1e-4)
    lat.set_porosity(varpi)
    J, _ = lat.adjoint_flux_grad(nsteps, every, None, grad)
    hb.hlbm_get_populations(lat.h, f)
    torch.cuda.synchronize()
    lat.close()
    return J, grad, f


@pytest.mark.parametrize("nsteps,every", [(1, 4), (8, 4), (9, 4), (11, 4), (13, 5), (12, 1), (14, 2), (7, 20)])
@pytest.mark.parametrize("shape,storage", [((128, 128, 128), hb.HLBM_F32), ((21, 23, 30), hb.HLBM_F32),
                                           ((21, 23, 30), hb.HLBM_F16DEV)])
def test_sweeps_equal_single_steps(shape, storage, nsteps, every):
    import torch
    own = torch.cuda.Stream()
    want = _gradient(shape, hb.HLBM_STEP_PER_CELL, storage, nsteps, every, None)
    for stream in (None, own.cuda_stream):
        got = _gradient(shape, hb.HLBM_STEP_AUTO, storage, nsteps, every, stream)
        assert got[0] == want[0]
        assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
