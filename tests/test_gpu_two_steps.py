"""Two time steps per launch (FP32 lattices larger than L2) against single steps of the per-cell
kernel: the same bits for every collision form, at tile and plane remainders in each axis,
for run lengths that mix graphs, pairs and single steps; and a replayed capture of a call."""
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


def _lattice(shape, form, variant, stream=None):
    import torch
    nz, ny, nx = shape
    g = torch.Generator(device="cuda").manual_seed(nx + 1000 * ny)
    lat = hb.Lattice(19, nx, ny, nz, stream=stream)
    lat.set_step_kernel(variant)
    lat.set_relaxation(0.7)
    lat.set_force(*((1e-4, 0.0, 0.0) if form == "fx" else (1e-4, -2e-4, 3e-4)))
    if form == "drag":
        lat.set_homogenization(hb.HLBM_HOMOG_DRAG)
    lat.set_porosity(0.2 + 0.8 * torch.rand(shape, device="cuda", generator=g))
    if form == "tensor":
        lat.set_porosity_tensor(0.2 + 0.8 * torch.rand((3,) + shape, device="cuda", generator=g))
    lat.init_equilibrium(1.0, (1e-3, 2e-3, -1e-3))
    return lat


# tiles are 32 x 7 and 24 x 9: rows that end in a narrow tile, in a full one, in one of 4 cells; y and z remainders
@pytest.mark.parametrize("form", ["fx", "shift", "drag", "tensor"])
@pytest.mark.parametrize("shape", [(160, 150, 128), (208, 151, 172), (186, 133, 228), (171, 133, 160), (96, 168, 288),
                                   (159, 152, 132), (384, 384, 32), (64, 63, 1024), (186, 105, 292),
                                   (168, 154, 240), (148, 134, 144)])
def test_same_bits_as_single_steps(shape, form):
    import torch
    a, b = _lattice(shape, form, hb.HLBM_STEP_AUTO), _lattice(shape, form, hb.HLBM_STEP_PER_CELL)
    fa = torch.empty((19,) + shape, dtype=torch.float64, device="cuda")
    fb = torch.empty_like(fa)
    for n in (4, 3, 15, 6, 8):
        a.step(n)
        b.step(n)
        hb.hlbm_get_populations(a.h, fa)
        hb.hlbm_get_populations(b.h, fb)
        assert torch.equal(fa, fb), n
    a.close()
    b.close()


@pytest.mark.parametrize("steps", [2, 4, 6])
def test_captured_call_replays(steps):
    """A captured call of an even number of steps advances the state at each replay."""
    import torch
    shape = (160, 150, 128)
    stream = torch.cuda.Stream()
    a = _lattice(shape, "fx", hb.HLBM_STEP_AUTO, stream.cuda_stream)
    b = _lattice(shape, "fx", hb.HLBM_STEP_PER_CELL)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.step(steps)
    with torch.cuda.stream(stream):
        for _ in range(3):
            graph.replay()
    stream.synchronize()
    for _ in range(3 * steps):
        b.step(1)
    np.testing.assert_array_equal(a.moments()[1], b.moments()[1])
    a.close()
    b.close()
