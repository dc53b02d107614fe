"""Server requests with more rows than one launch grid has blocks along y: a lattice of ten equal
periods gives the velocity of one period, bit for bit."""
import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs
from paper_2310_14746_gb300.serving import Server

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_14746_gb300 import build
    build.build()


def _solve(vp, storage):
    srv = Server(4 << 30, storage, 10)
    srv.submit(vp, tau=0.7, F=(1e-4, 0, 0), tol=1e-30, max_steps=10, want_u=True)
    (r,) = srv.run_until_idle()
    srv.close()
    assert r["steps"] == 10
    return r["u"]


@pytest.mark.parametrize("storage", [hb.HLBM_F32, hb.HLBM_F16DEV, hb.HLBM_BF16DEV])
@pytest.mark.parametrize("nx,ny", [(96, 70000), (33, 131080), (32, 262200)])
def test_tall_request(nx, ny, storage):
    vp = inputs.random_porosity((1, ny // 10, nx), seed=21, lo=0.2).astype(np.float32)
    one = _solve(vp, storage)
    tall = _solve(np.ascontiguousarray(np.tile(vp, (1, 10, 1))), storage)
    np.testing.assert_array_equal(tall, np.tile(one, (1, 1, 10, 1)))
