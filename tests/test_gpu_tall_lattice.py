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


def test_requests_beyond_the_grids_are_refused():
    """What no launch grid covers is refused when submitted, and the server goes on; the largest
    axes that are covered run."""
    srv = Server(4 << 30, hb.HLBM_F32, 10)
    kw = dict(tau=0.7, F=(1e-4, 0, 0), tol=1e-30, max_steps=10)
    for shape, want_u in (((1, 131071, 65), False), ((1, 262141, 33), False), ((1, 524281, 1), False),
                          ((65536, 2, 2), False), ((300000, 1, 1), False), ((65536, 1, 1), True)):
        with pytest.raises(hb.HlbmError) as e:
            srv.submit(np.full(shape, 0.5, np.float32), want_u=want_u, **kw)
        assert e.value.status == hb.HLBM_ERR_INVALID_ARG
    taken = [srv.submit(np.full(shape, 0.5, np.float32), want_u=want_u, **kw)
             for shape, want_u in (((1, 131070, 65), True), ((1, 524280, 1), True), ((65535, 2, 2), True), ((65536, 1, 2), False))]
    done = srv.run_until_idle()
    srv.close()
    assert sorted(r["id"] for r in done) == sorted(taken)
    assert all(r["steps"] == 10 for r in done)
