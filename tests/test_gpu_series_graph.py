"""hlbm_reduce_series against single steps and records: the same values for series that are
replayed from a graph, too short for one, that end within a replay, start at an odd step or
after a change of the settings, for both streaming patterns and both outputs."""
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


def _lattice(pattern, storage):
    lat = hb.Lattice(19, 20, 18, 26, storage=storage, pattern=pattern)  # above the resident kernel's range
    lat.set_relaxation(0.7)
    lat.set_force(1e-4)
    lat.set_porosity(inputs.random_porosity((26, 18, 20), seed=8, lo=0.2).astype(np.float32))
    return lat


@pytest.mark.parametrize("pattern,storage", [(hb.HLBM_TWO_LATTICE, hb.HLBM_F32), (hb.HLBM_TWO_LATTICE, hb.HLBM_F16DEV),
                                             (hb.HLBM_AA, hb.HLBM_F32)])
@pytest.mark.parametrize("every", [1, 3])
def test_series_equals_single_records(pattern, storage, every):
    import torch
    a, b = _lattice(pattern, storage), _lattice(pattern, storage)
    for call, (nsamples, lead) in enumerate([(31, 0), (32, 1), (40, 0), (45, 1), (50, 2)]):
        for lat in (a, b):
            if lead:
                lat.step(lead)
            if call == 3:
                lat.set_relaxation(0.8)
        if call % 2:
            out = torch.empty((nsamples, 8), dtype=torch.float64, device="cuda")
            a.reduce_series(nsamples, every, out)
            got = out.cpu().numpy()
        else:
            got = np.asarray(a.reduce_series(nsamples, every))
        want = []
        for k in range(nsamples):
            if k:
                b.step(every)
            want.append(b.reduce_series(1)[0])
        np.testing.assert_array_equal(got, np.array(want))
        assert a.steps_taken == b.steps_taken
        np.testing.assert_array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()
