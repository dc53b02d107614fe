"""The FP64 step on row lengths around its block widths (32, 16 and 8 cells), in the
shift form with the force along x and with a general force, against the FP64 oracle.
Tolerance: about 150 rounded operations per cell and step on populations of order 0.1
(1e-17 each) over 20 steps stay below 1e-13, the bound of the brute-force tests."""
import numpy as np
import pytest

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import inputs
from hlbm_testutil import make_lattice

pytestmark = pytest.mark.gpu

CASES = [(19, (2, 3, 7), (0, 0, 0)), (19, (2, 5, 8), (0, 1, 0)), (19, (3, 4, 9), (0, 0, 0)), (19, (2, 2, 17), (1, 0, 0)),
         (19, (1, 3, 33), (0, 0, 0)), (19, (3, 1, 32), (0, 0, 1)), (9, (1, 5, 31), (0, 1, 0)), (9, (1, 1, 24), (0, 0, 0))]


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("q,shape,bc", CASES)
def test_f64_step_row_lengths(q, shape, bc, general, oracle):
    f0 = inputs.random_populations(q, shape, seed=300 + sum(shape))
    vp = inputs.random_porosity(shape, seed=400 + sum(shape), lo=0.0, hi=1.0)
    F = (2e-4, -1e-4, 3e-4 if q == 19 else 0.0) if general else (2e-4, 0.0, 0.0)
    lat = make_lattice(q, shape, hb.HLBM_F64, hb.HLBM_TWO_LATTICE, 0.7, F, bc, varpi=vp, f0=f0)
    lat.step(20)
    got = lat.get_populations()
    lat.close()
    ref = oracle.run(f0, vp.astype(np.float64), 0.7, F, bc, 20)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-13)
