"""Blocks whose symmetry lets the reduced solve end in one iteration, after which residual and sums are rounding: rings
without disorder started from the Neel determinant, whose first block (it and its neighbours, all equivalent) is solved
exactly by one step.  Energies against the oracle's dense solve (1e-11 relative, as in the other Algorithm 2 tests)."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("sites", [6, 8, 10, 12])
@pytest.mark.parametrize("U", [2.0, 4.0, 8.0])
@pytest.mark.parametrize("m", [64, 160, 256, 300])
def test_first_block_of_a_ring(sites, U, m):
    h, g = inputs.hubbard_integrals((sites,), 1.0, U, True)
    ref = inputs.neel_reference((sites,), sites // 2, sites // 2)
    s = api.Solver(h, g, sites, sites // 2, sites // 2, ref_alpha=int(ref[0]), ref_beta=int(ref[1]), num_coordinates=m,
                   log2_capacity=20)
    o = oracle.CDFCI(sites, sites // 2, sites // 2, h, g, (int(ref[0]), int(ref[1])), 0.0, m)
    try:
        st = s.step(1)
        o.step(1)
        assert abs(st["energy"] - o.energy()) <= 1e-11 * abs(o.energy())
        st = s.step(30)                                 # and on: finite and falling
        assert np.isfinite(st["energy"]) and st["energy"] < o.energy()
    finally:
        s.close()
        o.close()
