"""xCDFCI with 4 to 8 states (the sums over a warp halve 4 values, or 8) and columns around a block of 128 elements,
against the oracle step by step: the same choices, energies within the rounding of the two summation orders."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import inputs
from gpu_util import require_gpu
from test_gpu_xcdfci import compare_rows, solver, start_keys

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("N,na,nb,k1,tau", [(7, 3, 1, 4, 0.0), (8, 3, 2, 5, 0.0), (8, 3, 2, 7, 1e-4), (9, 3, 2, 8, 0.0),
                                            (6, 2, 1, 6, 0.0)])
def test_trajectory_matches_oracle(N, na, nb, k1, tau):
    w = inputs.ab_initio(N, na, nb, seed=7)
    g = solver(w, k1, z_threshold=tau)
    o = oracle.XCDFCI(w.N, w.n_alpha, w.n_beta, w.h, w.g, start_keys(g, k1), tau=tau)
    try:
        for it in range(60):
            g.step(1)
            o.step(1)
            (kg,), _ = g.last_step()
            ko, _ = o.last_step()
            assert (int(kg[0]), int(kg[1])) == (int(ko[0]), int(ko[1])), it
            Eg, Eo = g.energies(), o.energies()
            assert np.abs(Eg - Eo).max() <= 1e-11 * np.abs(Eo).max(), (it, Eg, Eo)
        compare_rows(g, o)
    finally:
        g.close()
        o.close()
