"""OptOrbFCI at basis sizes around the line between one CTA and a cluster in the descent step (M N^2 = 4096), with one
orbital, and with odd shapes, against the oracle's outer loop.  The tolerances are those of the inner solution: it
stops at |c| errors of 1e-7 or less, which enter E squared and the RDMs, hence U, once."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("M,N,na,nb", [(3, 1, 1, 0), (7, 5, 2, 1), (16, 16, 1, 1), (17, 15, 1, 1), (17, 16, 1, 1),
                                       (20, 17, 2, 0)])
def test_descent_matches_the_oracle(M, N, na, nb):
    h, g = inputs.synthetic_integrals(M, np.random.Generator(np.random.PCG64(11 * M + N)))
    E_o, U_o = oracle.optorb_run(h, g, M, N, na, nb, outer=2, bb_steps=3)
    U, E = api.cdfci_optorb(h, g, M, N, na, nb, outer=2, bb_steps=3, inner_iterations=20000, log2_capacity=12)
    assert np.abs(E - E_o).max() < 1e-8, (E, E_o)
    assert np.abs(U.T @ U - np.eye(N)).max() < 1e-13
    assert np.abs(U - U_o).max() < 1e-6
