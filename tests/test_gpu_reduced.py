"""The reduced problem at the block sizes where its layout changes (threads a row 1, 2, 4, 8; one CTA or a cluster of
4; leading parts in registers or not), and the ordering of the chosen set there: three iterations against the oracle's
dense solve.

Tolerances as in the other Algorithm 2 tests: eta 1e-9 of its largest entry (the eigenvector's conditioning times the
1e-14 residual of both solvers), the energy, second order in that, 1e-11 relative."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("m", [2, 31, 39, 40, 79, 80, 127, 159, 160, 255, 319, 320])
def test_three_block_steps_match_the_oracle(m):
    w = inputs.ab_initio(10, 4, 3, seed=50)
    s = api.Solver(w.h, w.g, w.N, 4, 3, num_coordinates=m, log2_capacity=16)
    o = oracle.CDFCI(w.N, 4, 3, w.h, w.g, (0, 0), 0.0, m)
    try:
        for _ in range(3):
            st = s.step(1)
            o.step(1)
            keys, eta = s.last_step()
            okeys, oeta = o.last_step()
            assert abs(st["energy"] - o.energy()) <= 1e-11 * abs(o.energy())
            got = {tuple(k): x for k, x in zip(np.asarray(keys).tolist(), eta)}
            want = {tuple(k): x for k, x in zip(np.asarray(okeys).tolist(), oeta)}
            assert set(got) == set(want)
            top = max(abs(x) for x in want.values())
            assert max(abs(got[k] - want[k]) for k in want) <= 1e-9 * top
    finally:
        s.close()
        o.close()
