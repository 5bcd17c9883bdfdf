"""The first blocks of a run, which hold every candidate and are shorter than m, against the oracle's dense solve
(eta 1e-9 of its largest entry, the energy 1e-11 relative: the tolerances of the other block tests)."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("shape,na,nb,m", [((6,), 3, 3, 80), ((6,), 3, 3, 128), ((10,), 3, 2, 83), ((2, 4), 3, 3, 196)])
def test_short_first_blocks_match_the_oracle(shape, na, nb, m):
    h, g = inputs.hubbard_integrals(shape, 1.0, 2.0, True)
    N = len(h)
    h = h + np.diag(np.random.default_rng(5).uniform(-0.5, 0.0, N))
    ref = inputs.neel_reference(shape, na, nb)
    s = api.Solver(h, g, N, na, nb, ref_alpha=ref[0], ref_beta=ref[1], num_coordinates=m, log2_capacity=14)
    o = oracle.CDFCI(N, na, nb, h, g, ref, 0.0, m)
    short = 0
    try:
        for _ in range(3):
            st = s.step(1)
            o.step(1)
            keys, eta = s.last_step()
            okeys, oeta = o.last_step()
            if len(okeys) == m:
                break
            short += 1
            assert abs(st["energy"] - o.energy()) <= 1e-11 * abs(o.energy())
            got = {tuple(k): x for k, x in zip(np.asarray(keys).tolist(), eta)}
            want = {tuple(k): x for k, x in zip(np.asarray(okeys).tolist(), oeta)}
            assert set(got) == set(want)
            top = max(abs(x) for x in want.values())
            assert max(abs(got[k] - want[k]) for k in want) <= 1e-9 * top
        assert short >= 1
    finally:
        s.close()
        o.close()
