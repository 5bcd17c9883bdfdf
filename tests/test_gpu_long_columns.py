"""Columns of more elements than the m = 1 loop's threads take at once: several rounds of them, on a cluster and on a
cooperative grid, against the oracle's choice, step and energy."""
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("grid_blocks", [1, 16, 17, 40])   # 21.1 k elements; a round takes 1,056 a CTA
def test_rounds_match_the_oracle(grid_blocks):
    w = inputs.ab_initio(32, 5, 4, seed=6)
    s = api.Solver(w.h, w.g, w.N, 5, 4, log2_capacity=22, z_threshold=1e-5, grid_blocks=grid_blocks)
    o = oracle.CDFCI(w.N, 5, 4, w.h, w.g, (0, 0), 1e-5, 1)
    try:
        for it in range(40):
            st = s.step(1)
            o.step(1)
            (kg,), (eg,) = s.last_step()
            (ko,), (eo,) = o.last_step()
            assert tuple(kg) == tuple(ko), it
            assert abs(eg - eo) <= 1e-10 * max(1.0, abs(eo)), it
            assert abs(st["energy"] - o.energy()) <= 1e-11 * abs(o.energy()), it
        assert st["last_column"] > 21_000
        keys, c, _ = s.export()
        ref = o.export()
        got = {(int(a), int(b)): float(v) for (a, b), v in zip(keys, c)}
        assert all(abs(got[(int(a), int(b))] - v) <= 1e-10 for (a, b), v in zip(ref[0], ref[1]) if v)
    finally:
        s.close()
        o.close()
