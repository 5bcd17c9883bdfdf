"""A long start vector on several CTAs: every forced step reads its slot's c and b in every CTA while CTA 0 takes the step.
c, their number and mu = c.c depend on the given coefficients alone, so they are those of one CTA bit for bit, for a
cluster and a grid, with the list cut into launches or not, every time."""
import numpy as np
import pytest

from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _starts(grid_blocks, chunk, keys, c, times):
    s = api.Solver.hubbard_k((4, 4), 8, 8, U=4.0, log2_capacity=18, grid_blocks=grid_blocks, graph_chunk=chunk)
    try:
        for _ in range(times):
            s.set_initial(keys, c)
            k, x, _ = s.export()
            st = s.stats()
            on = x != 0.0
            yield {(int(a), int(b)): float(v) for (a, b), v in zip(k[on], x[on])}, st["mu"], st["nnz_c"], st["n_slots"]
    finally:
        s.close()


@pytest.fixture(scope="module")
def one_cta():
    keys = api.cdfci_degenerate_set(np.diag(inputs.hubbard_k_integrals((4, 4), 1.0, 4.0)[0]), 8, 8)
    rng = np.random.default_rng(3)
    keys = keys[rng.permutation(len(keys))]
    c = rng.uniform(1.0, 2.0, size=len(keys)) / len(keys)
    (want,) = _starts(1, 0, keys, c, 1)
    assert want[0] == {(int(a), int(b)): float(v) for (a, b), v in zip(keys, c)} and want[2] == len(keys) == 400
    return keys, c, want


@pytest.mark.parametrize("chunk", [0, 1, 7])
@pytest.mark.parametrize("grid_blocks", [2, 16, 23, 64])
def test_the_start_does_not_depend_on_the_ctas(one_cta, grid_blocks, chunk):
    keys, c, want = one_cta
    for got in _starts(grid_blocks, chunk, keys, c, 5):
        assert got == want
