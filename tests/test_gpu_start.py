"""A start vector's entries as the forced steps of the running m = 1 loop, the list cut into launches in several ways
(the loop's arithmetic does not depend on it: bit for bit), for one CTA, a cluster and a cooperative grid."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _start(w, n):
    o = oracle.CDFCI(w.N, 4, 3, w.h, w.g)
    o.step(3 * n)
    keys, c, _ = o.export()
    o.close()
    top = np.argsort(-np.abs(c), kind="stable")[:n]
    return keys[top], c[top]


def _sorted(s):
    keys, c, b = s.export()
    o = np.lexsort((keys[:, 1], keys[:, 0]))
    return keys[o], c[o], b[o]


@pytest.mark.parametrize("grid_blocks", [1, 5, 24])
@pytest.mark.parametrize("n", [1, 2, 17])
def test_a_start_vector_does_not_depend_on_how_it_is_cut(grid_blocks, n):
    w = inputs.ab_initio(10, 4, 3, seed=9)
    keys, c = _start(w, n)
    want = None
    for chunk in (1, 2, 16, 17, 0):
        s = api.Solver(w.h, w.g, w.N, 4, 3, log2_capacity=16, grid_blocks=grid_blocks, graph_chunk=chunk)
        try:
            s.set_initial(keys, c)
            first = _sorted(s)
            st = s.step(20)
            got = first + _sorted(s) + (np.array([st["energy"], st["mu"], st["elements"], st["iterations"]]),)
        finally:
            s.close()
        if want is None:
            want = got
            assert np.count_nonzero(first[1]) == n and st["iterations"] == 20
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
