"""Start vectors whose consecutive entries are a double excitation apart that the m = 1 loop does not enumerate:
doubles of a real-space lattice (every double vanishes) and opposite-spin doubles that do not conserve momentum.
Without compression b = Hc for every stored determinant, after the start and after every step.

Tolerance: an entry of b is a sum of at most 17 + 30 products H_ji eta_i and its recalculation; 64 additions of rounding
2^-53 relative to the sum of the magnitudes, (|H| t)_j with t_i the sum of the steps |eta_i| of coordinate i (the start's
c_i among them)."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _check_b(s, w, H, t):
    keys, c, b = s.export()
    at = [oracle.fci_index(w.N, w.n_alpha, w.n_beta, k) for k in keys]
    x = np.zeros(len(H))
    x[at] = c
    assert (np.abs(b - (H @ x)[at]) <= 64 * 2.0 ** -53 * (np.abs(H) @ t)[at]).all()
    return x


@pytest.mark.parametrize("grid_blocks", [1, 5, 24])
@pytest.mark.parametrize("system", ["real", "momentum"])
@pytest.mark.parametrize("start", ["pair", "scrambled"])
def test_b_of_a_start_vector_is_hc(system, start, grid_blocks):
    rng = np.random.default_rng(11)
    shape, na, nb = (6,), 3, 2
    w = (inputs.hubbard if system == "real" else inputs.hubbard_k)(shape, na, nb, U=3.0)
    H = oracle.dense_H(w.N, na, nb, w.h, w.g)
    dets = oracle.fci_dets(w.N, na, nb)
    if start == "pair":                                   # alpha 2 -> 3 with beta 1 -> 5: momenta 1 and 4, sum 5
        keys = np.array([[0b000111, 0b000011], [0b001011, 0b100001]], dtype=np.uint64)
    else:
        keys = dets[rng.permutation(len(dets))[:17]]
    c = rng.uniform(0.2, 1.0, size=len(keys))
    c /= np.linalg.norm(c)
    given = np.zeros(len(dets))
    given[[oracle.fci_index(w.N, na, nb, k) for k in keys]] = c
    kw = dict(log2_capacity=12, grid_blocks=grid_blocks)
    s = api.Solver(w.h, w.g, w.N, na, nb, **kw) if system == "real" else api.Solver.hubbard_k(shape, na, nb, U=3.0, **kw)
    try:
        s.set_initial(keys, c)
        assert np.array_equal(_check_b(s, w, H, given), given)
        t = given.copy()
        for _ in range(30):
            s.step(1)
            (k,), (eta,) = s.last_step()
            t[oracle.fci_index(w.N, na, nb, k)] += abs(eta)
            _check_b(s, w, H, t)
    finally:
        s.close()
