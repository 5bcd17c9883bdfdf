"""The pair sums over a stored vector (RDMs, exact Rayleigh quotient) at the sizes where their list and filters
change: a stated count below, at and far above the true one (the list redone; filter 1 sized for it; filter 1 left
out), one spin empty, a single determinant, orbitals in the upper half of the 64-bit words.

Tolerances: an entry is a sum of at most n_det terms c_I c_J / c.c whose absolute sum is at most n_e (n_e - 1) n_det
/ ... <= 1e3 here, so its rounding is below 1e3 x n_det x 2^-53 < 1e-10 of the largest entry in the worst case and
about the square root of that in practice; 1e-12 is the bound the other RDM tests use on sums as long."""
import numpy as np
import pytest

import oracle
from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def connected(N, na, nb, n, rng):
    """n distinct determinants reached from one another by single excitations."""
    A, B = (1 << na) - 1, ((1 << nb) - 1) << (N - nb)
    out = [(A, B)]
    for _ in range(200 * n):
        if len(out) == n:
            break
        A, B = out[rng.integers(len(out))]
        spin = 0 if nb == 0 or (na and rng.random() < 0.5) else 1
        X = (A, B)[spin]
        occ = [p for p in range(N) if X >> p & 1]
        vir = [p for p in range(N) if not X >> p & 1]
        X ^= 1 << occ[rng.integers(len(occ))] | 1 << vir[rng.integers(len(vir))]
        d = (X, B) if spin == 0 else (A, X)
        if d not in out:
            out.append(d)
    return np.array(out, dtype=np.uint64)


def load(w, keys, c, stated, log2_capacity):
    s = api.Solver(w.h, w.g, w.N, w.n_alpha, w.n_beta, log2_capacity=log2_capacity, z_threshold=1e9)
    hdr = api.cdfci_checkpoint_header()
    hdr.version, hdr.N, hdr.n_alpha, hdr.n_beta, hdr.num_coordinates = 1, w.N, w.n_alpha, w.n_beta, 1
    hdr.n_entries = hdr.n_slots = len(c)
    hdr.nnz_c = stated
    hdr.mu[0], hdr.scale[0] = float(c @ c), 1.0
    s.restore({"header": hdr, "keys": keys, "c": c, "b": np.zeros(len(c)), "flags": None})
    return s


@pytest.mark.parametrize("stated", [1, None, 1 << 30])
@pytest.mark.parametrize("N,na,nb,n,log2_capacity", [
    (6, 3, 2, 250, 9), (7, 2, 0, 19, 6), (5, 0, 2, 9, 5), (6, 3, 3, 1, 6), (9, 1, 4, 300, 22), (40, 5, 3, 60, 8),
    (33, 2, 2, 33, 22)])
def test_pair_sums_match_the_oracle(N, na, nb, n, log2_capacity, stated):
    rng = np.random.default_rng(100 * N + n)
    w = inputs.ab_initio(N, na, nb, seed=N + n, n_chol=6)
    keys = connected(N, na, nb, n, rng)
    c = rng.normal(size=len(keys))
    c[rng.random(len(c)) < 0.25] = 0.0
    c[0] = 1.0
    s = load(w, keys, c, int(np.count_nonzero(c)) if stated is None else stated, log2_capacity)
    try:
        g1, g2 = s.rdm()
        E = s.energy(1)
        w2 = inputs.ab_initio(N, na, nb, seed=N + n + 1, n_chol=6)
        E2 = s.energy_with(w2.h, w2.g)
    finally:
        s.close()
    o1, o2 = oracle.rdm(N, keys, c)
    assert np.abs(g1 - o1).max() <= 1e-12 * max(1.0, np.abs(o1).max())
    assert np.abs(g2 - o2).max() <= 1e-12 * max(1.0, np.abs(o2).max())
    for e, x in ((E, w), (E2, w2)):
        terms = np.abs(x.h * o1).sum() + 0.5 * np.abs(x.g * o2).sum()
        assert abs(e - (np.sum(x.h * o1) + 0.5 * np.sum(x.g * o2))) <= 1e-12 * terms
