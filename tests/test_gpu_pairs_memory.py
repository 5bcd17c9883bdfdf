"""The pair sums (RDMs, gradient, exact Rayleigh quotient) where the device has no room for the list of nonzero
determinants that they make for speed: walked in the solver's own table; and where only a wrongly stated count asks for
too much: counted first.

Tolerance: both ways add the same terms c_I c_J / c.c (or times H_IJ), in other orders: 1e-12 of the largest entry, or of
the sum of the magnitudes of the energy's terms, as in test_gpu_pairs.py."""
import math

import numpy as np
import pytest

from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu
N, NA, NB = 14, 5, 4
ROWS = (1 << 20) + 11


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _strings(n):
    return np.array([x for x in range(1 << N) if bin(x).count("1") == n], dtype=np.uint64)


def _vector(rows, seed):
    rng = np.random.default_rng(seed)
    A, B = _strings(NA), _strings(NB)
    pick = rng.permutation(len(A) * len(B))[:rows]
    keys = np.stack([A[pick // len(B)], B[pick % len(B)]], axis=1)
    return keys, rng.normal(size=rows) / (1.0 + np.arange(rows)) ** 0.5


def _load(w, keys, c, stated, log2_capacity):
    s = api.Solver(w.h, w.g, N, NA, NB, log2_capacity=log2_capacity, grid_blocks=1, z_threshold=1e9)
    hdr = api.cdfci_checkpoint_header()
    hdr.version, hdr.N, hdr.n_alpha, hdr.n_beta, hdr.num_coordinates = 1, N, NA, NB, 1
    hdr.n_entries = hdr.n_slots = len(c)
    hdr.nnz_c = stated
    hdr.mu[0], hdr.scale[0] = float(c @ c), 1.0
    s.restore({"header": hdr, "keys": keys, "c": c, "b": np.zeros(len(c)), "flags": None})
    return s


def _sums(s, w2):
    g1, g2 = s.rdm()
    return g1, g2, s.energy(1), s.energy_with(w2.h, w2.g), *s.gradient()


@pytest.mark.parametrize("rows,stated,log2_capacity,leave", [
    (ROWS, ROWS, 21, 96 << 20),              # 142 MiB wanted: no list
    (ROWS, 1 << 33, 21, 96 << 20),           # stated above 2^31, the true number does not fit either
    (1234, 1 << 22, 22, 96 << 20),           # 4 Mi stated: counted, then the list of 1,234
])
def test_pair_sums_without_room(rows, stated, log2_capacity, leave):
    import torch
    w, w2 = inputs.ab_initio(N, NA, NB, seed=1), inputs.ab_initio(N, NA, NB, seed=2)
    assert rows <= math.comb(N, NA) * math.comb(N, NB)
    keys, c = _vector(rows, 5)
    s = _load(w, keys, c, rows, log2_capacity)
    try:
        want = _sums(s, w2)
    finally:
        s.close()
    s = _load(w, keys, c, stated, log2_capacity)
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")
    try:
        got = _sums(s, w2)
    finally:
        del fill
        torch.cuda.empty_cache()
        s.close()
    for x, y in zip(got, want):
        if np.ndim(x):
            assert np.abs(x - y).max() <= 1e-12 * max(1.0, np.abs(y).max())
    for k, u in ((2, w), (3, w2)):
        terms = np.abs(u.h * want[0]).sum() + 0.5 * np.abs(u.g * want[1]).sum()
        assert abs(got[k] - want[k]) <= 1e-12 * terms
