"""Export and checkpoint of the stored rows at table sizes around the blocks the rows are appended in (1024 slots, a
warp's 32), sparse and nearly full: every row once, values as loaded (exact: nothing is computed)."""
import numpy as np
import pytest

from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("log2_capacity,n", [(5, 1), (5, 25), (7, 100), (10, 1), (10, 800), (11, 1600), (12, 3), (21, 4900)])
def test_rows_come_back_once(log2_capacity, n):
    w = inputs.config1()
    rng = np.random.default_rng(n)
    strings = [x for x in range(256) if bin(x).count("1") == 4]
    pick = rng.choice(len(strings) ** 2, size=n, replace=False)
    keys = np.array([(strings[p // 70], strings[p % 70]) for p in pick], dtype=np.uint64)
    c, b = rng.normal(size=n), rng.normal(size=n)
    s = api.Solver(w.h, w.g, w.N, 4, 4, log2_capacity=log2_capacity, z_threshold=1e9)
    try:
        hdr = api.cdfci_checkpoint_header()
        hdr.version, hdr.N, hdr.n_alpha, hdr.n_beta, hdr.num_coordinates = 1, w.N, 4, 4, 1
        hdr.n_entries = hdr.n_slots = hdr.nnz_c = n
        hdr.mu[0], hdr.scale[0] = float(c @ c), 1.0
        s.restore({"header": hdr, "keys": keys, "c": c, "b": b, "flags": None})
        ck = s.checkpoint()
        for k2, c2, b2 in (s.export(), (ck["keys"], ck["c"], ck["b"])):
            got = {tuple(k): (x, y) for k, x, y in zip(k2.tolist(), c2, b2)}
            assert len(k2) == n and got == {tuple(k): (x, y) for k, x, y in zip(keys.tolist(), c, b)}
    finally:
        s.close()
