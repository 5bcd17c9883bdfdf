"""Export into device arrays: written in place when they are aligned for the row stores (16 bytes for the keys),
else through a copy; any of them may be left out.  The rows are the ones of the export into host arrays (exact)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _sorted(keys, *cols):
    o = np.lexsort((keys[:, 0], keys[:, 1]))
    return [x[o] for x in (keys, *cols)]


@pytest.mark.parametrize("states", [1, 2, 3])
@pytest.mark.parametrize("shift", [0, 1])
def test_device_arrays_hold_the_host_rows(states, shift):
    w = inputs.ab_initio(8, 3, 2, seed=5)
    s = api.Solver(w.h, w.g, w.N, w.n_alpha, w.n_beta, num_states=states, log2_capacity=13)
    try:
        s.step(30)
        keys, c, b = s.export() if states == 1 else s.export_states()
        want = _sorted(keys, c, b)
        n, got = len(keys), ctypes.c_int64()
        call = api.lib().cdfci_export if states == 1 else api.lib().cdfci_export_states
        dk = torch.zeros(2 * n + 1, dtype=torch.int64, device="cuda")[shift:shift + 2 * n]
        dc = torch.zeros(n * states + 1, dtype=torch.float64, device="cuda")[shift:shift + n * states]
        db = torch.zeros_like(dc)
        api._check(call(s.handle, dk.data_ptr(), dc.data_ptr(), db.data_ptr(), n, ctypes.byref(got)))
        assert got.value == n
        have = _sorted(dk.cpu().numpy().view(np.uint64).reshape(n, 2), dc.cpu().numpy().reshape(np.shape(c)),
                       db.cpu().numpy().reshape(np.shape(b)))
        assert all(np.array_equal(x, y) for x, y in zip(have, want))
        dc.zero_()
        api._check(call(s.handle, None, dc.data_ptr(), None, n, ctypes.byref(got)))
        assert np.array_equal(np.sort(dc.cpu().numpy()), np.sort(np.ravel(c)))
    finally:
        s.close()
