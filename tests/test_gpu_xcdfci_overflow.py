"""xCDFCI with gradients whose square exceeds FP64: an error, not convergence; the same integrals at a scale whose squares
fit take their steps."""
import numpy as np
import pytest

from paper_2605_04483_gb300 import api, inputs
from gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("states", [2, 5])
def test_an_overflowing_gradient_is_an_error(states):
    w = inputs.ab_initio(8, 3, 2, seed=4)
    s = api.Solver(w.h * 1e155, w.g * 1e155, w.N, 3, 2, num_states=states, log2_capacity=12)
    try:
        with pytest.raises(api.CdfciError) as e:
            s.step(3)
        assert e.value.code == -2                       # CDFCI_ERR_NONFINITE
    finally:
        s.close()
    s = api.Solver(w.h, w.g, w.N, 3, 2, num_states=states, log2_capacity=12)
    try:
        st = s.step(3)
        assert st["iterations"] == 3 and st["converged"] == 0 and np.isfinite(s.energies()).all()
    finally:
        s.close()
