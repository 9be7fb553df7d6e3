"""A spin limit that no wait survives, on the FP32 tensor-core passes (one CTA a unit): the
gradient reports the timeout after its copies and MMAs in flight have landed, and the device
goes on."""
import numpy as np
import pytest

from oracle import model
from paper_1402_4089_gb300 import hmc, synthetic
from parity_util import assert_grad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chains", [1, 3])       # 19 and 57 columns
def test_gradient_times_out_and_leaves_the_device_usable(cuda, chains):
    X, y, _ = synthetic.make_problem(3000, 500, 20, seed=7)
    beta = (0.05 * np.random.default_rng(8).standard_normal((chains, 19, 500))).astype(np.float32)
    with hmc.create(X, y, 20, max_chains=chains, engine=4, spin_limit=1) as h:
        assert h.describe()["problems"][0]["tensor_cores"] is True
        for _ in range(3):
            with pytest.raises(hmc.HmcError) as ei:
                h.logpost_grad(beta)
            assert ei.value.status == hmc.ETIMEOUT
    with hmc.create(X, y, 20, max_chains=chains, engine=4) as h:
        _, g = h.logpost_grad(beta)
    assert_grad(g[0], model.grad_log_kernel(X, y, beta[0], "gaussian", 1.0), 1e-5)
