"""A spin limit that no wait survives, on the FP32 tensor-core passes (one CTA a unit): the
gradient reports the timeout after its copies and MMAs in flight have landed, and the device
goes on; a posterior predictive is formed by the general kernel, which has no waits."""
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


def test_predict_falls_back_on_the_general_kernel(cuda):
    import torch
    from oracle import predict as opredict
    rng = np.random.default_rng(9)
    n, p, K, draws = 900, 200, 6, 120
    X = rng.standard_normal((n, p)).astype(np.float32)
    d = (rng.standard_normal((draws, K - 1, p)) / np.sqrt(p)).astype(np.float32)
    with hmc.create(X[:20].copy(), np.zeros(20, np.int32), K, spin_limit=1) as h:
        prob, _ = h.predict(torch.from_numpy(d).to(cuda), torch.from_numpy(X).to(cuda))
    assert np.max(np.abs(prob.cpu().numpy() - opredict.predictive(X, d, "free")[0])) <= 1e-5   # as in test_gpu_predict
