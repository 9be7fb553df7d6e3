"""FP64 sums of FP32 terms lose nothing to the FP32 arithmetic that prepares them: the
log-prior of four coefficients (n = 0: log K is the prior's alone) and the posterior
predictive of eight draws (their probabilities, FP32 values, taken from calls of one draw;
p = 64: one step of the contraction, so that a draw's logits are the same in any company).
The terms are added exactly here (fsum); a few FP64 roundings: 4 x 2^-53 of the sum."""
import math

import numpy as np
import pytest

from paper_1402_4089_gb300 import hmc

pytestmark = pytest.mark.gpu
TOL = 4 * 2.0 ** -53


def test_log_prior(cuda):
    import torch
    chains, p = 512, 4
    b = np.random.default_rng(3).standard_normal((chains, 1, p)).astype(np.float32)
    with hmc.create(np.zeros((0, p), np.float32), np.zeros(0, np.int32), 2, "gaussian", 2.0, max_chains=chains) as h:
        lp = h.logpost_grad(torch.from_numpy(b).to(cuda))[0].cpu().numpy()
    x = b[:, 0] / np.float32(2.0)
    terms = np.float32(-0.5) * x * x
    for c in range(chains):
        want = math.fsum(float(t) for t in terms[c])
        assert abs(lp[c] - want) <= TOL * abs(want), c


def test_mean_probabilities(cuda):
    import torch
    n, p, K, draws = 600000, 64, 12, 8
    rng = np.random.default_rng(4)
    X = torch.from_numpy(rng.standard_normal((n, p)).astype(np.float32)).to(cuda)
    d = torch.from_numpy((1.0 * rng.standard_normal((draws, K - 1, p))).astype(np.float32)).to(cuda)
    with hmc.create(X[:20].cpu().numpy(), np.zeros(20, np.int32), K) as h:
        prob = h.predict(d, X)[0][:1500].cpu().numpy()
        one = [h.predict(d[i:i + 1].contiguous(), X)[0][:1500].cpu().numpy() for i in range(draws)]
    assert all(np.array_equal(o, o.astype(np.float32)) for o in one)
    for i in range(1500):
        for k in range(K):
            want = math.fsum(o[i, k] for o in one) / draws
            assert abs(prob[i, k] - want) <= TOL * want, (i, k)
