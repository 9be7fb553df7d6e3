"""Accuracy of the FP32 path on the tensor cores against 64 bits: no bias and no larger
error than FP32 arithmetic on the CUDA cores, whatever X holds (normal, sparse grey levels,
0/1 indicators, all positive), for 16, 32, 48 and 64 columns; sums that FP32 holds exactly
come out exactly; the posterior predictive.

Tolerances.  The gradient, a sum of residuals that mostly cancel, is compared with the one
that the CUDA-core engine forms from the same inputs: no more than half as far again from
64 bits.  Where that engine has no room for the classes, 2e-7 and 1e-6 for the largest of
thousands of coefficients: a logit (a few units) is a sum with errors of 3e-8 of the spread
of such sums (compensated additions, exact splits) and a rounding or two to FP32, about 1e-7
a row, and at most that of the gradient.  log K does not cancel: a drift common to all rows
is a few 1e-9, against 2.5e-8 and more of truncating sums, FP32 terms of a row are within
1e-7, random over 3000 rows or more (2e-9), expf and logf a few 1e-9: 1e-8."""
import numpy as np
import pytest

from oracle import model
from oracle import predict as opredict
from paper_1402_4089_gb300 import hmc
from parity_util import grad_errs

pytestmark = pytest.mark.gpu


def _design(kind, n, p, rng):
    if kind == "normal":
        return rng.standard_normal((n, p)).astype(np.float32)
    if kind == "pixels":
        return (rng.integers(1, 256, (n, p)) / 255.0 * (rng.random((n, p)) < 0.19)).astype(np.float32)
    if kind == "indicators":
        return (rng.random((n, p)) < 0.1).astype(np.float32)
    return rng.random((n, p)).astype(np.float32)


def _scale(kind, p):
    return 0.3 if kind in ("pixels", "indicators") else 2.0 / np.sqrt(p)


@pytest.mark.parametrize("kind", ["normal", "pixels", "indicators", "positive"])
@pytest.mark.parametrize("n,p,K,chains", [(20000, 785, 10, 1), (6000, 785, 20, 1), (6000, 500, 20, 2), (3000, 300, 33, 2)])
def test_gradient_and_log_kernel(cuda, kind, n, p, K, chains):
    import torch
    rng = np.random.default_rng(n + p + K)
    X = _design(kind, n, p, rng)
    beta = (rng.standard_normal((chains, K - 1, p)) * _scale(kind, p)).astype(np.float32)
    z = np.concatenate([X.astype(np.float64) @ beta[0].T.astype(np.float64), np.zeros((n, 1))], 1)
    y = np.argmax(z + rng.gumbel(size=z.shape), 1).astype(np.int32)
    got = {}
    for engine in (4, 1) if K <= 20 else (4,):
        with hmc.create(X, y, K, "gaussian", 10.0, max_chains=chains, engine=engine) as h:
            assert h.describe()["problems"][0].get("tensor_cores", False) is (engine == 4)
            lp, g = h.logpost_grad(torch.from_numpy(beta).to(cuda))
            got[engine] = lp.cpu().numpy(), g.cpu().numpy().astype(np.float64)
    X = X.astype(np.float64)
    for c in range(chains):
        b = beta[c].astype(np.float64)
        lo, go = model.log_kernel(X, y, b, "gaussian", 10.0), model.grad_log_kernel(X, y, b, "gaussian", 10.0)
        bound = [1.5 * e for e in grad_errs(got[1][1][c], go)] if 1 in got else (2e-7, 1e-6)
        norm, elem = grad_errs(got[4][1][c], go)
        assert norm <= bound[0] and elem <= bound[1], (kind, norm, elem, bound)
        assert abs(got[4][0][c] - lo) <= 1e-8 * abs(lo), (kind, (got[4][0][c] - lo) / lo)


@pytest.mark.parametrize("chains", [1, 4, 6, 8])       # 8, 32, 48 and 64 columns
def test_sums_that_fp32_holds_are_exact(cuda, chains):
    """At beta = 0 the residuals are 1 - 1/8 and -1/8: X of small integers makes every
    gradient a multiple of 1/8 below 2^18."""
    import torch
    rng = np.random.default_rng(41)
    n, p, K = 20000, 300, 8
    X = rng.integers(-8, 9, (n, p)).astype(np.float32)
    y = rng.integers(0, K, n).astype(np.int32)
    with hmc.create(X, y, K, "gaussian", 1.0, max_chains=chains, engine=4, layout="unconstrained") as h:
        assert h.describe()["problems"][0]["tensor_cores"] is True
        _, g = h.logpost_grad(torch.zeros((chains, K, p), device=cuda))
        g = g.cpu().numpy()
    want = ((y[:, None] == np.arange(K)) - 0.125).T @ X.astype(np.float64)
    for c in range(chains):
        assert np.array_equal(g[c], want)


@pytest.mark.parametrize("kind", ["normal", "indicators"])
@pytest.mark.parametrize("n,p,K,draws,tol", [(2000, 785, 10, 100, 2e-8), (500, 100, 3, 200, 1e-8)])
def test_predictive_probabilities(cuda, kind, n, p, K, draws, tol):
    """FP32 probabilities of one draw are within about 1e-7 of p (1 - p); the mean of 100 and
    200 random ones is within 1e-8, 5e-9, and FP32 rounding of the probabilities as much again."""
    import torch
    rng = np.random.default_rng(n + draws)
    X = _design(kind, n, p, rng)
    s = _scale(kind, p)
    d = (s * rng.standard_normal((1, K - 1, p)) + 0.3 * s * rng.standard_normal((draws, K - 1, p))).astype(np.float32)
    with hmc.create(X[:50].copy(), np.zeros(50, np.int32), K) as h:
        prob, _ = h.predict(torch.from_numpy(d).to(cuda), torch.from_numpy(X).to(cuda))
        prob = prob.cpu().numpy()
    ref, _ = opredict.predictive(X, d, "free")
    assert np.linalg.norm(prob - ref) <= tol * np.linalg.norm(ref)
