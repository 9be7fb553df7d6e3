"""Infinite and NaN coefficients (a diverging chain) beside finite chains, on every path of
FP32 X and the one-launch path of FP64: an infinite coefficient makes infinite logits where X
is positive, so a class at minus infinity has probability zero and the rest of the gradient
is what it is without that class; plus infinity and NaN make NaN; finite chains of the same
call are bit for bit what they are without the others.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

from oracle import model
from paper_1402_4089_gb300 import hmc
from parity_util import assert_grad

pytestmark = pytest.mark.gpu


# FP32 on the tensor cores with 32 and 64 columns, both CUDA-core engines, the one-launch path.
@pytest.mark.parametrize("n,p,K,xs,engine", [(700, 130, 9, "f32", 4), (700, 130, 17, "f32", 4), (20000, 70, 5, "f32", 4),
                                             (700, 130, 9, "f32", 1), (40, 400, 6, "f32", 4), (60, 20, 5, "f32", 0),
                                             (60, 20, 5, "f64", 0)])
def test_infinite_coefficients(cuda, n, p, K, xs, engine):
    import torch
    dt = np.float64 if xs == "f64" else np.float32
    rng = np.random.default_rng(n + K)
    X = (np.abs(rng.standard_normal((n, p))) + 0.1).astype(dt)
    y = rng.integers(0, K, n).astype(np.int32)
    good = (rng.standard_normal((4, K - 1, p)) * 0.3 / np.sqrt(p)).astype(dt)
    bad = good.copy()
    bad[1, 2, 5], bad[2, 1, 3], bad[3, 0, 7] = -np.inf, np.inf, np.nan
    with hmc.create(X, y, K, "gaussian", 2.0, x_storage=xs, state=xs, max_chains=4, engine=engine) as h:
        run = lambda b: [v.cpu().numpy() for v in h.logpost_grad(torch.from_numpy(b).to(cuda))]  # noqa: E731
        lp0, g0 = run(good)
        lp, g = run(bad)
    assert lp[0] == lp0[0] and np.array_equal(g[0], g0[0])
    assert lp[1] == -np.inf and g[1, 2, 5] == np.inf
    b = good[1].astype(np.float64)
    b[2] = -1e6                                            # probability zero, as at minus infinity
    X64 = X.astype(np.float64)
    want = model.grad_log_kernel(X64, y, b, "gaussian", 2.0) + b / 4.0 - good[1].astype(np.float64) / 4.0
    g[1, 2, 5] = want[2, 5] = 0.0
    assert_grad(g[1], want, 1e-11 if xs == "f64" else 1e-5)
    for c in (2, 3):
        assert not np.isfinite(lp[c]) and np.all(np.isnan(g[c]))
