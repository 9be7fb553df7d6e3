"""The prior's derivative to the last bit: with X = 0 the gradient is the prior's alone, and
IEEE division fixes it (Gaussian: -b / s^2; FP64 one-launch path and FP64, FP32 CUDA cores)."""
import numpy as np
import pytest

from paper_1402_4089_gb300 import hmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("xs,engine", [("f64", 0), ("f64", 1), ("f32", 0), ("f32", 1)])
@pytest.mark.parametrize("scale", [3.0, 0.7, 1e-155, 1e155])
def test_gaussian_derivative(cuda, xs, engine, scale):
    import torch
    dt = np.float64 if xs == "f64" else np.float32
    if xs == "f32" and not 1e-10 < scale < 1e10:
        pytest.skip("the square leaves FP32")
    rng = np.random.default_rng(5)
    n, p, K = 20, 50, 4
    b = rng.standard_normal((1, K - 1, p)).astype(dt) * dt(min(scale, 1.0))
    with hmc.create(np.zeros((n, p), dt), np.zeros(n, np.int32), K, "gaussian", scale, x_storage=xs, state=xs,
                    engine=engine) as h:
        assert bool(h.describe()["problems"][0].get("one_launch")) is (engine == 0)
        g = h.logpost_grad(torch.from_numpy(b).to(cuda))[1].cpu().numpy()
    assert np.array_equal(g, -b / dt(scale * scale))
