"""Paths that the default choice no longer takes at the sizes of older tests, each on request:
replayed call graphs of the fused CUDA-core engine and of the FP32 tensor-core chain, with
buffer contents, buffers, chains and step size changing between calls; the FP32 two-pass
CUDA-core kernels with more than 16 columns; edge shapes and FP64 on the fused kernel; a batch
of FP32 problems on the two-pass engine; non-finite rows of a posterior predictive against
calls of few draws, which the general kernel answers.  Against the FP64 oracle; tolerances as
in test_gpu_parity (FP32 1e-5, FP64 1e-11, states 1e-4 and 1e-10 of their scale)."""
import numpy as np
import pytest

from oracle import hmc as ohmc
from oracle import model
from paper_1402_4089_gb300 import hmc, synthetic
from parity_util import assert_grad, lk_err

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-5, "f64": 1e-11}
STATE = {"f32": 1e-4, "f64": 1e-10}


def _problem(n, p, K, xs, seed):
    return synthetic.make_problem(n, p, K, seed=seed, dtype=np.float64 if xs == "f64" else np.float32)[:2]


def _route(h):
    d = h.describe()
    pr = d["problems"][0]
    return d["engine"], bool(pr.get("tensor_cores")), bool(pr.get("one_launch"))


@pytest.mark.parametrize("xs,engine,route", [("f64", 1, ("simt", False, False)), ("f32", 1, ("simt", False, False)),
                                             ("f32", 4, ("simt_2pass", True, False))])
def test_gradient_replays_follow_buffer_contents(cuda, xs, engine, route):
    import torch
    n, p, K, chains = 1500, 70, 12, 3
    X, y = _problem(n, p, K, xs, 71)
    rng = np.random.default_rng(72)
    with hmc.create(X, y, K, "cauchy", 1.0, x_storage=xs, state=xs, max_chains=chains, engine=engine) as h:
        assert _route(h) == route
        beta = torch.zeros((chains, K - 1, p), dtype=h.torch_dtype(), device=cuda)
        other = torch.zeros_like(beta)
        grads = [torch.empty_like(beta), torch.empty_like(beta)]
        lp = torch.empty(chains, dtype=torch.float64, device=cuda)

        def check(src, out, m, what):
            b = (0.2 * rng.standard_normal((m, K - 1, p))).astype(X.dtype)
            src[:m].copy_(torch.from_numpy(b))
            h.logpost_grad(src[:m], chains=m, logpost=lp[:m], grad=out[:m])
            torch.cuda.synchronize()
            for c in range(m):
                b64 = b[c].astype(np.float64)
                assert lk_err(lp[c].item(), model.log_kernel(X, y, b64, "cauchy", 1.0)) <= TOL[xs], (what, c)
                assert_grad(out[c].cpu().numpy(), model.grad_log_kernel(X, y, b64, "cauchy", 1.0), TOL[xs], (what, c))
        for it in range(5):                        # captured with the second call, replayed from the third
            check(beta, grads[0], chains, it)
        check(beta, grads[1], chains, "another gradient buffer")
        check(other, grads[1], chains, "another coefficient buffer")
        for it in range(3):
            check(other, grads[1], 2, ("fewer chains", it))
        check(beta, grads[0], chains, "the first buffers again")


@pytest.mark.parametrize("xs,engine,route", [("f64", 1, ("simt", False, False)), ("f32", 4, ("simt_2pass", True, False))])
def test_leapfrog_replays_continue_the_trajectory(cuda, xs, engine, route):
    import torch
    n, p, K, L, eps, chains = 1500, 30, 12, 5, 0.004, 2
    X, y = _problem(n, p, K, xs, 73)
    rng = np.random.default_rng(74)
    b0 = (0.1 * rng.standard_normal((chains, K - 1, p))).astype(X.dtype)
    e0 = rng.standard_normal((chains, K - 1, p)).astype(X.dtype)
    with hmc.create(X, y, K, "gaussian", 2.0, x_storage=xs, state=xs, max_chains=chains, engine=engine) as h:
        assert _route(h) == route
        q, m = torch.from_numpy(b0).to(cuda), torch.from_numpy(e0).to(cuda)
        g = torch.empty_like(q)
        lp = torch.empty(chains, dtype=torch.float64, device=cuda)
        h.logpost_grad(q, logpost=lp, grad=g)
        ref = [(b0[c].astype(np.float64), e0[c].astype(np.float64)) for c in range(chains)]
        for it in range(6):
            step = eps if it != 3 else 0.5 * eps     # call 4 changes eps: a new graph
            h.leapfrog(q, m, L, step, grad=g, logpost=lp)
            torch.cuda.synchronize()
            for c in range(chains):
                bo, eo, lko, go = ohmc.leapfrog(X, y, *ref[c], step, L, "gaussian", 2.0)
                ref[c] = bo, eo
                for got, want in ((q, bo), (m, eo)):
                    assert np.max(np.abs(got[c].cpu().numpy() - want)) <= STATE[xs] * max(1.0, np.max(np.abs(want))), (it, c)
                assert lk_err(lp[c].item(), lko) <= 10 * TOL[xs], (it, c)
                assert_grad(g[c].cpu().numpy(), go, 20 * TOL[xs], (it, c))


# Wide X with few rows stays on the CUDA cores: 38, 60 and 64 columns, 19 and 11 with fewer classes.
@pytest.mark.parametrize("n,p,K,chains", [(100, 5000, 39, 1), (130, 1100, 21, 3), (60, 2000, 65, 1), (300, 5000, 20, 1),
                                          (257, 3001, 12, 1)])
def test_two_pass_cuda_cores_with_many_columns(cuda, n, p, K, chains):
    import torch
    X, y = _problem(n, p, K, "f32", 75)
    beta = (np.random.default_rng(76).standard_normal((chains, K - 1, p)) * 0.5 / np.sqrt(p)).astype(np.float32)
    with hmc.create(X, y, K, "cauchy", 1.0, max_chains=chains, engine=4) as h:
        assert _route(h) == ("simt_2pass", False, False)
        runs = [h.logpost_grad(torch.from_numpy(beta).to(cuda)) for _ in range(2)]
        assert all(torch.equal(a, b) for a, b in zip(*runs))
        lp, g = (v.cpu().numpy() for v in runs[0])
    for c in range(chains):
        b = beta[c].astype(np.float64)
        assert lk_err(lp[c], model.log_kernel(X, y, b, "cauchy", 1.0)) <= TOL["f32"]
        assert_grad(g[c], model.grad_log_kernel(X, y, b, "cauchy", 1.0), TOL["f32"], c)


@pytest.mark.parametrize("xs", ["f32", "f64"])
@pytest.mark.parametrize("n,p,K,chains", [(1, 1, 2, 1), (1, 300, 4, 2), (37, 5, 3, 1), (65, 257, 6, 2), (100, 10, 2, 4)])
def test_edge_shapes_of_the_fused_kernel(cuda, xs, n, p, K, chains):
    import torch
    X, y = _problem(n, p, K, xs, 77)
    beta = (np.random.default_rng(78).standard_normal((chains, K - 1, p)) * 0.5 / np.sqrt(p)).astype(X.dtype)
    with hmc.create(X, y, K, "cauchy", 0.7, x_storage=xs, state=xs, max_chains=chains, engine=1) as h:
        assert _route(h) == ("simt", False, False)
        lp, g = (v.cpu().numpy() for v in h.logpost_grad(torch.from_numpy(beta).to(cuda)))
    for c in range(chains):
        b = beta[c].astype(np.float64)
        assert lk_err(lp[c], model.log_kernel(X, y, b, "cauchy", 0.7)) <= TOL[xs]
        assert_grad(g[c], model.grad_log_kernel(X, y, b, "cauchy", 0.7), TOL[xs], c)


def test_batch_of_fp32_problems_on_the_two_pass_engine(cuda):
    import torch
    shapes = [(2500, 130, 12), (20000, 64, 9), (90, 400, 21), (1, 5, 3)]
    probs = [_problem(n, p, K, "f32", 79 + i) for i, (n, p, K) in enumerate(shapes)]
    rng = np.random.default_rng(80)
    betas = [(0.1 * rng.standard_normal((2, K - 1, p))).astype(np.float32) for _, p, K in shapes]
    with hmc.create_batch([q[0] for q in probs], [q[1] for q in probs], [s[2] for s in shapes], "gaussian", 3.0,
                          max_chains=2, engine=4) as h:
        assert h.describe()["engine"] == "simt_2pass"
        lp, g = h.logpost_grad(torch.from_numpy(np.concatenate([b.ravel() for b in betas])).to(cuda), chains=2)
        lp, g = lp.cpu().numpy(), g.cpu().numpy()
    off = 0
    for b, ((X, y), (n, p, K)) in enumerate(zip(probs, shapes)):
        gb = g[off:off + 2 * (K - 1) * p].reshape(2, K - 1, p)
        off += gb.size
        for c in range(2):
            b64 = betas[b][c].astype(np.float64)
            assert lk_err(lp[2 * b + c], model.log_kernel(X, y, b64, "gaussian", 3.0)) <= TOL["f32"]
            assert_grad(gb[c], model.grad_log_kernel(X, y, b64, "gaussian", 3.0), TOL["f32"], (b, c))


def test_non_finite_rows_of_a_predictive(cuda):
    """Against the mean over calls of ten draws of the same 24 rows (0.6 x 10 x 7 us of work by
    the general kernel's own estimate: below what the tensor cores take).  A row at minus
    infinity where every coefficient is positive belongs to the last class."""
    import torch
    rng = np.random.default_rng(81)
    n, p, K, draws = 2000, 200, 5, 100
    X = rng.standard_normal((n, p)).astype(np.float32)
    X[3, 7], X[5, 7], X[9, 1], X[11, :], X[13, :] = -np.inf, np.inf, np.nan, 3e38, -3e38
    d = rng.standard_normal((draws, K - 1, p)).astype(np.float32)
    d[:, :, 7] = np.abs(d[:, :, 7]) + 0.1
    d[40:, 0, 3] = np.inf                                   # and draws that have diverged
    with hmc.create(X[100:120].copy(), np.zeros(20, np.int32), K) as h:
        Xt, dt = torch.from_numpy(X).to(cuda), torch.from_numpy(d).to(cuda)
        for D in (40, draws):
            prob, cls = (v.cpu().numpy() for v in h.predict(dt[:D].contiguous(), Xt))
            few = [h.predict(dt[i:i + 10].contiguous(), Xt[:24].contiguous())[0].cpu().numpy() for i in range(0, D, 10)]
            want = np.mean(few, axis=0)
            assert np.allclose(prob[:24], want, rtol=0, atol=1e-5, equal_nan=True)
            if D == 40:
                assert np.array_equal(prob[3], [0, 0, 0, 0, 1]) and cls[3] == 4
                assert np.all(np.isnan(prob[5])) and np.all(np.isnan(prob[9])) and np.all(np.isfinite(prob[:3]))
