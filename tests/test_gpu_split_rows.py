"""Estimator kernels whose CTA's warps share one particle's rows (few particles) against one warp per
particle (many): the same particles, alone and padded past the line between the two forms, and both
against the FP64 oracle; the cache's block sums where blocks straddle sweeps, are single rows, or
are fewer than the warps."""
import numpy as np
import pytest
import torch

from gpu_common import make_pair, state_round, tol
from oracle import oracle as O
from smc_workloads import small_glm

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def S():
    import paper_1805_03317_gb300 as pkg
    return pkg


def _problem(x_dtype, p, m, G, N, family="student_t"):
    wl = small_glm(family, n=5000, p=p, N=N, m=m, G=G, L=2, x_dtype=x_dtype, seed=19)
    prob, ctx = make_pair(wl)
    rng = np.random.default_rng(4)
    th = state_round(prob.theta_bar + 0.05 * rng.standard_normal((N, p)), x_dtype)
    u = rng.integers(0, wl.n, size=(N, m)).astype(np.int64)
    return wl, prob, ctx, th, u


# (rows, blocks): one sweep or less, fewer sweeps than warps, ragged last sweeps, one row per block
SHAPES = [(1, 1), (31, 31), (33, 2), (64, 3), (97, 5), (130, 1), (257, 64), (1000, 3)]


@pytest.mark.parametrize("x_dtype,p", [("bf16", 3), ("bf16", 20), ("bf16", 50), ("bf16", 101),
                                       ("f32", 13), ("f64", 6)])
@pytest.mark.parametrize("m,G", SHAPES)
def test_shared_and_single_warp_forms_match_oracle(x_dtype, p, m, G):
    few, many = 24, 700  # above 4 x 152 particles every storage type takes one warp per particle
    wl, prob, ctx, th, u = _problem(x_dtype, p, m, G, many)
    t = tol(x_dtype)
    ref = O.loglik_batch(prob, m, G, th[:few], u[:few], a=0.7, blocks=True)
    outs = []
    for n in (few, many):
        td, ud = torch.from_numpy(th[:n]).to(DEV), torch.from_numpy(u[:n]).to(DEV)
        g, ell, s2 = (v.cpu().double().numpy()[:few] for v in S().loglik_grad(ctx, td, ud, 0.7))
        e2 = S().loglik_est(ctx, td, ud)[0].cpu().numpy()[:few]
        np.testing.assert_allclose(ell, ref["ell"], rtol=t["ell"])
        np.testing.assert_allclose(e2, ref["ell"], rtol=t["ell"])
        s_scale = np.max(np.abs(ref["sigma2"])) * t["sig2"] + t["ell"] * np.max(np.abs(ref["ell"]))
        assert np.max(np.abs(s2 - ref["sigma2"])) <= s_scale
        gs = np.maximum(np.max(np.abs(ref["grad"]), axis=1, keepdims=True), 1.0)
        assert np.max(np.abs(g - ref["grad"]) / gs) <= t["grad"]
        # the autograd pair
        ta = td.to(ctx.state_dtype).clone().requires_grad_(True)
        el, sg = S().SubsampledLoglik.apply(ta, ud, ctx)
        (0.7 * el - 0.245 * sg).sum().backward()
        prior = -(th[:few] - wl.prior_mean) / wl.prior_var
        ga = ta.grad.cpu().double().numpy()[:few] + prior
        assert np.max(np.abs(ga - ref["grad"]) / gs) <= t["grad"]
        outs.append(ell)
    S().smc_free(ctx)


@pytest.mark.parametrize("x_dtype,p", [("bf16", 20), ("bf16", 50), ("f32", 13), ("f64", 6)])
@pytest.mark.parametrize("m,G", SHAPES)
@pytest.mark.parametrize("N", [24, 700])
def test_cache_block_sums_match_oracle(x_dtype, p, m, G, N):
    wl, prob, ctx, th, u = _problem(x_dtype, p, m, G, N)
    S().smc_set_particles(ctx, torch.from_numpy(th).to(DEV), torch.from_numpy(u).to(DEV))
    ell, s2, blk = (v.cpu().numpy()[:24] for v in S().smc_get_cache(ctx))
    S().smc_free(ctx)
    t = tol(x_dtype)
    ref = O.loglik_batch(prob, m, G, th[:24], u[:24], grad=False, blocks=True)
    np.testing.assert_allclose(ell, ref["ell"], rtol=t["ell"])
    s_scale = np.max(np.abs(ref["sigma2"])) * t["sig2"] + t["ell"] * np.max(np.abs(ref["ell"]))
    assert np.max(np.abs(s2 - ref["sigma2"])) <= s_scale
    for k in range(2):  # (sum d, sum d^2), to 1e-4 of the largest of each (1e-8 for FP64 rows)
        bar = (1e-8 if x_dtype == "f64" else 1e-4) * np.max(np.abs(ref["blocks"][..., k]))
        assert np.max(np.abs(blk[..., k] - ref["blocks"][..., k])) <= bar
