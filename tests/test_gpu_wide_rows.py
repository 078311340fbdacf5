"""The resident tiles for BF16 rows of 41 to 64 covariates (hmc_kernel 26: up to 56, 27: up to 64)
compute what the streamed trajectory kernel (hmc_kernel 1) computes: the same theta and u bit for bit,
since one last bit of theta where |theta| is a few units is enough to move sigma2_hat by 1e-5. What
they write back (l_hat, sigma2_hat, block sums) is held against the FP64 oracle too."""
import numpy as np
import pytest
import torch

from gpu_common import device_arrays, make_pair, state_round, tol
from oracle import oracle as O
from smc_workloads import small_glm

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def S():
    import paper_1805_03317_gb300 as pkg
    return pkg


def _moved(wl, th, u, theta_bar, hmc_kernel, a=0.3, eps=0.3, moves=1, **kw):
    prob, ctx = make_pair(wl, theta_bar=theta_bar, hmc_kernel=hmc_kernel, **kw)
    S().smc_set_particles(ctx, torch.from_numpy(th).to(DEV), torch.from_numpy(u).to(DEV))
    S().smc_set_scalars(ctx, 2, a, eps, 0.0)
    S().smc_reweight(ctx)
    acc = S().smc_move(ctx, moves)
    out = [t.cpu() for t in (*S().smc_get_particles(ctx), *S().smc_get_cache(ctx))]
    S().smc_free(ctx)
    return prob, acc, out


def _compare(wl, hmc_kernel, spread=0.03, **kw):
    prob, ctx = make_pair(wl)
    S().smc_free(ctx)
    rng = np.random.default_rng(5)
    th = state_round(prob.theta_bar + spread * rng.standard_normal((wl.N, wl.p)), "bf16")
    u = rng.integers(0, wl.n, size=(wl.N, wl.m)).astype(np.int64)
    _, acc_s, ref = _moved(wl, th, u, prob.theta_bar, 1, **kw)
    _, acc_w, got = _moved(wl, th, u, prob.theta_bar, hmc_kernel, **kw)
    moved = torch.any(ref[0].double() != torch.from_numpy(th), dim=1).float().mean()
    assert moved > 0.1, moved
    assert acc_s == acc_w
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    # estimates: the block sums of the two kernels differ by FP32 rounding of at most 13 additions
    # (8 rows per lane, 5 shuffles): 13 x 2^-24 < 1e-6 of the sums of |e|, |e|^2
    scale = ref[5].abs().amax(dim=(0, 1))
    assert torch.all((got[5] - ref[5]).abs() <= 1e-5 * scale)
    np.testing.assert_allclose(got[3], ref[3], rtol=1e-6)
    assert torch.all((got[4] - ref[4]).abs() <= 1e-5 * ref[4].abs().amax())
    return prob, got


FAMILIES = ["logistic", "poisson", "probit", "gaussian", "student_t"]


@pytest.mark.parametrize("family", FAMILIES)
@pytest.mark.parametrize("p,hmc_kernel", [(41, 26), (48, 26), (49, 26), (56, 26), (50, 27),
                                          (57, 27), (64, 27)])
def test_wide_tiles_move_particles_as_the_streamed_kernel(family, p, hmc_kernel):
    kw = dict(x_scale=0.3) if family == "poisson" else {}
    wl = small_glm(family, n=6000, p=p, N=320, m=90, G=6, L=4, x_dtype="bf16", seed=23, **kw)
    _compare(wl, hmc_kernel)


@pytest.mark.parametrize("m,G", [(1, 1), (31, 3), (32, 1), (33, 33), (257, 2), (300, 1), (1025, 9)])
@pytest.mark.parametrize("p", [52, 60])
def test_wide_tiles_row_edges(m, G, p):
    """Partial sweeps, fewer sweeps than row warps, one row per block, blocks of more than eight
    rows per lane."""
    wl = small_glm("student_t", n=6000, p=p, N=320, m=m, G=G, L=3, x_dtype="bf16", seed=29)
    _compare(wl, 26 if p <= 56 else 27)


def test_wide_tiles_first_order_control_variates():
    wl = small_glm("logistic", n=6000, p=50, N=320, m=90, G=6, L=3, x_dtype="bf16", seed=7)
    _compare(wl, 26, cv_order=1)


@pytest.mark.parametrize("p,hmc_kernel", [(50, 26), (61, 27)])
@pytest.mark.parametrize("family", ["logistic", "student_t"])
def test_wide_tiles_cache_after_moves_matches_oracle(family, p, hmc_kernel):
    wl = small_glm(family, n=6000, p=p, N=320, m=257, G=5, L=4, x_dtype="bf16", seed=31)
    prob, got = _compare(wl, hmc_kernel)
    th, u = got[0].double().numpy(), got[1].numpy().astype(np.int64)
    ref = O.loglik_batch(prob, wl.m, wl.G, th, u, grad=False, blocks=True)
    t = tol("bf16")
    ell, s2, blk = (v.numpy() for v in got[3:])
    np.testing.assert_allclose(ell, ref["ell"], rtol=t["ell"])
    s_scale = np.max(np.abs(ref["sigma2"])) * t["sig2"] + t["ell"] * np.max(np.abs(ref["ell"]))
    assert np.max(np.abs(s2 - ref["sigma2"])) <= s_scale
    for k in range(2):
        # 1e-4 of the largest, and what the FP32 logistic form past |D| = 1/2 may err by (3e-7
        # absolute per row's d, a block of 52 rows)
        bar = 1e-4 * np.max(np.abs(ref["blocks"][..., k])) + 52 * 3e-7
        assert np.max(np.abs(blk[..., k] - ref["blocks"][..., k])) <= bar


def _batch_equals_singles(shapes, kernels, N=40):
    """A batch of (family, p, m, G) problems, stepped with and without a graph, against the problems
    alone: particles and cache bit for bit."""
    wls = [small_glm(f, n=3000, p=p, N=N, m=m, G=G, L=2, x_dtype="bf16", seed=80 + p)
           for f, p, m, G in shapes]
    dicts = []
    for w in wls:
        X, y = device_arrays(w)
        dicts.append(dict(X=X, y=y, family=w.family, prior_mean=w.prior_mean,
                          prior_var=w.prior_var, N=w.N, m=w.m, G=w.G, L=w.L, seed=w.seed,
                          noise_sigma=w.sigma, dof=w.dof))
    b = S().smc_batch_init(dicts)
    got = [S().smc_batch_hmc_kernel(b, q) for q in range(len(wls))]
    assert got[:len(kernels)] == kernels
    singles = [make_pair(w, tile_hint=S().smc_batch_tile(b), hmc_kernel=got[q],
                         theta_bar=S().smc_get_centre(S().smc_batch_context(b, q))[0])[1]
               for q, w in enumerate(wls)]
    for use_graph in (False, True):
        S().smc_batch_stage(b, 1, use_graph=use_graph)
        for c in singles:
            S().smc_reweight(c)
            S().smc_resample(c)
            S().smc_move(c, 1)
    for q, c in enumerate(singles):
        m = S().smc_batch_context(b, q)
        for x, y in zip((*S().smc_get_particles(m), *S().smc_get_cache(m)),
                        (*S().smc_get_particles(c), *S().smc_get_cache(c))):
            assert torch.equal(x, y), q
        S().smc_free(c)
    S().smc_batch_free(b)


def test_wide_batch_equals_single_problems():
    """The row terms have one rounding in every kernel (alone and in a batch)."""
    _batch_equals_singles([("student_t", 50, 700, 20), ("logistic", 56, 300, 7),
                           ("probit", 41, 200, 5), ("gaussian", 60, 257, 3),
                           ("student_t", 63, 150, 4), ("poisson", 9, 120, 4)],
                          [26, 26, 26, 27, 27])


def test_batch_group_whose_members_fit_alone_but_not_together():
    """p = 50 with m = 1500, G = 50 and p = 45 with m = 600, G = 200 each leave room on an SM, a plan
    of m = 1500 and G = 200 does not: the batch runs them as two groups of one tile."""
    _batch_equals_singles([("student_t", 50, 1500, 50), ("logistic", 45, 600, 200),
                           ("student_t", 47, 1490, 40), ("probit", 9, 120, 4)], [26, 26, 26])
