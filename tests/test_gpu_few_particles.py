"""The estimator's two orders of summation: few particles (a CTA's warps share one) and many (one warp
each). A context's calls of up to N particles use one of them, so a particle's values do not depend on
the rest of the call; and the two agree to FP32 (FP64) rounding, also far from the centre, where
the warps' shifts, the d of their first rows, lie far apart."""
import numpy as np
import pytest
import torch

from gpu_common import make_pair, state_round
from oracle import oracle as O
from smc_workloads import small_glm

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
FEW, MANY = 40, 700  # above four particles per SM every storage type takes one warp per particle


def S():
    import paper_1805_03317_gb300 as pkg
    return pkg


def _contexts(x_dtype, p, m, G, spread):
    wl = small_glm("student_t", n=5000, p=p, N=MANY, m=m, G=G, L=2, x_dtype=x_dtype, seed=41)
    prob, many = make_pair(wl)
    wl.N = FEW
    _, few = make_pair(wl, theta_bar=prob.theta_bar)
    rng = np.random.default_rng(9)
    th = state_round(prob.theta_bar + spread * rng.standard_normal((MANY, p)), x_dtype)
    u = rng.integers(0, wl.n, size=(MANY, m)).astype(np.int64)
    return wl, prob, few, many, th, u


def _calls(ctx, th, u):
    """Everything an estimator call returns for these particles."""
    t, i = torch.from_numpy(th).to(DEV), torch.from_numpy(u).to(DEV)
    g, ell, s2 = S().loglik_grad(ctx, t, i, 0.7)
    out = [g, ell, s2, *S().loglik_est(ctx, t, i)]
    ta = t.to(ctx.state_dtype).clone().requires_grad_(True)
    el, sg = S().SubsampledLoglik.apply(ta, i, ctx)
    (0.7 * el - 0.245 * sg).sum().backward()
    return out + [el.detach(), sg.detach(), ta.grad]


@pytest.mark.parametrize("x_dtype,p", [("bf16", 20), ("f32", 13), ("f64", 6)])
def test_values_do_not_depend_on_the_rest_of_the_call(x_dtype, p):
    wl, prob, few, many, th, u = _contexts(x_dtype, p, 130, 5, 0.1)
    for ctx, n in ((few, FEW), (many, MANY)):
        whole = _calls(ctx, th[:n], u[:n])
        for a, b in ((0, 1), (3, 30)):
            for x, y in zip(_calls(ctx, th[a:b], u[a:b]), whole):
                assert torch.equal(x, y[a:b])
        S().smc_free(ctx)


@pytest.mark.parametrize("x_dtype,p", [("bf16", 3), ("bf16", 20), ("bf16", 50), ("bf16", 101),
                                       ("f32", 13), ("f64", 6)])
@pytest.mark.parametrize("m,G", [(1, 1), (31, 4), (97, 5), (1000, 3)])
@pytest.mark.parametrize("spread", [0.05, 0.5])
def test_the_two_orders_agree_to_rounding(x_dtype, p, m, G, spread):
    wl, prob, few, many, th, u = _contexts(x_dtype, p, m, G, spread)
    a = [v.cpu().double().numpy() for v in _calls(few, th[:FEW], u[:FEW])]
    b = [v.cpu().double().numpy()[:FEW] for v in _calls(many, th, u)]
    S().smc_free(few)
    S().smc_free(many)
    # A sum of m terms is 1 + m/32 additions in a lane, 5 over the lanes and 3 over the warps: with
    # unit rounding eps it errs by (m/32 + 9) eps of sum |e|, |e| <= |d| + |K|, and K is one of the d
    eps = (m / 32 + 9) * 2.0 ** (-53 if x_dtype == "f64" else -24)
    ref = O.loglik_batch(prob, m, G, th[:FEW], u[:FEW], a=0.7, blocks=True)
    nm = wl.n / m
    q = ref["blocks"][..., 1].sum(1)  # sum d^2
    dmax = np.sqrt(q)                 # >= |d| of every row
    s1 = np.sqrt(m * q) + m * dmax    # >= sum |e|
    s2 = 2 * (q + m * dmax ** 2)      # >= sum e^2
    for k in (1, 3, 5):
        assert np.all(np.abs(a[k] - b[k]) <= 2 * eps * nm * s1 + 1e-12 * np.abs(b[k])), k
    for k in (2, 4, 6):
        assert np.all(np.abs(a[k] - b[k]) <= 2 * eps * nm ** 2 * (s2 + 2 * s1 ** 2 / m)
                      + 1e-12 * np.abs(b[k])), k
    # gradients: r and x are O(1) here, so nm times the same sums with |x| <= xm
    xm, rm = np.abs(wl.X).max(), 10.0
    bar = 2 * eps * (0.7 * nm * m * rm * xm + 0.49 * nm ** 2 * 2 * s1 * rm * xm)
    for k in (0, 7):
        assert np.all(np.abs(a[k] - b[k]) <= bar[:, None] + 1e-6 * np.abs(b[k])), k
