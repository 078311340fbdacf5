"""What the kernels give for FP32 particle states, held to recorded outputs (tests/golden/fp32_pins.npz).

An FP32 trajectory multiplies rounding: one last bit of theta where |theta| is a few units is 1e-5 of
theta - theta_bar, and sigma2_hat goes with about the sixth power of that. So row terms, row sums and
the moments at the centre keep their order of operations, and a move's end points are compared bit
for bit; estimates to 1e-6 of their norm, a twentieth of what a last bit of theta can do."""
import os

import numpy as np
import pytest
import torch

from gpu_common import make_pair, state_round
from smc_workloads import small_glm

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
PINS = os.path.join(os.path.dirname(__file__), "golden", "fp32_pins.npz")

# name: family, storage, sizes (n, p, N, m, G, L), scale of theta, spread of the cloud, temperature
GRADS = {
    "grad_logistic_f32_p2": ("logistic", "f32", (5000, 2, 64, 810, 7, 2), 0.5, 0.17, 0.05),
    "grad_logistic_f32_p4": ("logistic", "f32", (5000, 4, 64, 300, 5, 2), 1.0, 0.12, 0.05),
    "grad_logistic_bf16_p20": ("logistic", "bf16", (5000, 20, 64, 300, 5, 2), 0.3, 0.06, 0.05),
}
MOVES = {
    "move_logistic_bf16_p3": ("logistic", "bf16", (6000, 3, 256, 58, 4, 17), 1.0, 0.05, 0.03),
    "move_student_t_bf16_p50": ("student_t", "bf16", (6000, 50, 192, 200, 8, 6), 3.0, 0.03, 0.1),
    "move_student_t_bf16_p60": ("student_t", "bf16", (6000, 60, 192, 90, 8, 6), 3.0, 0.03, 0.1),
    "move_student_t_bf16_p101": ("student_t", "bf16", (6000, 101, 128, 200, 8, 4), 3.0, 0.03, 0.1),
    "move_student_t_bf16_p12": ("student_t", "bf16", (6000, 12, 256, 300, 11, 10), 3.0, 0.03, 0.1),
    "move_student_t_bf16_p12_n60000": (
        "student_t", "bf16", (60000, 12, 256, 300, 11, 10), 3.0, 0.01, 0.02),
    "move_student_t_bf16_p50_n120000": (
        "student_t", "bf16", (120000, 50, 128, 300, 11, 6), 3.0, 0.01, 0.02),
    "move_logistic_bf16_p20": ("logistic", "bf16", (6000, 20, 256, 300, 7, 10), 0.5, 0.05, 0.03),
    "move_logistic_f32_p13": ("logistic", "f32", (6000, 13, 256, 130, 7, 10), 0.5, 0.05, 0.03),
    "move_probit_f32_p13": ("probit", "f32", (6000, 13, 256, 130, 7, 10), 0.5, 0.05, 0.03),
    "move_poisson_bf16_p8": ("poisson", "bf16", (6000, 8, 256, 130, 7, 10), 0.5, 0.05, 0.03),
}


def S():
    import paper_1805_03317_gb300 as pkg
    return pkg


def _setup(case, theta_bar=None):
    family, x_dtype, (n, p, N, m, G, L), scale, spread, a = case
    kw = dict(x_scale=0.3) if family == "poisson" else {}
    wl = small_glm(family, n=n, p=p, N=N, m=m, G=G, L=L, x_dtype=x_dtype, seed=77,
                   theta_scale=scale, **kw)
    prob, ctx = make_pair(wl, theta_bar=theta_bar)
    rng = np.random.default_rng(6)
    th = state_round(prob.theta_bar + spread * rng.standard_normal((N, p)), x_dtype)
    u = rng.integers(0, n, size=(N, m)).astype(np.int64)
    return prob, ctx, torch.from_numpy(th).to(DEV), torch.from_numpy(u).to(DEV), a


def outputs(name, theta_bar=None):
    """{"theta_bar", "ell", "sigma2", "grad" or "theta"} of a case as float64 arrays."""
    prob, ctx, th, u, a = _setup((GRADS | MOVES)[name], theta_bar)
    if name in GRADS:
        grad, ell, s2 = S().loglik_grad(ctx, th, u, a)
        out = dict(grad=grad, ell=ell, sigma2=s2)
    else:
        S().smc_set_particles(ctx, th, u)
        S().smc_set_scalars(ctx, 20, 0.9 * a, 0.3, 0.0)
        S().smc_reweight(ctx)  # the mass matrix of this cloud
        S().smc_set_scalars(ctx, 20, a, 0.3, 0.0)
        S().smc_move(ctx, 1)
        ell, s2, _ = S().smc_get_cache(ctx)
        out = dict(theta=S().smc_get_particles(ctx)[0], ell=ell, sigma2=s2)
        assert torch.any(out["theta"] != th.to(out["theta"].dtype), dim=1).float().mean() > 0.3
    S().smc_free(ctx)
    return dict({k: v.cpu().double().numpy() for k, v in out.items()}, theta_bar=prob.theta_bar)


@pytest.mark.parametrize("name", [*GRADS, *MOVES])
def test_fp32_outputs_match_the_recorded_ones(name):
    with np.load(PINS) as z:
        ref = {k.split("/")[1]: z[k] for k in z.files if k.startswith(name + "/")}
    got = outputs(name, ref["theta_bar"])
    if name in MOVES:
        assert np.array_equal(got["theta"], ref["theta"])
    for k in set(ref) - {"theta", "theta_bar"}:
        assert np.linalg.norm(got[k] - ref[k]) <= 1e-6 * np.linalg.norm(ref[k]), k
