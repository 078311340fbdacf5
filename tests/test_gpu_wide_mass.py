"""The mass matrix of FP32 states at its widest: up to 112 covariates the factor and its inverse are both
in shared memory, from 113 the inverse is built in global memory. Sigma, its factor and a move that
draws with the inverse, against the FP64 oracle; a batch with problems on both sides of the line."""
import numpy as np
import pytest
import torch

from gpu_common import make_pair
from oracle import oracle as O
from smc_workloads import small_glm
from test_gpu_parity import _moves_reduced_precision
from test_gpu_wide_rows import _batch_equals_singles

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def S():
    import paper_1805_03317_gb300 as pkg
    return pkg


@pytest.mark.parametrize("x_dtype", ["f32", "bf16"])
@pytest.mark.parametrize("p", [111, 112, 113, 126])
def test_wide_mass_matrix_matches_oracle(x_dtype, p):
    wl = small_glm("logistic", n=3000, p=p, N=400, m=40, G=4, L=3, x_dtype=x_dtype, seed=51)
    prob, ctx = make_pair(wl)
    S().smc_reweight(ctx)
    th, _, W = (v.cpu().double().numpy() for v in S().smc_get_particles(ctx))
    Sg, Lg = S().smc_get_mass(ctx)
    S().smc_free(ctx)
    _, Sig, Lc, _ = O.moments(W, th)
    np.testing.assert_allclose(Sg, Sig, rtol=1e-9, atol=1e-12)
    # backward error of a Cholesky factor: (p + 1) eps |L| |L'|, a few 1e-14 of Sigma's scale
    np.testing.assert_allclose(Lg @ Lg.T, Sig, rtol=0, atol=1e-12 * np.abs(Sig).max())
    assert np.allclose(Lg, np.tril(Lg))


@pytest.mark.parametrize("x_dtype", ["f32", "bf16"])
@pytest.mark.parametrize("p", [112, 113, 126])
def test_wide_moves_match_oracle(x_dtype, p):
    wl = small_glm("logistic", n=5000, p=p, N=256, m=90, G=6, L=4, x_dtype=x_dtype, seed=11)
    _moves_reduced_precision(wl, x_dtype, 1)


def test_batch_on_both_sides_of_the_line_equals_single_problems():
    _batch_equals_singles([("logistic", 112, 60, 3), ("student_t", 120, 50, 2),
                           ("probit", 7, 40, 2)], [1, 1], N=200)
