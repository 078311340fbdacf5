"""The resident trajectory kernels' row gather.

- The tiles for 41 to 64 covariates (hmc_kernel 26: 56 slots, 27: 64 slots; ldmatrix / mma.sync rows)
  against the FP64 oracle, at the edges of their 64-row groups, 8-column units and index chunks.
- CTAs that take several particles fetch the next particle's rows during the current one's acceptance
  test: a launch over all particles equals launches over slices small enough for one particle per
  CTA, bit for bit, and a problem's particles in a batch those of the problem alone."""
import numpy as np
import pytest
import torch

from gpu_common import make_pair, state_round
from smc_workloads import small_glm
from test_gpu_parity import _moves_reduced_precision, _wl

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def S():
    import paper_1805_03317_gb300 as pkg
    return pkg


@pytest.mark.parametrize("family", ["logistic", "poisson", "probit", "gaussian", "student_t"])
@pytest.mark.parametrize("p,hmc_kernel", [(41, 26), (48, 26), (56, 27), (57, 27), (64, 27)])
def test_wide_tiles_match_oracle(family, p, hmc_kernel):
    _moves_reduced_precision(_wl(family, "bf16", p=p, N=256, m=90, G=6), "bf16", hmc_kernel)


@pytest.mark.parametrize("m,G", [(31, 3), (32, 1), (33, 33), (64, 4), (65, 2), (129, 7), (1025, 9)])
def test_wide_tile_row_edges_match_oracle(m, G):
    """Partial 32-row halves and 64-row groups, one group more than the warps, more rows than the
    1024 indices staged at a time."""
    wl = _wl("student_t", "bf16", p=50, n=9000, N=256, m=m, G=G)
    _moves_reduced_precision(wl, "bf16", 26)


def test_wide_rows_are_resident_by_default_and_refused_by_narrow_tiles():
    wl = _wl("logistic", "bf16", p=50, N=64, m=90, G=6)
    _, a = make_pair(wl)
    _, b = make_pair(wl, hmc_kernel=26)
    for c in (a, b):
        S().smc_reweight(c)
        S().smc_move(c, 2)
    assert torch.equal(S().smc_get_particles(a)[0], S().smc_get_particles(b)[0])
    with pytest.raises(S()._abi.SmcError):
        make_pair(wl, hmc_kernel=11)  # 40 slots
    with pytest.raises(S()._abi.SmcError):
        make_pair(_wl("logistic", "bf16", p=57, N=64, m=90, G=6), hmc_kernel=26)


@pytest.mark.parametrize("x_dtype,p,m,L", [("bf16", 20, 200, 3), ("bf16", 5, 40, 2),
                                           ("f32", 13, 130, 3), ("f64", 4, 50, 2),
                                           ("bf16", 50, 70, 2), ("bf16", 50, 1100, 1)])
def test_several_particles_per_cta_equal_one(x_dtype, p, m, L):
    """3500 particles in one launch (several per CTA on any tile) against slices of 152."""
    N, step = 3500, 152
    wl = small_glm("logistic", n=8000, p=p, N=N, m=m, G=4, L=L, x_dtype=x_dtype, seed=31)
    rng = np.random.default_rng(8)
    prob, full = make_pair(wl)
    th = torch.from_numpy(state_round(prob.theta_bar + 0.05 * rng.standard_normal((N, p)),
                                      x_dtype)).to(DEV)
    u = torch.from_numpy(rng.integers(0, wl.n, size=(N, m))).to(DEV)

    def moved(ctx):
        S().smc_set_particles(ctx, th, u)
        S().smc_set_scalars(ctx, 2, 0.3, 0.4, 0.0)
        S().smc_reweight(ctx)
        S().smc_move(ctx, 1)
        out = S().smc_get_particles(ctx, u=False)[0], *S().smc_get_cache(ctx)
        S().smc_free(ctx)
        return out

    ref = moved(full)
    assert torch.any(ref[0] != th.to(ref[0].dtype), dim=1).float().mean() > 0.2
    for b in (0, 152 * 7, 152 * 23):
        n = min(step, N - b)
        _, c = make_pair(wl, theta_bar=prob.theta_bar, shard_base=b, shard_count=n)
        for x, y in zip(moved(c), ref):
            assert torch.equal(x[b:b + n], y[b:b + n])


def test_batch_with_wide_rows_matches_single_problems():
    """Batch groups of the wide tiles whose CTAs go from one problem's particles to the next one's."""
    wls = [small_glm(f, n=3000 + 500 * q, p=p, N=150 + 40 * q, m=60 + 21 * q, G=4, L=3,
                     x_dtype="bf16", seed=60 + q)
           for q, (f, p) in enumerate([("logistic", 44), ("probit", 51), ("student_t", 60),
                                       ("logistic", 56), ("gaussian", 7)])]
    from gpu_common import device_arrays
    dicts = []
    for w in wls:
        X, y = device_arrays(w)
        dicts.append(dict(X=X, y=y, family=w.family, prior_mean=w.prior_mean,
                          prior_var=w.prior_var, N=w.N, m=w.m, G=w.G, L=w.L, seed=w.seed,
                          noise_sigma=w.sigma, dof=w.dof))
    b = S().smc_batch_init(dicts)
    kernels = [S().smc_batch_hmc_kernel(b, q) for q in range(len(wls))]
    assert kernels[:4] == [26, 26, 27, 26]
    singles = [make_pair(w, tile_hint=S().smc_batch_tile(b), hmc_kernel=kernels[q],
                         theta_bar=S().smc_get_centre(S().smc_batch_context(b, q))[0])[1]
               for q, w in enumerate(wls)]
    for use_graph in (False, True):
        S().smc_batch_stage(b, 2, use_graph=use_graph)
        for c in singles:
            S().smc_reweight(c)
            S().smc_resample(c)
            S().smc_move(c, 2)
    for q, c in enumerate(singles):
        for x, y in zip(S().smc_get_particles(S().smc_batch_context(b, q)),
                        S().smc_get_particles(c)):
            assert torch.equal(x, y), q
        S().smc_free(c)
    S().smc_batch_free(b)
