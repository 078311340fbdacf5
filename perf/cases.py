"""The calls that users of the subsampling-SMC library make, at the sizes they make them.

Every case goes through the package's public entry points (``smc_init``, ``loglik_grad``,
``SubsampledLoglik``, ``loglik_full``, ``smc_move``, ``smc_stage``, ``smc_batch_stage``). Sizes are
those of the seeded workloads in ``smc_workloads`` and of the tests: from the plain FP64 problem
(n = 10^4, p = 5, 256 particles) to the GAM (n = 10^7, p = 101, 16384 particles of 5000 rows).

A context, its data and the particles' indices are what a program holds between calls, so
``prepare`` makes them. Moves and stages start from a checkpointed cloud, restored by
``smc_set_particles`` and ``smc_set_scalars`` in every pass, so a pass does the same work each time.

Estimates of problems stored in 32 or 16 bits are formed from FP32 row terms; they are handed on
in the state type (float32), the type that the gradients and the particles of such problems have.
"""
import math

import numpy as np
import torch

import paper_1805_03317_gb300 as S

DEV = "cuda"
TYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


# ------------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # The smallest calls: the estimator and its gradient for the plain FP64 problem
        # (n = 10^4, p = 5, N = 256, m = 100); launches and latency count.
        dict(name="grad_logistic_f64", kind="grad", family="logistic", dtype="f64", design="iid",
             n=10_000, p=5, N=256, m=100, G=10, L=10, a=0.3),
        # The estimator on the whole cloud of the flagship logistic problem: what an outside
        # sampler or a cache refresh asks for.
        dict(name="grad_logistic_bf16", kind="grad", family="logistic", dtype="bf16", design="ar1",
             n=1_000_000, p=20, N=4096, m=1000, G=10, L=20, a=0.002),
        # Poisson counts, X far larger than the L2 cache: every row comes from device memory.
        dict(name="grad_poisson_bf16", kind="grad", family="poisson", dtype="bf16",
             design="iid0.1", n=5_000_000, p=50, N=8192, m=2000, G=20, L=20, a=0.001),
        # The largest: the additive model's shape (10 covariates in 10 B-splines each, and an
        # intercept), here for counts (a Gaussian response leaves the rows nothing but rounding).
        dict(name="grad_gam_bf16", kind="grad", family="poisson", dtype="bf16", design="spline",
             n=10_000_000, p=101, N=16384, m=5000, G=10, L=25, a=0.001),
        # The differentiable estimator, forward and backward, in a caller's own optimiser: the
        # paper's Student-t regression (50 correlated covariates, M = 280 particles), FP32 storage.
        dict(name="autograd_student_f32", kind="autograd", family="student_t", dtype="f32",
             design="equi", n=500_000, p=50, N=280, m=1250, G=100, L=20, a=0.01),
        # The comparison method: the exact log-likelihood and gradient over all rows.
        dict(name="full_logistic_bf16", kind="full", family="logistic", dtype="bf16", design="ar1",
             n=1_000_000, p=20, N=4096, m=1000, G=10, L=20, a=0.01),
        # Starting a run: packing X, the posterior mode by Newton's method, the control-variate
        # moments, the initial particles and their estimates.
        dict(name="init_logistic_bf16", kind="init", family="logistic", dtype="bf16", design="ar1",
             n=1_000_000, p=20, N=4096, m=1000, G=10, L=20),
        # One Markov move of the flagship run in the middle of the annealing.
        dict(name="move_logistic_bf16", kind="move", family="logistic", dtype="bf16",
             design="ar1", n=1_000_000, p=20, N=4096, m=1000, G=10, L=20, R=1, a=0.002),
        # The paper's Student-t run with subsampling: M = 280, m = 1250, 100 blocks, 50 covariates.
        dict(name="move_student_bf16", kind="move", family="student_t", dtype="bf16",
             design="equi", n=500_000, p=50, N=280, m=1250, G=100, L=20, R=1, a=0.02),
        # FP32 storage, an odd width and ragged blocks.
        dict(name="move_probit_f32", kind="move", family="probit", dtype="f32", design="iid",
             n=200_000, p=13, N=512, m=477, G=7, L=20, R=1, a=0.002),
        # A whole stage (temperature search, reweighting, mass matrix, resampling, a move) of the
        # conjugate problem of the flagship's shape with half its particles, as one replayed graph.
        dict(name="stage_gaussian_bf16", kind="stage", family="gaussian", dtype="bf16",
             design="iid", n=1_000_000, p=20, N=2048, m=1000, G=10, L=20, R=1, a=1e-4),
        # Many posteriors of uneven n and p stepped together (logistic and probit in turn), one
        # more stage after each has reached its posterior.
        dict(name="batch_uneven_bf16", kind="batch", dtype="bf16", design="iid", P=16,
             n_lo=10_000, n_hi=100_000, p_lo=5, p_hi=40, N=256, m_lo=100, m_hi=1000, G=10, L=20,
             R=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grad", "grad", "autograd", "full", "init", "move", "move", "stage",
                       "batch"])
    if kind == "batch":
        n_lo = _log_int(rng, 5_000, 20_000)
        return dict(kind="batch", dtype="bf16", design="iid", P=rng.randint(2, 16), n_lo=n_lo,
                    n_hi=n_lo * rng.randint(2, 8), p_lo=rng.randint(2, 8),
                    p_hi=rng.randint(9, 40), N=_log_int(rng, 64, 300), m_lo=rng.randint(50, 150),
                    m_hi=rng.randint(200, 1000), G=rng.randint(2, 12), L=rng.randint(4, 20), R=1)
    family = rng.choice(["logistic", "probit", "poisson", "gaussian", "student_t"])
    dtype = rng.choice(["bf16", "bf16", "f32", "f64"])
    p = _log_int(rng, 2, 101)
    design = "iid0.1" if family == "poisson" else rng.choice(["iid", "ar1"])
    case = dict(kind=kind, family=family, dtype=dtype, design=design,
                n=_log_int(rng, 10_000, 1_000_000), p=p, N=_log_int(rng, 64, 4096),
                m=_log_int(rng, 50, 2000), G=rng.randint(1, 25), L=rng.randint(3, 20))
    if kind == "full":
        case.update(dtype="bf16", p=_log_int(rng, 2, 64))
    if kind == "init":
        case.update(N=_log_int(rng, 64, 1024), m=_log_int(rng, 50, 500))
    if kind in ("move", "stage"):
        case.update(N=_log_int(rng, 64, 700), p=_log_int(rng, 2, 60), m=_log_int(rng, 50, 1250),
                    n=_log_int(rng, 10_000, 200_000), R=1)
    if kind == "stage":
        # a stage chooses ancestors by the weights: the responses whose estimates are exact
        case.update(family="gaussian", design="iid")
    if case["dtype"] == "f64":
        case.update(N=min(case["N"], 300), m=min(case["m"], 200), n=min(case["n"], 100_000),
                    p=min(case["p"], 30))
    # the middle of an annealing run: a posterior of 30 to 3000 rows' worth of information
    case["a"] = math.exp(rng.uniform(math.log(30.0), math.log(3000.0))) / case["n"]
    return case


# ------------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------------
SIGMA = {"gaussian": 0.5}
NU = 5.0


def _prior_var(case):
    return {"poisson": 0.1, "gaussian": 100.0 if case["design"] == "spline" else 10.0}.get(
        case["family"], 10.0)


def _splines(u):
    """Cubic B-spline basis (10 functions, 6 interior knots on [0, 1], clamped) of u [n]: [n, 10]."""
    t = [0.0] * 4 + [k / 7.0 for k in range(1, 7)] + [1.0] * 4
    B = [((u >= t[i]) & (u < t[i + 1])).float() if t[i] < t[i + 1] else torch.zeros_like(u)
         for i in range(13)]
    for d in range(1, 4):
        nxt = []
        for i in range(13 - d):
            v = torch.zeros_like(u)
            if t[i + d] > t[i]:
                v += (u - t[i]) / (t[i + d] - t[i]) * B[i]
            if t[i + d + 1] > t[i + 1]:
                v += (t[i + d + 1] - u) / (t[i + d + 1] - t[i + 1]) * B[i + 1]
            nxt.append(v)
        B = nxt
    return torch.stack(B, 1)


def _covariates(case, n, p, g):
    X = torch.empty(n, p, dtype=TYPES[case["dtype"]], device=DEV)
    f = torch.float64 if case["dtype"] == "f64" else torch.float32
    design = case["design"]
    for r0 in range(0, n, 1_000_000):  # row chunks: the working copy stays small
        k = min(1_000_000, n - r0)
        if design == "spline":
            cols = [torch.ones(k, 1, device=DEV)]
            cols += [_splines(torch.rand(k, generator=g, device=DEV)) for _ in range((p - 1) // 10)]
            X[r0:r0 + k] = torch.cat(cols, 1)[:, :p]
            continue
        Z = torch.randn(k, p, generator=g, device=DEV, dtype=f)
        if design == "equi":  # pairwise correlation 0.9
            Z = math.sqrt(0.9) * torch.randn(k, 1, generator=g, device=DEV, dtype=f) + \
                math.sqrt(0.1) * Z
        else:
            if design == "ar1":  # correlation 0.5 between neighbours
                for c in range(2, p):
                    Z[:, c] = 0.5 * Z[:, c - 1] + math.sqrt(0.75) * Z[:, c]
            if design == "iid0.1":
                Z *= 0.1
            Z[:, 0] = 1.0
        X[r0:r0 + k] = Z
    return X


def _theta_true(case, p, g):
    z = torch.randn(p, generator=g, device=DEV, dtype=torch.float64)
    if case.get("family") == "poisson":
        th = 0.2 * z
        th[0] = 1.0
    elif case.get("family") == "student_t":
        th = 10.0 * torch.rand(p, generator=g, device=DEV, dtype=torch.float64) - 5.0
    else:
        th = (0.3 if p <= 20 else 1.3 / math.sqrt(p)) * z
    return th.float().double()  # a centre that every storage type holds exactly


def _eta(X, th, chunk=1_000_000):
    return torch.cat([X[r:r + chunk].double() @ th for r in range(0, X.shape[0], chunk)])


def _response(family, eta, g):
    if family == "logistic":
        y = torch.rand(eta.shape, generator=g, device=DEV, dtype=torch.float64) < torch.sigmoid(eta)
    elif family == "probit":
        y = torch.randn(eta.shape, generator=g, device=DEV, dtype=torch.float64) < eta
    elif family == "poisson":
        y = torch.poisson(torch.exp(eta), generator=g)
    elif family == "gaussian":
        y = eta + SIGMA[family] * torch.randn(eta.shape, generator=g, device=DEV,
                                              dtype=torch.float64)
    else:
        z = torch.randn((1 + int(NU),) + eta.shape, generator=g, device=DEV, dtype=torch.float64)
        y = eta + z[0] / torch.sqrt((z[1:] ** 2).sum(0) / NU)
    return y


def _data(case, seed, family=None, n=None, p=None):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    n, p = n or case["n"], p or case["p"]
    family = family or case["family"]
    X = _covariates(case, n, p, g)
    th = _theta_true(dict(case, family=family), p, g)
    y = _response(family, _eta(X, th), g).to(
        torch.float64 if case["dtype"] == "f64" else torch.float32)
    return X, y, th, g


def _curvature(family, eta):
    """Expected -l'' of a row."""
    if family == "logistic":
        s = torch.sigmoid(eta)
        return s * (1 - s)
    if family == "probit":
        pdf = torch.exp(-0.5 * eta * eta) / math.sqrt(2 * math.pi)
        c = torch.special.ndtr(eta)
        return pdf * pdf / (c * (1 - c)).clamp_min(1e-12)
    if family == "poisson":
        return torch.exp(eta)
    if family == "gaussian":
        return torch.full_like(eta, 1.0 / SIGMA[family] ** 2)
    return torch.full_like(eta, (NU + 1.0) / (NU + 3.0))


def _cloud(case, X, th, g, family, N, a):
    """Particles of the tempered posterior at temperature a: N(th, (a n H + 1 / v)^-1)."""
    k = min(X.shape[0], 50_000)
    Xs = X[:k].double()
    H = Xs.T @ (_curvature(family, Xs @ th)[:, None] * Xs) * (a * X.shape[0] / k)
    H += torch.eye(X.shape[1], dtype=torch.float64, device=DEV) / _prior_var(
        dict(case, family=family))
    Linv = np.linalg.inv(np.linalg.cholesky(H.cpu().numpy()))  # H^-1 = Linv' Linv
    z = torch.randn(N, X.shape[1], generator=g, device=DEV, dtype=torch.float64)
    c = th + z @ torch.from_numpy(Linv).to(DEV)
    return c.to(torch.float64 if case["dtype"] == "f64" else torch.float32).contiguous()


def _init_args(case, seed, p, family):
    return dict(family=family, prior_mean=np.zeros(p),
                prior_var=np.full(p, _prior_var(dict(case, family=family))), N=case["N"],
                m=case["m"], G=min(case["G"], case["m"]), L=case["L"], seed=seed,
                noise_sigma=SIGMA.get(family, 1.0), dof=NU)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    X, y, th, g = _data(case, seed)
    kw = _init_args(case, seed, case["p"], case["family"])
    s = {"case": case, "kind": kind}
    if kind == "init":
        return dict(s, X=X, y=y, kw=kw)
    ctx = S.smc_init(X, y, theta_bar=th.cpu().numpy(), **kw)
    a = case["a"]
    s.update(ctx=ctx, a=a, theta=_cloud(case, X, th, g, case["family"], case["N"], a),
             u=torch.randint(0, case["n"], (case["N"], case["m"]), generator=g, device=DEV,
                             dtype=torch.int32))
    if kind == "autograd":
        s["w"] = torch.rand(case["N"], generator=g, device=DEV, dtype=torch.float64) / case["n"]
    if kind in ("move", "stage"):
        s["eps"] = 0.5 * case["p"] ** -0.25
        S.smc_set_particles(ctx, s["theta"], s["u"])
        S.smc_set_scalars(ctx, 20, 0.9 * a, s["eps"])
        S.smc_reweight(ctx)  # the mass matrix of this cloud
    return s


def _batch_sizes(case, q):
    """Problem q of the batch: family, n, p, m (spread over the case's ranges, log-uniform in n)."""
    f = (q * 0.6180339887) % 1.0
    h = (q * 0.7548776662 + 0.3) % 1.0
    n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** f))
    return ("logistic" if q % 2 == 0 else "probit", n,
            case["p_lo"] + int(h * (case["p_hi"] - case["p_lo"] + 1)),
            case["m_lo"] + int(f * (case["m_hi"] - case["m_lo"] + 1)))


def _prepare_batch(case, seed):
    probs, clouds = [], []
    for q in range(case["P"]):
        family, n, p, m = _batch_sizes(case, q)
        X, y, th, g = _data(case, seed * 1000 + q, family, n, p)
        clouds.append((_cloud(case, X, th, g, family, case["N"], 1.0),
                       torch.randint(0, n, (case["N"], m), generator=g, device=DEV,
                                     dtype=torch.int32)))
        probs.append(dict(X=X, y=y, **_init_args(dict(case, m=m), seed * 1000 + q, p, family)))
    return {"case": case, "kind": "batch", "b": S.smc_batch_init(probs), "clouds": clouds}


# ------------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------------
def _state(case, t):
    return t if case["dtype"] == "f64" else t.float()


def _particles(case, ctx):
    theta, u, W = S.smc_get_particles(ctx)
    ell, s2, _ = S.smc_get_cache(ctx)
    out = {"theta": theta, "u": u, "W": W, "ell": _state(case, ell)}
    if case.get("family") != "gaussian":  # (its sigma2 is zero but for rounding)
        out["sigma2"] = _state(case, s2)
    return out


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "grad":
        grad, ell, s2 = S.loglik_grad(s["ctx"], s["theta"], s["u"], s["a"])
        out = {"grad": grad, "ell": _state(case, ell)}
        if case["family"] != "gaussian":
            out["sigma2"] = _state(case, s2)
        return out
    if kind == "autograd":
        theta = s["theta"].clone().requires_grad_(True)
        ell, s2 = S.SubsampledLoglik.apply(theta, s["u"], s["ctx"])
        a = s["a"]
        loss = (s["w"] * (a * ell - 0.5 * a * a * s2)).sum()
        loss.backward()
        out = {"grad": theta.grad, "ell": _state(case, ell.detach())}
        if case["family"] != "gaussian":
            out["sigma2"] = _state(case, s2.detach())
        return out
    if kind == "full":
        grad, ell = S.loglik_full(s["ctx"], s["theta"], s["a"])
        return {"grad": grad, "ell": ell.float()}
    if kind == "init":
        kw = s["kw"]
        ctx = S.smc_init(s["X"], s["y"], **kw)
        theta_bar, A, _, C = S.smc_get_centre(ctx)
        out = _particles(case, ctx)
        S.smc_free(ctx)
        if case["dtype"] != "f64":  # the moments as the kernels hold them
            theta_bar, C = theta_bar.astype(np.float32), C.astype(np.float32)
        return dict(out, theta_bar=theta_bar, A=A, C=C)
    if kind == "move":
        S.smc_set_particles(s["ctx"], s["theta"], s["u"])
        S.smc_set_scalars(s["ctx"], 20, s["a"], s["eps"])
        S.smc_move(s["ctx"], case["R"])
        return _particles(case, s["ctx"])
    if kind == "stage":
        S.smc_set_particles(s["ctx"], s["theta"], s["u"])
        S.smc_set_scalars(s["ctx"], 20, s["a"], s["eps"])
        S.smc_stage(s["ctx"], case["R"])
        st = S.smc_get_status(s["ctx"])
        return dict(_particles(case, s["ctx"]), a=st["a"], log_z=st["log_z"])
    b = s["b"]
    for ctx, (theta, u) in zip(b.contexts, s["clouds"]):
        S.smc_set_particles(ctx, theta, u)
        S.smc_set_scalars(ctx, 20, 1.0, 0.5 * ctx.p ** -0.25)
    S.smc_batch_stage(b, case["R"])
    out = []
    for ctx in b.contexts:
        theta, u, _ = S.smc_get_particles(ctx)
        out.append({"theta": theta, "u": u})
    return out


# ------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------------
def _row_work(case, N, m, p, n, passes):
    """Rows through the estimator: each covariate row that is drawn comes in once (or all of X, if
    that is less), its index and response with it; 2p operations for the predictor, 4p for the two
    gradient sums and about 20 for the row's terms in each pass."""
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    state = 8 if case["dtype"] == "f64" else 4
    distinct = n * (1.0 - math.exp(-N * m / n))
    return (distinct * (p * size + state) + 4.0 * N * m + 2.0 * N * p * state + 16.0 * N,
            float(passes) * N * m * (6 * p + 20))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        byts = flops = 0.0
        for q in range(case["P"]):
            _, n, p, m = _batch_sizes(case, q)
            x, f = _row_work(case, case["N"], m, p, n, 1 + (case["L"] + 1) * case["R"])
            byts, flops = byts + x + 4.0 * case["N"] * m, flops + f
        return {"bytes": byts, "flops": flops}
    n, p, N, m = case["n"], case["p"], case["N"], case["m"]
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    if kind == "full":
        return {"bytes": n * (p * size + 4.0) + 8.0 * N * p + 8.0 * N,
                "flops": float(N) * n * (4 * p + 10)}
    if kind == "init":
        x, f = _row_work(case, N, m, p, n, 1)
        # Newton: about three passes over the rows (2p for the predictor, p^2 for the Hessian)
        return {"bytes": x + 2.0 * n * (p * size + 4.0), "flops": f + 3.0 * n * (p * p + 4 * p)}
    passes = {"grad": 1, "autograd": 1}.get(kind) or 1 + (case["L"] + 1) * case["R"]
    x, f = _row_work(case, N, m, p, n, passes)
    if kind in ("move", "stage"):
        x += 4.0 * N * m
    return {"bytes": x, "flops": f}


# ------------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------------
def _rows64(family, eta, y, want_l=True):
    """l, l', l'' of rows at eta from the densities (theta-free constants included)."""
    if family == "logistic":
        s = torch.sigmoid(eta)
        return y * eta - torch.nn.functional.softplus(eta, threshold=60), y - s, -s * (1 - s)
    if family == "probit":
        sg = 2 * y - 1
        z = sg * eta
        lp = torch.special.log_ndtr(z)
        lam = torch.exp(-0.5 * z * z - lp) / math.sqrt(2 * math.pi)
        return lp, sg * lam, -lam * (z + lam)
    if family == "poisson":
        mu = torch.exp(eta)
        return y * eta - mu - torch.lgamma(y + 1), y - mu, -mu
    if family == "gaussian":
        v = SIGMA[family] ** 2
        r = y - eta
        return -0.5 * math.log(2 * math.pi * v) - r * r / (2 * v), r / v, torch.full_like(r, -1 / v)
    r = y - eta
    q = NU + r * r
    c = math.lgamma((NU + 1) / 2) - math.lgamma(NU / 2) - 0.5 * math.log(math.pi * NU)
    return (c - 0.5 * (NU + 1) * torch.log1p(r * r / NU), (NU + 1) * r / q,
            (NU + 1) * (r * r - NU) / (q * q))


def exact(case, seed):
    """The estimator (Sec. 3.2 of the paper) and the full-data sums from their definitions."""
    kind = case["kind"]
    if kind not in ("grad", "autograd", "full"):
        return None
    X, y, th, g = _data(case, seed)
    family, n, p, N, m, a = (case[k] for k in ("family", "n", "p", "N", "m", "a"))
    theta = _cloud(case, X, th, g, family, N, a).double()
    u = torch.randint(0, n, (N, m), generator=g, device=DEV, dtype=torch.int32)
    w = torch.rand(N, generator=g, device=DEV, dtype=torch.float64) / n if kind == "autograd" \
        else None
    y = y.double()
    var = _prior_var(case)
    ell = torch.zeros(N, dtype=torch.float64, device=DEV)
    if kind == "full":
        grad = torch.zeros(N, p, dtype=torch.float64, device=DEV)
        for r0 in range(0, n, 20_000):
            Xc, yc = X[r0:r0 + 20_000].double(), y[r0:r0 + 20_000]
            l0, l1, _ = _rows64(family, theta @ Xc.T, yc[None, :])
            ell += l0.sum(1)
            grad += l1 @ Xc
        return {"grad": a * grad - theta / var, "ell": ell}
    A = 0.0
    B = torch.zeros(p, dtype=torch.float64, device=DEV)
    C = torch.zeros(p, p, dtype=torch.float64, device=DEV)
    for r0 in range(0, n, 500_000):
        Xc = X[r0:r0 + 500_000].double()
        l0, l1, l2 = _rows64(family, Xc @ th, y[r0:r0 + 500_000])
        A = A + l0.sum()
        B += Xc.T @ l1
        C += Xc.T @ (l2[:, None] * Xc)
    grad = torch.empty(N, p, dtype=torch.float64, device=DEV)
    s2 = torch.empty(N, dtype=torch.float64, device=DEV)
    step = max(1, 20_000_000 // (m * p))
    for i0 in range(0, N, step):
        t = theta[i0:i0 + step]
        idx = u[i0:i0 + step].long()
        Xu = X[idx].double()
        yu = y[idx]
        dl = t - th
        eb = Xu @ th
        D = torch.einsum("imp,ip->im", Xu, dl)
        l0, l1, _ = _rows64(family, eb + D, yu)
        b0, b1, b2 = _rows64(family, eb, yu)
        d = (l0 - b0) - b1 * D - 0.5 * b2 * D * D
        r = (l1 - b1) - b2 * D
        Cd = dl @ C
        ell[i0:i0 + step] = A + dl @ B + 0.5 * (dl * Cd).sum(1) + (n / m) * d.sum(1)
        dc = d - d.mean(1, keepdim=True)
        s2[i0:i0 + step] = (n / m) ** 2 * (dc * dc).sum(1)
        ge = B + Cd + (n / m) * torch.einsum("im,imp->ip", r, Xu)
        gs = 2 * (n / m) ** 2 * torch.einsum("im,imp->ip", dc * r, Xu)
        if kind == "grad":
            grad[i0:i0 + step] = a * ge - 0.5 * a * a * gs - t / var
        else:
            grad[i0:i0 + step] = w[i0:i0 + step, None] * (a * ge - 0.5 * a * a * gs)
    out = {"grad": grad, "ell": ell}
    if family != "gaussian":
        out["sigma2"] = s2
    return out
