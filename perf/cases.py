"""The calls whose time a user of this library pays for, as cases that can be
prepared, run and checked one by one.

* ``listed()``   the fixed cases, from the smallest likelihood to a step of the
  N = 40,000 workload;
* ``draw(rng)``  one more case out of the same ranges;
* ``prepare``    what a caller holds before the call: a context, device
  tensors and, for the calls that take one, a kept factor;
* ``run``        one call (or the few that belong together) through the public
  entry points;
* ``work``       the bytes and operations of a pass that no implementation can
  leave out;
* ``exact``      the same outputs from plain FP64 torch: K_nu by quadrature of
  its integral representation, dense Cholesky, triangular solves.

Inputs depend on the seed alone: locations on a jittered grid, observations as
a random-frequency draw of the Matern field itself (cosines whose frequencies
follow the field's spectral density), so that z' Sigma^-1 z and the predictions
have the size they have on data.
"""
import math

import numpy as np
import torch

import paper_2008_07437_gb300 as geo

DEV = "cuda:0"
F64 = torch.float64

# theta of the workloads: (sigma2, a, nu, upper triangle of beta)
THETAS = {
    "fig5": ((1.0, 1.0), 0.09, (0.5, 1.0), (0.5,)),
    "short": ((1.0, 1.0), 0.03, (0.5, 1.5), (0.5,)),
    "mixed": ((1.0, 1.0), 0.1, (0.5, 1.0), (0.7,)),
    "trivariate": ((1.0, 1.0, 1.0), 0.05, (0.5, 1.0, 1.5), (0.5, 0.3, 0.4)),
}


def listed():
    return [
        # one evaluation of the smallest workload (N = 800): what an optimiser of a small field calls
        # hundreds of times, all latency
        {"name": "loglik fp64 n400", "kind": "loglik", "form": "fp64", "theta": "fig5", "n": 400, "nb": 128, "m": 0},
        # an evaluation in native FP64 with the default tile (N = 8,002): the library's default form
        {"name": "loglik fp64 n4001", "kind": "loglik", "form": "fp64", "theta": "box", "n": 4001, "nb": 960, "m": 0},
        # a step of the N = 40,000 workload: likelihood with the factor kept, then cokriging of 2,000 places
        {"name": "loglik f64e8 n20000 m2000", "kind": "loglik", "form": "f64e8", "theta": "short", "n": 20000,
         "nb": 512, "m": 2000},
        # a request of the serving stream in the 5-slice form: any size, any theta of the box
        {"name": "loglik f64e5 n7001", "kind": "loglik", "form": "f64e5", "theta": "box", "n": 7001, "nb": 512, "m": 0},
        # the FP32 / FP16 form with refinement (FP32 band of 4 tiles)
        {"name": "loglik mixed n3001", "kind": "loglik", "form": "mixed", "theta": "mixed", "n": 3001, "nb": 256,
         "m": 0},
        # trivariate tile low rank at 1e-9, ten tile columns
        {"name": "loglik tlr n3000", "kind": "loglik", "form": "tlr", "theta": "trivariate", "n": 3000, "nb": 900,
         "m": 0},
        # many small uneven likelihoods in one call
        {"name": "batch 512", "kind": "batch", "count": 512, "n_lo": 50, "n_hi": 1000},
        # cokriging on a resident factor: a map of new places
        {"name": "predict n10000 m2000", "kind": "predict", "theta": "box", "n": 10000, "m": 2000},
        # cokriging on many small resident factors in one call
        {"name": "predict batch 128x100", "kind": "predict_batch", "count": 128, "n_lo": 50, "n_hi": 1000, "m": 100},
        # prediction variances beside the predictions
        {"name": "predict var n3001 m301", "kind": "predict_var", "theta": "fig5", "n": 3001, "m": 301, "nb": 512},
        # a cross-covariance matrix of its own (trivariate, ragged)
        {"name": "covgen p3 5003x2777", "kind": "covgen", "theta": "trivariate", "n1": 5003, "n2": 2777},
        # the FP64-class product as a standalone operation, a ragged trailing update
        {"name": "gemm f64e 8191x4099x512", "kind": "gemm", "m": 8191, "n": 4099, "k": 512, "slices": 8},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["fp64", "f64e8", "f64e5", "mixed", "tlr", "batch", "predict", "predict_batch", "predict_var",
                       "covgen", "gemm"])
    if what == "fp64":
        return {"kind": "loglik", "form": what, "theta": rng.choice(["fig5", "short", "box"]),
                "n": _log_int(rng, 100, 4500), "nb": rng.choice([128, 256, 512, 960]), "m": 0}
    if what == "f64e8":
        return {"kind": "loglik", "form": what, "theta": rng.choice(["fig5", "short"]), "n": _log_int(rng, 1000, 19000),
                "nb": rng.choice([256, 512]), "m": rng.choice([0, rng.randint(100, 2000)])}
    if what == "f64e5":
        return {"kind": "loglik", "form": what, "theta": "box", "n": _log_int(rng, 1000, 20000),
                "nb": rng.choice([256, 512, 768]), "m": 0}
    if what == "mixed":
        return {"kind": "loglik", "form": what, "theta": "mixed", "n": _log_int(rng, 1000, 8000),
                "nb": rng.choice([256, 512]), "m": 0}
    if what == "tlr":
        return {"kind": "loglik", "form": what, "theta": rng.choice(["fig5", "trivariate"]),
                "n": _log_int(rng, 800, 3000), "nb": rng.choice([240, 480, 900]), "m": 0}
    if what == "batch":
        return {"kind": "batch", "count": _log_int(rng, 16, 512), "n_lo": 50, "n_hi": _log_int(rng, 200, 1000)}
    if what == "predict":
        return {"kind": "predict", "theta": rng.choice(["fig5", "short", "box", "trivariate"]),
                "n": _log_int(rng, 500, 10000), "m": _log_int(rng, 100, 2000)}
    if what == "predict_batch":
        return {"kind": "predict_batch", "count": _log_int(rng, 8, 128), "n_lo": 50, "n_hi": _log_int(rng, 200, 1000),
                "m": _log_int(rng, 10, 400)}
    if what == "predict_var":
        return {"kind": "predict_var", "theta": rng.choice(["fig5", "short", "trivariate"]),
                "n": _log_int(rng, 300, 3000), "m": _log_int(rng, 10, 300), "nb": rng.choice([128, 512])}
    if what == "covgen":
        return {"kind": "covgen", "theta": rng.choice(["fig5", "short", "box", "trivariate"]),
                "n1": _log_int(rng, 100, 8000), "n2": _log_int(rng, 100, 3000)}
    return {"kind": "gemm", "m": _log_int(rng, 300, 8192), "n": _log_int(rng, 300, 8192), "k": _log_int(rng, 64, 1024),
            "slices": rng.choice([5, 6, 8])}


# ---- inputs, from the seed alone ------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _theta(name, rng):
    """A workload's theta, or one of the box an optimiser or a request stream moves in."""
    if name == "box":
        u = rng.uniform(size=6)
        return geo.Theta((0.5 + 1.5 * u[0], 0.5 + 1.5 * u[1]), 0.03 + 0.17 * u[2], (0.5 + u[3], 0.5 + u[4]),
                         (-0.7 + 1.4 * u[5],))
    sigma2, a, nu, beta = THETAS[name]
    return geo.Theta(sigma2, a, nu, beta)


def _places(n, g):
    """n locations, one per cell of a square grid, each jittered by up to 0.4 cell; cells in random order."""
    side = int(math.ceil(math.sqrt(n)))
    cell = torch.randperm(side * side, generator=g, device=DEV)[:n]
    jit = (2.0 * torch.rand(n, 2, generator=g, device=DEV, dtype=F64) - 1.0) * 0.4
    return ((torch.stack([cell % side, cell // side], 1).to(F64) + 0.5 + jit) / side).contiguous()


def _field(places, theta, g, rng, waves=512):
    """Observations z[p l + i]: per variable a sum of cosines with frequencies from the Matern spectral density
    (a bivariate t with 2 nu degrees of freedom), one common phase and direction set, mixed by beta's square root."""
    p = len(theta.sigma2)
    d = torch.randn(waves, 2, generator=g, device=DEV, dtype=F64)
    out = []
    for i in range(p):
        chi2 = torch.as_tensor(2.0 * rng.gamma(theta.nu[i], size=waves), device=DEV)
        ph = 2.0 * math.pi * torch.rand(waves, generator=g, device=DEV, dtype=F64)
        out.append(math.sqrt(2.0 / waves) * torch.cos(places @ (d / (theta.a * chi2.sqrt())[:, None]).T + ph).sum(1))
    low = torch.as_tensor(np.linalg.cholesky(theta.beta_matrix()), device=DEV)
    z = torch.stack(out, 1) @ low.T
    return (z * torch.as_tensor(theta.sigma2, device=DEV, dtype=F64).sqrt()).reshape(-1).contiguous()


def _observed(case, seed):
    """theta, locations, observations and new places of a case with one problem."""
    g, rng = _gen(seed), np.random.default_rng(int(seed))
    theta = _theta(case["theta"], rng)
    both = _places(case["n"] + case["m"], g)
    locs, new = both[: case["n"]].contiguous(), both[case["n"]:].contiguous()
    return theta, locs, _field(locs, theta, g, rng), new


def _many(case, seed):
    """(locations, observations, theta, new places) of each of a batch's problems."""
    g, rng = _gen(seed), np.random.default_rng(int(seed))
    out = []
    for _ in range(case["count"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        theta = _theta("box", rng)
        both = _places(n + case.get("m", 0), g)
        locs = both[:n].contiguous()
        out.append((locs, _field(locs, theta, g, rng, 64), theta, both[n:].contiguous()))
    return out


def _sizes(case):
    """Locations per problem of a batch, as expected: what work() counts."""
    return np.linspace(case["n_lo"], case["n_hi"], case["count"])


def _operands(case, seed):
    """A, B, C of a product, column-major: rows of very different sizes, as in a factor's panels."""
    g = _gen(seed)

    def one(r, c):
        x = torch.randn(c, r, generator=g, device=DEV, dtype=F64)
        return x * torch.exp2(-20.0 * torch.rand(r, generator=g, device=DEV, dtype=F64))

    k = case["k"]
    a, b = one(case["m"], k), one(case["n"], k)
    return a.t(), b.t(), torch.randn(case["n"], case["m"], generator=g, device=DEV, dtype=F64).t()


def _options(case):
    form, nb = case["form"], case["nb"]
    if form == "fp64":
        return geo.opts(nb=nb)
    if form == "f64e8":
        return geo.opts(nb=nb, fp64_gemm=1, oz_slices=8, oz_cut=1)
    if form == "f64e5":
        return geo.opts(nb=nb, fp64_gemm=1, oz_slices=5, oz_cut=1)
    if form == "mixed":
        return geo.opts(prec=geo.GEO_PREC_MIXED, nb=nb, band=4, refine_iters=2)
    return geo.opts(prec=geo.GEO_PREC_TLR, nb=nb, tlr_tol=1e-9, tlr_kmax=200)


# ---- state and pass ---------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "ctx": geo.geo_create(0)}
    if kind == "loglik":
        s["theta"], s["locs"], s["z"], s["new"] = _observed(case, seed)
        s["options"] = _options(case)
    elif kind == "batch":
        s["problems"] = [(locs, z, theta) for locs, z, theta, _ in _many(case, seed)]
    elif kind in ("predict", "predict_var"):
        theta, locs, z, s["new"] = _observed(case, seed)
        o = geo.opts(nb=512, fp64_gemm=1, oz_slices=8, oz_cut=1) if kind == "predict" else geo.opts(nb=case["nb"])
        _, s["factor"] = geo.geo_loglik(s["ctx"], locs, z, theta, o, keep=True)
        s["out"] = torch.empty(len(theta.sigma2) * case["m"], dtype=F64, device=DEV)
    elif kind == "predict_batch":
        s["entries"] = []
        for locs, z, theta, new in _many(case, seed):
            _, f = geo.geo_loglik(s["ctx"], locs, z, theta, geo.opts(nb=128), keep=True)
            s["entries"].append((f, new, torch.empty(2 * case["m"], dtype=F64, device=DEV)))
    elif kind == "covgen":
        g, rng = _gen(seed), np.random.default_rng(int(seed))
        s["theta"] = _theta(case["theta"], rng)
        s["locs1"], s["locs2"] = _places(case["n1"], g), _places(case["n2"], g)
        p = len(s["theta"].sigma2)
        s["out"] = torch.empty(p * case["n2"], p * case["n1"], dtype=F64, device=DEV)
    else:
        s["A"], s["B"], s["C"] = _operands(case, seed)
        s["slices"] = case["slices"]
    return s


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "loglik":
        if s["new"].shape[0] == 0:
            return np.float64(geo.geo_loglik(ctx, s["locs"], s["z"], s["theta"], s["options"])[0])
        ll, factor = geo.geo_loglik(ctx, s["locs"], s["z"], s["theta"], s["options"], keep=True)
        zhat = torch.empty(len(s["theta"].sigma2) * s["new"].shape[0], dtype=F64, device=DEV)
        geo.geo_predict(ctx, factor, s["new"], zhat)
        factor.free()
        return np.float64(ll), zhat
    if kind == "batch":
        return geo.geo_loglik_batch(ctx, s["problems"])
    if kind == "predict":
        return geo.geo_predict(ctx, s["factor"], s["new"], s["out"])
    if kind == "predict_var":
        return geo.geo_predict_var(ctx, s["factor"], s["new"], s["out"])
    if kind == "predict_batch":
        return torch.cat(geo.geo_predict_batch(ctx, s["entries"]))
    if kind == "covgen":
        return geo.geo_covgen(ctx, s["locs1"], s["theta"], s["out"], locs2=s["locs2"])
    return geo.geo_gemm_f64e(ctx, s["A"], s["B"], s["C"], slices=s["slices"])


# ---- what a pass cannot do without ---------------------------------------------------
COV_OPS = 40.0   # FP64 operations of one distinct C_ij at one distance (a short expansion, a distance)


def _p(case):
    return 2 if case.get("theta", "box") == "box" else len(THETAS[case["theta"]][0])


def work(case):
    kind, p = case["kind"], _p(case)
    pairs = p * (p + 1) / 2.0
    if kind == "loglik":
        n, m = case["n"], case["m"]
        N = p * n
        flops = N ** 3 / 3.0 + COV_OPS * pairs * n * n / 2.0 + 2.0 * N * N + (COV_OPS * pairs + 2.0 * p * p) * n * m
        return {"bytes": 8.0 * ((2 + p) * (n + m) + 1), "flops": flops}
    if kind == "batch":
        n = _sizes(case)
        return {"bytes": float(np.sum(8.0 * (4 * n + 1))), "flops": float(np.sum((2 * n) ** 3 / 3.0 + 60.0 * n * n))}
    if kind == "predict":
        n, m = case["n"], case["m"]
        return {"bytes": 8.0 * (2 + p) * (n + m), "flops": (COV_OPS * pairs + 2.0 * p * p) * n * m}
    if kind == "predict_batch":
        n = float(np.sum(_sizes(case)))
        return {"bytes": 8.0 * 4 * (n + case["count"] * case["m"]), "flops": (COV_OPS * 3 + 8.0) * n * case["m"]}
    if kind == "predict_var":
        n, m = case["n"], case["m"]
        N = p * n
        return {"bytes": 8.0 * (N * (N + 1) / 2.0 + 2 * (n + m) + p * m),
                "flops": float(N) * N * p * m + COV_OPS * pairs * n * m}
    if kind == "covgen":
        a, b = case["n1"], case["n2"]
        return {"bytes": 8.0 * (2 * (a + b) + p * p * a * b), "flops": COV_OPS * pairs * a * b}
    m, n, k = case["m"], case["n"], case["k"]
    return {"bytes": 8.0 * (m * k + n * k + 2.0 * m * n), "flops": 2.0 * m * n * k}


# ---- the same outputs in plain FP64 ----------------------------------------------------
STEP, LAST = 1.0 / 12.0, 17.0   # trapezoid rule of the integral below: error far below 1e-16 for x up to ~60


def _matern(x, theta):
    """{(i, j): C_ij} at the scaled distances x = h / a: x^nu K_nu(x), K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt."""
    p = len(theta.sigma2)
    beta = theta.beta_matrix()
    orders = {(i, j): 0.5 * (theta.nu[i] + theta.nu[j]) for i in range(p) for j in range(i, p)}
    x = torch.where(x > 0, x, torch.full_like(x, 1e-300))
    sums = {nu: torch.zeros_like(x) for nu in set(orders.values())}
    # exp(-x cosh t) has died out once x cosh t passes 750
    last = min(LAST, math.acosh(1.0 + 750.0 / max(float(x[x > 1e-200].min()) if (x > 1e-200).any() else 1.0, 1e-6)))
    for k in range(int(last / STEP) + 2):
        t = k * STEP
        e = torch.exp(-(math.cosh(t) - 1.0) * x) * (0.5 * STEP if k == 0 else STEP)
        for nu, acc in sums.items():
            acc.add_(e, alpha=math.cosh(nu * t))
    e = torch.exp(-x)
    out = {}
    for (i, j), nu in orders.items():
        rho = beta[i, j] * math.sqrt(theta.nu[i] * theta.nu[j]) / nu
        c0 = rho * math.sqrt(theta.sigma2[i] * theta.sigma2[j])
        v = sums[nu] * e * x.pow(nu) * (c0 / (2.0 ** (nu - 1.0) * math.gamma(nu)))
        out[i, j] = torch.where(x > 1e-200, v, torch.full_like(v, c0))
    return out


def _cov(s1, s2, theta):
    """(p n1) x (p n2) cross-covariance, location-major."""
    p = len(theta.sigma2)
    out = torch.empty(s1.shape[0], p, s2.shape[0], p, dtype=F64, device=DEV)
    rows = max(1, int(2.5e7 // max(1, s2.shape[0])))
    for a in range(0, s1.shape[0], rows):
        d = s1[a:a + rows, None, :] - s2[None, :, :]
        for (i, j), v in _matern(torch.sqrt((d * d).sum(2)) / theta.a, theta).items():
            out[a:a + rows, i, :, j] = v
            out[a:a + rows, j, :, i] = v
    return out.reshape(p * s1.shape[0], p * s2.shape[0])


def _factor(locs, theta):
    return torch.linalg.cholesky(_cov(locs, locs, theta))


def _loglik(low, z):
    y = torch.linalg.solve_triangular(low, z[:, None], upper=False)[:, 0]
    n = z.shape[0]
    return np.float64(-0.5 * n * math.log(2.0 * math.pi) - float(low.diagonal().log().sum()) - 0.5 * float((y * y).sum())), y


def _weights(low, y):
    return torch.linalg.solve_triangular(low.T, y[:, None], upper=True)[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("loglik", "predict", "predict_var"):
        theta, locs, z, new = _observed(case, seed)
        if z.shape[0] > 24000:
            return None   # the dense factorisation alone would take too long
        low = _factor(locs, theta)
        ll, y = _loglik(low, z)
        if kind == "loglik" and case["m"] == 0:
            return ll
        cross = _cov(locs, new, theta)
        if kind == "predict_var":
            v = torch.linalg.solve_triangular(low, cross, upper=False)
            c0 = torch.as_tensor(theta.sigma2, device=DEV, dtype=F64).repeat(case["m"])
            return c0 - (v * v).sum(0)
        zhat = cross.T @ _weights(low, y)
        return (ll, zhat) if kind == "loglik" else zhat
    if kind == "batch":
        return np.array([_loglik(_factor(locs, theta), z)[0] for locs, z, theta, _ in _many(case, seed)]), None
    if kind == "predict_batch":
        out = []
        for locs, z, theta, new in _many(case, seed):
            low = _factor(locs, theta)
            out.append(_cov(locs, new, theta).T @ _weights(low, _loglik(low, z)[1]))
        return torch.cat(out)
    if kind == "covgen":
        g, rng = _gen(seed), np.random.default_rng(int(seed))
        theta = _theta(case["theta"], rng)
        s1, s2 = _places(case["n1"], g), _places(case["n2"], g)
        return _cov(s2, s1, theta)
    A, B, C = _operands(case, seed)
    return C - A @ B.t()
