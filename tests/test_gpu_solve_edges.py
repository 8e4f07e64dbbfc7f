"""The triangular solves at the edges of their 64-row blocks and 32-row triangles, through the cokriging weights.
Backward alone: w = L^-T y from the kept factor, residual |L' w - y| <= g |L'| |w| with g = 4 (N + 1) u (the
componentwise bound of substitution, a factor of 4 for inverted triangles with one correction).  Forward and
backward: the mixed form's refined weights, |Sigma w - z| <= g |Sigma| |w| once its sweeps have converged.  Seen
through the predictor c' w that is |c'| |L^-T| g |L'| |w| (|c'| |Sigma^-1| g |Sigma| |w|), plus g |c'| |w| for the sum
over N and 2^-44 |c'| |w| for the entries of c (relative error below 256 u)."""
import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.mark.parametrize("mixed", [False, True], ids=["fp64", "mixed"])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 129, 320, 1000])
def test_weights_at_block_edges(n, mixed):
    import torch
    import paper_2008_07437_gb300 as geo
    th = geo.Theta((1.0,), 0.09, (0.5,))
    l, ln = inputs.jittered_grid(n, 31), inputs.jittered_grid(12, 32)
    z = inputs.normals(33, n)
    dev = lambda a: torch.as_tensor(a, device="cuda")
    ctx = geo.geo_create(0)
    try:
        kw = dict(prec=geo.GEO_PREC_MIXED, band=1, refine_iters=5) if mixed else {}
        _, fac = geo.geo_loglik(ctx, dev(l), dev(z), th, geo.opts(nb=128, morton=0, **kw), keep=True)
        zhat = torch.empty(12, dtype=torch.float64, device="cuda")
        geo.geo_predict(ctx, fac, dev(ln), zhat)
        h = lambda a, b: np.exp(-np.hypot(*(a[:, None, :] - b[None, :, :]).transpose(2, 0, 1)) / 0.09)
        c, g = h(ln, l), 4 * (n + 1) * U
        if mixed:
            M, rhs = h(l, l), z
        else:
            M = np.tril(geo.geo_factor_read(fac, 0, 0, n, 0, n)).T
            rhs = geo.geo_factor_read(fac, 1, 0, n)
        w = np.linalg.solve(M, rhs)
        for _ in range(3):   # to the last bits, by residuals in extended precision
            w = w + np.linalg.solve(M, (rhs - M.astype(np.longdouble) @ w).astype(float))
        bound = np.abs(c) @ (g * np.abs(np.linalg.inv(M)) @ (np.abs(M) @ np.abs(w)) + (g + 2.0 ** -44) * np.abs(w))
        assert (np.abs(zhat.cpu().numpy() - c @ w) <= bound).all()
    finally:
        ctx.close()
