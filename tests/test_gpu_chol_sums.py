"""How the native factorisation sums a tile's products.  The residual (L L' - Sigma)_ii of a row i is what its roundings
add up to, and is formed here exactly.  With sums of 64 columns a diagonal entry of 1 is rounded some 62 times for the
blocks before its own at N = 4,000, up to 64 times within it, and the sums themselves up to 64 times at the size of the
one that carries most: about 180 roundings of standard deviation 0.29 u (u = 2^-53) at the most, 3.9 u; column by column
4,000 roundings come to 18 u.  The bound of 8 u on the rms lies between.  Also large orders against plain products and
triangular solves, past 8,192 columns and on and off a tile's edge."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def test_diagonal_residuals_are_those_of_short_sums():
    import paper_2008_07437_gb300 as geo
    n, th = 4000, geo.Theta((1.0,), 0.09, (0.5,), None)
    ctx = geo.geo_create(0)
    try:
        _, fac = geo.geo_loglik(ctx, dev(inputs.jittered_grid(n, 11)), dev(np.zeros(n)), th, geo.opts(), keep=True)
        res = []
        for i in range(3000, n, 20):
            row = geo.geo_factor_read(fac, 0, i, i + 1, 0, i + 1)[0]
            res.append(float(sum(Fraction(v) * Fraction(v) for v in row.tolist()) - 1))
    finally:
        ctx.close()
    rms = np.sqrt(np.mean(np.square(res))) / U
    print("rms residual %.2f u" % rms)
    assert rms <= 8.0


@pytest.mark.parametrize("n", [8192, 8225, 9217])
def test_past_8192_columns(n):
    import torch
    import paper_2008_07437_gb300 as geo
    th = geo.Theta((1.0,), 0.05, (0.5,), None)
    pts = inputs.jittered_grid(n + 40, 13)
    locs, new, z = dev(pts[:n]), dev(pts[n:]), dev(inputs.normals(14, n))
    ctx = geo.geo_create(0)
    try:
        _, fac = geo.geo_loglik(ctx, locs, z, th, geo.opts(morton=0), keep=True)
        L, y = dev(geo.geo_factor_read(fac, 0, 0, n, 0, n)), dev(geo.geo_factor_read(fac, 1, 0, n))
        S = torch.empty(n, n, dtype=torch.float64, device="cuda")
        geo.geo_covgen(ctx, locs, th, S)
        g = 4 * (n + 1) * U
        assert bool(((L @ L.T - S).abs() <= g).all())
        assert bool(((L @ y - z).abs() <= g * (L.abs() @ y.abs())).all())
        var = torch.empty(40, dtype=torch.float64, device="cuda")
        geo.geo_predict_var(ctx, fac, new, var)
        c = torch.exp(-torch.cdist(locs, new, compute_mode="donot_use_mm_for_euclid_dist") / 0.05)
        ref = 1.0 - torch.linalg.solve_triangular(L, c, upper=False).square().sum(0)
        assert bool(((var - ref).abs() <= 1e-10 + 1e-8 * ref.abs()).all())
    finally:
        ctx.close()
