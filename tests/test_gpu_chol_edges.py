"""The one-launch Cholesky factorisation at the edges of its 32 x 32 tiles: L L' against Sigma and L y against Z,
entry by entry.  Bound: the backward error of Cholesky, |L L' - Sigma|_ij <= (N + 1) u sqrt(s_ii s_jj), with a
factor of 4 for scaling by rounded reciprocals (u = 2^-53); L y - z: (N + 1) u sum_k |L_ik| |y_k|, the same factor."""
import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def _check(p, n, **kw):
    import torch
    import paper_2008_07437_gb300 as geo
    nu, beta = [(0.5,), (0.5, 1.0)][p - 1], [None, (0.5,)][p - 1]
    th = geo.Theta((1.0,) * p, 0.09, nu, beta)
    N = p * n
    locs = torch.as_tensor(inputs.jittered_grid(n, 77), device="cuda")
    z = torch.as_tensor(inputs.normals(78, N), device="cuda")
    ctx = geo.geo_create(0)
    try:
        _, fac = geo.geo_loglik(ctx, locs, z, th, geo.opts(morton=0, **kw), keep=True)
        L = torch.as_tensor(geo.geo_factor_read(fac, 0, 0, N, 0, N), device="cuda")
        y = torch.as_tensor(geo.geo_factor_read(fac, 1, 0, N), device="cuda")
        S = torch.empty(N, N, dtype=torch.float64, device="cuda")
        geo.geo_covgen(ctx, locs, th, S)
        g = 4 * (N + 1) * U
        d = S.diagonal().sqrt()
        assert bool(((L @ L.T - S).abs() <= g * d[:, None] * d[None, :]).all())
        assert bool(((L @ y - z).abs() <= g * (L.abs() @ y.abs())).all())
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 97, 160, 1000, 4097])
def test_native_tile_edges(n):
    _check(1, n, nb=128)


@pytest.mark.parametrize("n", [64, 65, 96, 97, 129, 161, 400])
def test_emulated_tile_edges(n):
    # diagonal tiles of 128 with their inverse: last tiles of 2, 64, 66, ... columns
    _check(2, n, nb=128, fp64_gemm=1)


def test_indefinite_row_is_the_first():
    # duplicate location (Sigma singular): the failing row is a row of the second copy, in whichever tile it falls
    import torch
    import paper_2008_07437_gb300 as geo
    for n, dup in ((40, 35), (200, 130)):
        l = inputs.jittered_grid(n, 5)
        l[dup] = l[3]
        ctx = geo.geo_create(0)
        try:
            with pytest.raises(geo.GeoError) as e:
                geo.geo_loglik(ctx, torch.as_tensor(l, device="cuda"),
                               torch.as_tensor(inputs.normals(6, n), device="cuda"), geo.Theta((1.0,), 0.09, (0.5,)),
                               geo.opts(nb=64, morton=0))
            assert e.value.code == geo.GEO_ENOTSPD and e.value.info == dup + 1
        finally:
            ctx.close()
