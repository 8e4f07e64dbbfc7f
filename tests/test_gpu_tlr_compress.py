"""Compression of off-diagonal tiles (QR of the sketch, R of the projection, Jacobi) at the edges of its kernels: tile
and sketch sizes off the multiples of 8 and 16, the widest sketch that fits a cluster's shared memory, the forms
beyond it and beyond 256 columns.  Per tile of the first column: the rank within 1 of the exact SVD's at the accuracy,
and the 2-norm error within 4 times the accuracy (the dropped singular values and the sketch's share)."""
import numpy as np
import pytest

import oracle
from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,nb,tol,kmax", [
    (1, 97, 65, 1e-7, 20),        # a last tile of 32 rows, sketches of at most 36 columns
    (2, 300, 102, 1e-9, 75),      # sketches of 32, 64, 91
    (2, 450, 226, 1e-10, 200),    # up to 216 of 226
    (2, 1060, 1060, 1e-8, 200),   # rows times columns beyond a cluster's shared memory
    (2, 640, 320, 1e-11, 300),    # sketches of more than 256 columns
])
def test_first_column_ranks_and_errors(p, n, nb, tol, kmax):
    import torch
    import paper_2008_07437_gb300 as geo
    nu, beta = [(1.0,), (0.5, 1.0)][p - 1], [None, (0.5,)][p - 1]
    th = geo.Theta((1.0,) * p, 0.09, nu, beta)
    locs = inputs.jittered_grid(n, 61)
    N, T = p * n, (p * n + nb - 1) // nb
    S = oracle.covgen(oracle.Theta(list(th.sigma2), th.a, list(nu), th.beta_matrix()), locs[oracle.morton_order(locs)])
    ctx = geo.geo_create(0)
    try:
        _, fac = geo.geo_loglik(ctx, torch.as_tensor(locs, device="cuda"),
                                torch.as_tensor(inputs.normals(62, N), device="cuda"), th,
                                geo.opts(prec=geo.GEO_PREC_TLR, nb=nb, tlr_tol=tol, tlr_kmax=kmax), keep=True)
        D0 = geo.geo_tlr_tile(fac, 0, 0, "D")
        for i in range(1, T):
            tile = S[i * nb:min(N, (i + 1) * nb), :nb]
            want = int((np.linalg.svd(tile, compute_uv=False) > tol).sum())
            U, V = geo.geo_tlr_tile(fac, i, 0, "U"), geo.geo_tlr_tile(fac, i, 0, "V")
            assert np.linalg.norm(tile - U @ (D0 @ V).T, 2) <= 4 * tol, i
            assert U.shape[1] == nb or abs(U.shape[1] - want) <= 1, (i, U.shape[1], want)   # nb: stored dense
            assert U.shape[1] != nb or want > min(kmax, nb) - 8, (i, want)
    finally:
        ctx.close()
