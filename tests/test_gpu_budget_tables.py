"""The covariance tables that only save time make room for what a call needs: with an HBM budget that holds the matrix,
the locations, the K_nu tables and the small vectors, and 4 KB more, every call runs as without a budget (within the two
evaluations' difference, far inside 1e-10 of the oracle)."""
import numpy as np
import pytest

import oracle
from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu

TAB = 10 * (12 * 24 + 4 * 24)   # doubles of a theta's K_nu tables
N, n = 800, 400
MATRIX = 8 * 832 * N            # leading dimension: N + 1 rows rounded up to 32


@pytest.fixture(scope="module")
def problem():
    th = oracle.Theta([1.0, 1.0], 0.09, [0.5, 1.0], np.array([[1.0, 0.5], [0.5, 1.0]]))
    pts = inputs.jittered_grid(n + 30, 21)
    z = oracle.simulate(th, pts[:n], inputs.normals(22, N))
    return pts[:n], pts[n:], z, oracle.loglik(th, pts[:n], z).loglik, oracle.predict(th, pts[:n], z, pts[n:])


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _theta():
    import paper_2008_07437_gb300 as geo
    return geo.Theta((1.0, 1.0), 0.09, (0.5, 1.0), 0.5)


def test_likelihood_and_predictions(problem):
    import torch
    import paper_2008_07437_gb300 as geo
    locs, new, z, ll, pred = problem
    ctx = geo.geo_create(0, MATRIX + 8 * (2 * n + TAB) + 2 * 4 * n + 8 * N + 4096)
    try:
        got, fac = geo.geo_loglik(ctx, dev(locs), dev(z), _theta(), geo.opts(), keep=True)
        assert got == pytest.approx(ll, rel=1e-10)
        zhat = torch.empty(60, dtype=torch.float64, device="cuda")
        geo.geo_predict(ctx, fac, dev(new), zhat)
        assert np.linalg.norm(zhat.cpu().numpy() - pred) <= 1e-8 * np.linalg.norm(pred)
        fac.free()
        assert geo.geo_loglik(ctx, dev(locs), dev(z), _theta(), geo.opts())[0] == got   # nothing leaked
    finally:
        ctx.close()


def test_tables_go_when_a_later_buffer_needs_the_room(problem):
    # room for the tables beside the matrix, but not beside the digit slices of the emulated form, which come after
    import paper_2008_07437_gb300 as geo
    locs, _, z, ll, _ = problem
    o = geo.opts(nb=128, fp64_gemm=1)
    # the slices' bytes: 8 digits of 2 bytes for 929 and 128 rows of 128 columns, and 64 columns for 128 rows, W, and
    # the exponents with their padding (under 16 KB)
    slices = 16 * 128 * (929 + 128) + 16 * 64 * 128 + 8 * 128 * 128 + 16384
    ctx = geo.geo_create(0, MATRIX + 8 * (2 * n + TAB) + 2 * 4 * n + slices + 4096)
    try:
        assert geo.geo_loglik(ctx, dev(locs), dev(z), _theta(), o)[0] == pytest.approx(ll, rel=1e-10)
    finally:
        ctx.close()


def test_batch(problem):
    import paper_2008_07437_gb300 as geo
    locs, _, z, ll, _ = problem
    ctx = geo.geo_create(0, MATRIX + 8 * TAB + 4096)
    try:
        got, info = geo.geo_loglik_batch(ctx, [(dev(locs), dev(z), _theta())])
        assert info[0] == 0 and got[0] == pytest.approx(ll, rel=1e-10)
    finally:
        ctx.close()
