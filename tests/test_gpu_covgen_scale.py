"""Covariances of variances at the ends of the double range: C(s2) = s2 C(1), to the two evaluations' bound of 1e-14 +
1e-15 x relative (x = h / a) each, where s2 C is a normal number; through geo_covgen with enough pairs for the fine
tables, and in a cross-covariance whose coefficient is tiny while the variances are not."""
import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


def _cov(s2, nu, beta, l):
    import torch
    import paper_2008_07437_gb300 as geo
    p, n = len(nu), len(l)
    out = torch.empty(p * n, p * n, dtype=torch.float64, device="cuda")
    ctx = geo.geo_create(0)
    try:
        geo.geo_covgen(ctx, torch.as_tensor(l, device="cuda"), geo.Theta((s2,) * p, 0.05, nu, beta), out)
        return out.cpu().numpy()
    finally:
        ctx.close()


@pytest.mark.parametrize("nu", [(0.8,), (0.5,)])
@pytest.mark.parametrize("e", [-864, -1000, 996])
def test_variance(e, nu):
    l = inputs.jittered_grid(450, 4)
    one, far = _cov(1.0, nu, None, l), _cov(2.0 ** e, nu, None, l)
    x = np.hypot(*(l[:, None, :] - l[None, :, :]).transpose(2, 0, 1)) / 0.05
    want = np.ldexp(one, e)
    live = want > 2.0 ** -1021
    assert live.mean() > 0.9 if e > -1000 else live.any()
    assert np.all((np.abs(far - want) <= 2 * (1e-14 + 1e-15 * x) * want)[live])


def test_cross_coefficient():
    l = inputs.jittered_grid(300, 4)
    one, far = _cov(1.0, (0.5, 1.0), 0.5, l), _cov(1.0, (0.5, 1.0), 0.5 * 2.0 ** -870, l)
    x = np.hypot(*(l[:, None, :] - l[None, :, :]).transpose(2, 0, 1)) / 0.05
    want = np.ldexp(one[0::2, 1::2], -870)
    live = want > 2.0 ** -1021
    assert np.all((np.abs(far[0::2, 1::2] - want) <= 2 * (1e-14 + 1e-15 * x) * want)[live])
    assert np.all(np.abs(far[0::2, 0::2] - one[0::2, 0::2]) <= 2 * (1e-14 + 1e-15 * x) * one[0::2, 0::2])
