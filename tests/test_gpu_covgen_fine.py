"""C_ij from the fine tables (taken from 32,768 location pairs on) over their whole range and past both ends, against
the oracle: the same bound per entry as the sweep without them, 1e-14 + 1e-15 x relative (x = h / a; a few roundings,
and x times that of the exponent's argument)."""
import numpy as np
import pytest

import oracle
from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


def _edges():
    # x = sqrt(u) on, just below and just above interval edges of the table, and its two ends
    u = np.concatenate([2.0 ** e * (1 + np.arange(0, 32, 5) / 32.0) for e in range(-15, 13)])
    x = np.sqrt(u)
    return np.concatenate([x, np.nextafter(x, 0), np.nextafter(x, 1e9), [0.0, 1e-6, 63.999999, 64.0, 100.0, 1100.0]])


@pytest.mark.parametrize("nu", [(0.5,), (0.5, 1.0), (0.05, 2.9), (0.35, 1.75, 2.5), (0.4, 0.9, 1.3, 3.6)])
def test_fine_tables_every_interval(nu):
    import torch
    import paper_2008_07437_gb300 as geo
    p, a = len(nu), 0.5   # a power of two: h / a is exact
    x = np.concatenate([_edges(), np.geomspace(1e-3, 80.0, 4000)])
    h = a * np.concatenate([x, np.zeros(32768 - len(x))])
    theta = geo.Theta((1.0, 2.0, 0.5, 1.5)[:p], a, nu, tuple([0.2] * (p * (p - 1) // 2)) or None)
    l1, l2 = np.zeros((1, 2)), np.stack([h, np.zeros_like(h)], axis=1)
    out = torch.zeros((p * len(h), p), dtype=torch.float64, device="cuda")
    ctx = geo.geo_create(0)
    try:
        geo.geo_covgen(ctx, torch.as_tensor(l1, device="cuda"), theta, out, locs2=torch.as_tensor(l2, device="cuda"))
        got = out.cpu().numpy()[: p * len(x)].T
    finally:
        ctx.close()
    ref = oracle.covgen(oracle.Theta(list(theta.sigma2), a, list(nu), theta.beta_matrix()), l1, l2[: len(x)])
    xx = np.repeat(x, p)[None, :]
    live = np.abs(ref) > 1e-280
    assert np.all(np.abs(got[~live]) < 1e-280)
    assert np.all((np.abs(got - ref) <= (1e-14 + 1e-15 * xx) * np.abs(ref))[live])


def test_symmetric_matrix_and_predictions_use_the_same_entries():
    # n = 300: Sigma from the fine tables through the factor, the predictor through its own kernel
    import torch
    import paper_2008_07437_gb300 as geo
    th = geo.Theta((1.0, 1.3, 0.7), 0.05, (0.5, 1.0, 1.5), (0.5, 0.3, 0.4))
    allp = inputs.jittered_grid(333, 9)
    locs, new = allp[:300], allp[300:]
    o = oracle.Theta(list(th.sigma2), th.a, list(th.nu), th.beta_matrix())
    Z = oracle.simulate(o, locs, inputs.normals(10, 900))
    ctx = geo.geo_create(0)
    try:
        ll, fac = geo.geo_loglik(ctx, torch.as_tensor(locs, device="cuda"), torch.as_tensor(Z, device="cuda"), th,
                                 geo.opts(nb=128), keep=True)
        zhat = torch.zeros(3 * len(new), dtype=torch.float64, device="cuda")
        geo.geo_predict(ctx, fac, torch.as_tensor(new, device="cuda"), zhat)
        got = zhat.cpu().numpy()
    finally:
        ctx.close()
    ref = oracle.loglik(o, locs, Z)
    assert abs(ll - ref.loglik) <= 1e-10 * abs(ref.loglik)
    rp = oracle.predict(o, locs, Z, new)
    assert np.linalg.norm(got - rp) <= 1e-8 * np.linalg.norm(rp)
