"""More extra rows than the progress words of one factorisation or solve launch hold (32 rows to a word, 32,768 words):
rows do not depend on one another, so every result equals that of a call with fewer places, and the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2008_07437_gb300 as geo
    c = geo.geo_create(0)
    yield c
    c.close()


def dev(a):
    import torch
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def test_variances_at_more_places_than_words(ctx):
    import torch
    import paper_2008_07437_gb300 as geo
    th, n, m = geo.Theta((1.3,), 0.09, (0.8,), None), 33, 32 * 32768 + 65
    locs, new = inputs.jittered_grid(n, 3), np.random.default_rng(4).random((m, 2))
    _, fac = geo.geo_loglik(ctx, dev(locs), dev(np.zeros(n)), th, geo.opts(nb=128), keep=True)
    dn = dev(new)
    out = torch.empty(m, dtype=torch.float64, device="cuda")
    geo.geo_predict_var(ctx, fac, dn, out)
    for a, b in ((0, 1000), (m // 2, m // 2 + 1000), (m - 1000, m)):
        part = torch.empty(b - a, dtype=torch.float64, device="cuda")
        geo.geo_predict_var(ctx, fac, dn[a:b].clone(), part)
        assert bool((part == out[a:b]).all())
        ref = oracle.predict_var(oracle.Theta([1.3], 0.09, [0.8], np.eye(1)), locs, new[a:b])
        assert np.all(np.abs(part.cpu().numpy() - ref) <= 1e-10 + 1e-8 * np.abs(ref))
    fac.free()


def test_mloe_at_more_places_than_words(ctx):
    import paper_2008_07437_gb300 as geo
    t, a = geo.Theta((1.0,), 0.09, (0.5,), None), geo.Theta((1.0,), 0.07, (0.7,), None)
    n, m = 33, 16 * 32768 + 65          # two rows a place
    locs, new = inputs.jittered_grid(n, 3), np.random.default_rng(5).random((m, 2))
    mloe, mmom, loe, mom = geo.geo_mloe_mmom(ctx, dev(locs), dev(new), t, a)
    assert mloe == pytest.approx(loe.mean(), rel=1e-10) and mmom == pytest.approx(mom.mean(), rel=1e-10)
    for i in (0, m // 2, m - 500):
        _, _, l, o = geo.geo_mloe_mmom(ctx, dev(locs), dev(new[i : i + 500]), t, a)
        np.testing.assert_array_equal(l, loe[i : i + 500])
        np.testing.assert_array_equal(o, mom[i : i + 500])
