"""A batch problem whose first tile has no positive pivot passes its remaining units on without working on them: sixty-four
of order 1,000 (two equal locations at the front) must take less than half the time of sixty-four that are positive
definite (whose cubic work it would otherwise do), report their row, and leave a good problem's bits alone."""
import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_failed_problems_are_cheap_and_reported():
    import torch
    import paper_2008_07437_gb300 as geo
    th = geo.Theta((1.0,), 0.09, (0.5,), None)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    good = [(dev(inputs.jittered_grid(1000, k)), dev(inputs.normals(k, 1000)), th) for k in range(64)]
    bad = []
    for l, z, _ in good:
        l2 = l.clone()
        l2[1] = l2[0]
        bad.append((l2, z, th))
    ctx = geo.geo_create(0)
    try:
        def ms(items):
            best = 1e9
            for _ in range(4):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                out = geo.geo_loglik_batch(ctx, items)
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
            return best, out
        t_good, (want, info) = ms(good)
        assert np.all(info == 0)
        t_bad, (ll, info) = ms(bad)
        assert np.all(info == 2) and np.all(np.isnan(ll))
        print("good %.2f ms, failed %.2f ms" % (t_good, t_bad))
        assert t_bad < 0.5 * t_good
        mix, info = geo.geo_loglik_batch(ctx, [x for p in zip(bad, good) for x in p])
        assert np.array_equal(mix[1::2], want) and np.all(info[0::2] == 2) and np.all(info[1::2] == 0)
    finally:
        ctx.close()
