"""C_ij beyond the fine tables' middle part: at 64 to 1,024 ranges and at 2^-15 to 2^-7 of one (their outer parts), on,
just below and just above the intervals' edges, and past both ends, against K_nu with forty digits.  Bound per entry as
elsewhere, 1e-14 + 1e-15 x relative (x = h / a).  And the time: domains of 200 ranges, where most pairs lie beyond 64 of
them, and of a fiftieth of one take no more than both evaluations' operations over one's, and pairs past 1,024 ranges
no more than those."""
import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


def _places():
    far = np.concatenate([2.0 ** e * (1 + np.arange(8) / 8.0) for e in range(6, 11)])
    near = np.sqrt(np.concatenate([2.0 ** e * (1 + np.arange(0, 8, 3) / 8.0) for e in range(-32, -13)]))
    e = np.concatenate([far, near])
    return np.concatenate([e, np.nextafter(e, 0), np.nextafter(e, 1e9), np.geomspace(64, 1030, 70),
                           np.geomspace(2.0 ** -17, 2.0 ** -7, 70), [1e-9, 3000.0, 1e200]])


@pytest.mark.parametrize("nu", [(0.5,), (0.5, 1.0), (0.05, 2.9), (1.5, 2.5), (0.35, 1.75, 2.5), (0.4, 0.9, 1.3, 3.6), (5.9,), (12.3,),
                                (40.0,)])
def test_outer_parts(nu):
    import torch
    mp = pytest.importorskip("mpmath")
    import paper_2008_07437_gb300 as geo
    p, a = len(nu), 0.5   # a power of two: h / a is exact
    x = _places()
    if max(nu) > 4:   # (closer in, their evaluation's many upward steps take more than this bound)
        x = x[x >= 64]
    # (closed forms alone take the tables from 163,840 pairs on)
    h = a * np.concatenate([x, np.zeros(32768 - len(x))])
    reps = 6 if all(2 * v % 2 == 1 for v in nu) and p == 1 else 1
    theta = geo.Theta((1.0, 2.0, 0.5, 1.5)[:p], a, nu, tuple([0.2] * (p * (p - 1) // 2)) or None)
    l1, l2 = np.zeros((reps, 2)), np.stack([h, np.zeros_like(h)], axis=1)
    out = torch.zeros((p * len(h), p * reps), dtype=torch.float64, device="cuda")
    ctx = geo.geo_create(0)
    try:
        geo.geo_covgen(ctx, torch.as_tensor(l1, device="cuda"), theta, out, locs2=torch.as_tensor(l2, device="cuda"))
        got = out.cpu().numpy()[: p * len(x), :p].reshape(len(x), p, p)   # [place, j, i]
    finally:
        ctx.close()
    worst = 0.0
    with mp.workdps(40):
        for i in range(p):
            for j in range(i, p):
                n = (mp.mpf(nu[i]) + mp.mpf(nu[j])) / 2
                rho = (1 if i == j else mp.mpf(0.2)) * mp.sqrt(mp.mpf(nu[i]) * mp.mpf(nu[j])) / n
                c = rho * mp.sqrt(mp.mpf(theta.sigma2[i]) * mp.mpf(theta.sigma2[j])) / (2 ** (n - 1) * mp.gamma(n))
                for k, v in enumerate(x):
                    X = mp.mpf(float(v))
                    ref = c * X ** n * mp.besselk(n, X) if v < 2000 else mp.mpf(0)
                    for g in (got[k, j, i], got[k, i, j]):
                        if ref > 1e-280:
                            err = float(abs(mp.mpf(float(g)) - ref) / ref) / (1e-14 + 1e-15 * v)
                            worst = max(worst, err)
                        else:
                            assert abs(g) < 1e-280
    print("%s: worst error / bound %.3f" % (nu, worst))
    assert worst <= 1.0


@pytest.mark.parametrize("nu", [(0.5,), (0.5, 1.0, 1.5)])
def test_time_does_not_depend_on_the_range(nu):
    import torch
    import paper_2008_07437_gb300 as geo
    p, n = len(nu), 3000
    l = torch.as_tensor(inputs.jittered_grid(n, 5), dtype=torch.float64, device="cuda")
    out = torch.empty(p * n, p * n, dtype=torch.float64, device="cuda")
    ctx = geo.geo_create(0)

    def ms(a):
        th = geo.Theta((1.0,) * p, a, nu, (0.5, 0.3, 0.4) if p == 3 else None)
        best = 1e9
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            geo.geo_covgen(ctx, l, th, out)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    try:
        mid, far, near, past = ms(0.1), ms(0.005), ms(50.0), ms(0.0005)
    finally:
        ctx.close()
    print("%s: domain of 10 ranges %.3f ms, of 200 %.3f ms, of 1/50 %.3f ms, of 2,000 %.3f ms" % (nu, mid, far, near, past))
    # a warp with pairs on both sides does both evaluations: the middle one's 9 (p = 1) or 48 FP64 operations a pair
    # and at most 7 per C_ij, a root and an exponential (some 40) for the other
    lim = (9 + 8 + 40) / 9 if p == 1 else (48 + 6 * 8 + 40) / 48
    assert far < lim * mid and near < lim * mid and past < lim * mid
