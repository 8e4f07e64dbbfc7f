"""geo_covgen below the number of pairs that pays for tables: one pair a thread, so that a call takes one evaluation's
time and not four in a row; every entry the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [(3.5,), (0.5, 1.5), (0.4, 0.9, 1.3), (0.4, 0.9, 1.3, 3.6)])
@pytest.mark.parametrize("n1,n2", [(1, 1), (65, 3), (63, 130), (181, 181)])
def test_entries_below_the_tables(nu, n1, n2):
    import torch
    import paper_2008_07437_gb300 as geo
    p = len(nu)
    th = geo.Theta((1.0, 2.0, 0.5, 1.5)[:p], 0.1, nu, tuple([0.2] * (p * (p - 1) // 2)) or None)
    l1, l2 = inputs.jittered_grid(n1, 1), inputs.jittered_grid(n2, 2)
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    out = torch.zeros((p * n2, p * n1), dtype=torch.float64, device="cuda")
    ctx = geo.geo_create(0)
    try:
        geo.geo_covgen(ctx, dev(l1), th, out, locs2=dev(l2))
    finally:
        ctx.close()
    ref = oracle.covgen(oracle.Theta(list(th.sigma2), 0.1, list(nu), th.beta_matrix()), l1, l2)
    got = out.cpu().numpy().T
    # the sweep's bound per entry, 1e-14 + 1e-15 x relative, and that of x = h / a rounded (h of a difference of
    # coordinates below 1: 3 u / a in x)
    x = np.repeat(np.repeat(np.hypot(*(l1[:, None, :] - l2[None, :, :]).transpose(2, 0, 1)) / 0.1, p, 0), p, 1)
    assert np.all(np.abs(got - ref) <= (1e-14 + 1e-15 * x + 3.4e-15) * np.abs(ref))


def test_time_of_few_pairs():
    # 64 places on a circle around 4 and around 16 copies of its centre: every pair costs the same evaluation (h / a =
    # 2.1), and more threads and not more pairs a thread are to do the second call's
    import torch
    import paper_2008_07437_gb300 as geo
    th = geo.Theta((1.0,), 0.1, (3.5,), None)
    phi = np.arange(64) * (2 * np.pi / 64)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    circle = dev(0.5 + 0.21 * np.stack([np.cos(phi), np.sin(phi)], axis=1))
    ctx = geo.geo_create(0)

    def ms(n2):
        centre, out = dev(np.full((n2, 2), 0.5)), torch.empty(n2, 64, dtype=torch.float64, device="cuda")
        best = 1e9
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            geo.geo_covgen(ctx, circle, th, out, locs2=centre)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    try:
        four, sixteen = ms(4), ms(16)
    finally:
        ctx.close()
    print("64 x 4 %.3f ms, 64 x 16 %.3f ms" % (four, sixteen))
    assert sixteen < 1.5 * four
