"""Native FP64 factors the same way whatever nb, so tuning it runs one candidate: one warm-up and the samples."""
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_native_form_times_one_candidate():
    import torch
    import paper_2008_07437_gb300 as geo
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    n, th = 150, geo.Theta((1.0,), 0.09, (0.5,), None)
    l, z = dev(inputs.jittered_grid(n, 3)), dev(inputs.normals(4, n))
    ctx = geo.geo_create(0)
    try:
        def launches(f):
            geo.geo_profile_enable(ctx, True)
            out = f()
            k = sum(v["launches"] for v in geo.geo_profile_read(ctx).values())
            geo.geo_profile_enable(ctx, False)
            return k, out
        one, _ = launches(lambda: geo.geo_loglik(ctx, l, z, th, geo.opts(nb=128)))
        k, (nb, band, ms) = launches(lambda: geo.geo_autotune(ctx, l, z, th, [32, 128, 256, 512], [], samples=3))
        assert nb == 128 and ms > 0 and k == 4 * one     # 32 is no valid tile size
        k, (nb, band, ms) = launches(lambda: geo.geo_autotune(ctx, l, z, th, [128, 256], [], samples=3,
                                                              options=geo.opts(fp64_gemm=1)))
        assert nb in (128, 256) and k > 4 * one
    finally:
        ctx.close()
