"""geo_covgen inside a stream capture, on a context that has served no call before and after a smaller one: it allocates
and synchronises nothing.  The replayed entries are those of an ordinary call."""
import numpy as np
import pytest

from paper_2008_07437_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu,warm", [((0.5,), 0), ((0.5, 1.0), 0), ((0.5, 1.0), 20)])
def test_covgen_is_capturable(nu, warm):
    import torch
    import paper_2008_07437_gb300 as geo
    p, n = len(nu), 450
    th = geo.Theta((1.0,) * p, 0.1, nu, 0.5 if p == 2 else None)
    l = torch.as_tensor(inputs.jittered_grid(n, 1), dtype=torch.float64, device="cuda")
    out, ref = (torch.zeros(p * n, p * n, dtype=torch.float64, device="cuda") for _ in range(2))
    ctx, other = geo.geo_create(0), geo.geo_create(0)
    try:
        if warm:
            geo.geo_covgen(ctx, l[:warm].clone(), th, torch.empty(p * warm, p * warm, dtype=torch.float64, device="cuda"))
        geo.geo_covgen(other, l, th, ref)
        torch.cuda.synchronize()
        g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(g, stream=s):
            geo.geo_covgen(ctx, l, th, out, stream=s)
        g.replay()
        torch.cuda.synchronize()
        assert bool((out == ref).all())
    finally:
        ctx.close()
        other.close()
