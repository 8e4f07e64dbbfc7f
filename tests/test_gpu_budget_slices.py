"""The emulated products' workspace holds S digits of two bytes per operand entry and no padding to a multiple of four
slices: a budget of that (and the rows' exponents) must do, for slice counts with full and with ragged groups, K in one
chunk and in several, and the product must agree with FP64 to the form's own bound, (S + 2) 2^-(7 S) K max|a| max|b| per
entry plus K u |a||b| for the reference's sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("m,n,k", [(2048, 1024, 512), (300, 129, 1000), (128, 128, 16), (1, 5, 33)])
def test_workspace_is_s_slices(S, m, n, k):
    import torch
    import paper_2008_07437_gb300 as geo
    Kp, nchunk = (k + 31) // 32 * 32, -(-k // (4096 // S // 32 * 32))
    slices = lambda r: S * r * Kp * 2 + 4 * r * nchunk + 8 * ((r + 31) // 32) * nchunk + 768
    g = torch.Generator(device="cuda").manual_seed(S * 1000 + k)
    A, B, C = (torch.randn(c, r, generator=g, dtype=torch.float64, device="cuda").t() for r, c in ((m, k), (n, k), (m, n)))
    ref = C - A @ B.t()
    a, b = float(A.abs().max()), float(B.abs().max())
    ctx = geo.geo_create(0, slices(m) + slices(n) + 1024)
    try:
        geo.geo_gemm_f64e(ctx, A, B, C, slices=S)
    finally:
        ctx.close()
    # row maxima are within a power of two of what scales the digits
    bound = 4 * (S + 2) * 2.0 ** (-7 * S) * 4 * k * a * b + 2 * k * 2.0 ** -53 * k * a * b
    assert float((C - ref).abs().max()) <= bound
