"""Emulated products of few tiles: where a tile's columns are shared out over two or four CTAs, at ragged row and column
counts and at the number of tiles where the sharing ends, the result is bit for bit that of the same columns computed
as part of a product with many tiles (every entry has its own fixed order of operations)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [3, 5, 6, 8])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (128, 17, 40), (33, 65, 64), (100, 1000, 32), (129, 127, 900), (640, 900, 48),
                                   (1152, 1024, 32), (1300, 1024, 32)])
def test_same_bits_as_in_a_large_product(S, m, n, k):
    import torch
    import paper_2008_07437_gb300 as geo
    g = torch.Generator(device="cuda").manual_seed(m + 7 * n + k)
    rnd = lambda r, c: torch.randn(c, r, generator=g, dtype=torch.float64, device="cuda").t()
    A, B, C = rnd(m, k), rnd(n, k), rnd(m, n)
    # the same rows and columns at the front of 3,000 x 3,000: 576 tiles, no sharing
    A2, B2, C2 = rnd(3000, k), rnd(3000, k), rnd(3000, 3000)
    A2[:m], B2[:n], C2[:m, :n] = A, B, C
    ctx = geo.geo_create(0)
    try:
        geo.geo_gemm_f64e(ctx, A, B, C, slices=S)
        geo.geo_gemm_f64e(ctx, A2, B2, C2, slices=S)
    finally:
        ctx.close()
    assert bool((C == C2[:m, :n]).all())
