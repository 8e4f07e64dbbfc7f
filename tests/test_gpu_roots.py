"""The factorisations' square roots and reciprocals (csrc/chol_tile.cuh) against sqrt() and division over all exponents
they are used for, and pivots outside those.  The root is correctly rounded and so is the reciprocal but for values within 2^-30
of the middle of two doubles: of 2^28 values at most a handful may differ, by one unit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2008_07437_gb300 import build, inputs

pytestmark = pytest.mark.gpu

SRC = r"""
#include "chol_tile.cuh"
__global__ void k(unsigned long long *out) {   // {roots that differ, reciprocals that differ, by more than one unit}
    unsigned long long n[3] = {0, 0, 0};
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 28); i += gridDim.x * blockDim.x) {
        // exponents in turn, mantissas by a multiplicative hash, some at the ends
        unsigned long long h = (i + 1ull) * 0x9E3779B97F4A7C15ull;
        h ^= h >> 29;
        h *= 0xBF58476D1CE4E5B9ull;
        unsigned long long m = (h ^ h >> 32) & 0xFFFFFFFFFFFFFull;
        if (i % 64 == 0) m &= 7;
        if (i % 64 == 1) m |= 0xFFFFFFFFFFFF8ull;
        const double d = __longlong_as_double((long long)((unsigned long long)(i / 64 % 2047) << 52 | m));
        if (!df_positive(d) || d < 0x1p-960 || d > 0x1p960) continue;
        double l, inv;
        df_root(d, &l, &inv);
        const double rl = sqrt(d), ri = 1.0 / rl;
        const long long dl = llabs(__double_as_longlong(l) - __double_as_longlong(rl));
        const long long di = llabs(__double_as_longlong(inv) - __double_as_longlong(ri));
        n[0] += dl != 0;
        n[1] += di != 0;
        n[2] += dl > 1 || di > 1;
    }
    for (int q = 0; q < 3; ++q) atomicAdd(out + q, n[q]);
}
extern "C" int run(unsigned long long *host) {
    unsigned long long *d;
    if (cudaMalloc(&d, 24) != cudaSuccess || cudaMemset(d, 0, 24) != cudaSuccess) return 1;
    k<<<152 * 4, 256>>>(d);
    const int rc = cudaMemcpy(host, d, 24, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(d);
    return rc;
}
"""


def test_roots_and_reciprocals_round_correctly(tmp_path):
    src, lib = tmp_path / "roots.cu", tmp_path / "roots.so"
    src.write_text(SRC)
    subprocess.run([build.NVCC, "-shared", "-o", str(lib), str(src)] + build._flags(False), check=True)
    out = (ctypes.c_ulonglong * 3)()
    assert ctypes.CDLL(str(lib)).run(out) == 0
    assert out[0] <= 4 and out[1] <= 4 and out[2] == 0, list(out)


@pytest.mark.parametrize("s2", [3e-308, 1e-290, 1e300])
def test_variances_at_the_ends_of_the_range(s2):
    # l(s2 Sigma, sqrt(s2) z) = l(Sigma, z) - N / 2 log s2; with s2 = 3e-308 pivots are subnormal, with 2^-50 of
    # their value left at the least (the smallest is 0.30 s2), far inside 1e-10 of l
    import torch
    import paper_2008_07437_gb300 as geo
    n = 150
    locs = inputs.jittered_grid(n, 5)
    z = oracle.simulate(oracle.Theta([1.0], 0.09, [0.5], np.eye(1)), locs, inputs.normals(6, n))
    ref = oracle.loglik(oracle.Theta([1.0], 0.09, [0.5], np.eye(1)), locs, z).loglik - 0.5 * n * np.log(s2)
    ctx = geo.geo_create(0)
    try:
        got, _ = geo.geo_loglik(ctx, torch.as_tensor(locs, device="cuda"), torch.as_tensor(z * np.sqrt(s2), device="cuda"),
                                geo.Theta((s2,), 0.09, (0.5,), None))
    finally:
        ctx.close()
    assert got == pytest.approx(ref, rel=1e-10)
