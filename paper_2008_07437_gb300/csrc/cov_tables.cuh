// Construction of the covariance tables of a theta (matern.cuh) on the device (covgen.cu, batch.cu).
#pragma once

#include "geo_internal.cuh"

namespace {

// cos(pi j / 22), j = 0 .. 22, and the powers of t in the Chebyshev polynomials T_0 .. T_10.
__constant__ double c_cos22[23] = {
    1.0, 0.98982144188093273238, 0.95949297361449738989, 0.90963199535451837141, 0.84125353283118116886,
    0.75574957435425828377, 0.65486073394528506406, 0.54064081745559758211, 0.41541501300188642553,
    0.28173255684142969771, 0.14231483827328514044, 0.0, -0.14231483827328514044, -0.28173255684142969771,
    -0.41541501300188642553, -0.54064081745559758211, -0.65486073394528506406, -0.75574957435425828377,
    -0.84125353283118116886, -0.90963199535451837141, -0.95949297361449738989, -0.98982144188093273238, -1.0};
__constant__ double c_cheb_pow[GEO_FINE_NODES][GEO_FINE_NODES] = {
    {1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0},
    {0, 1, 0, 0, 0, 0, 0, 0, 0, 0, 0},
    {-1, 0, 2, 0, 0, 0, 0, 0, 0, 0, 0},
    {0, -3, 0, 4, 0, 0, 0, 0, 0, 0, 0},
    {1, 0, -8, 0, 8, 0, 0, 0, 0, 0, 0},
    {0, 5, 0, -20, 0, 16, 0, 0, 0, 0, 0},
    {-1, 0, 18, 0, -48, 0, 32, 0, 0, 0, 0},
    {0, -7, 0, 56, 0, -112, 0, 64, 0, 0, 0},
    {1, 0, -32, 0, 160, 0, -256, 0, 128, 0, 0},
    {0, 9, 0, -120, 0, 432, 0, -576, 0, 256, 0},
    {-1, 0, 50, 0, -400, 0, 1120, 0, -1280, 0, 512},
};

// Tables of a theta, one block of 128 threads of those of a pair i <= j.  by < FINE_BLOCKS: eight intervals of its fine
// table, sixteen threads to each, eleven of them at its Chebyshev nodes.  The transform works on differences to the
// middle node (they are small, so its rounding is too), and the Chebyshev coefficients, which fall by a factor
// of 60 or more each, go over to powers of t.  Beyond: four intervals of its K_nu table (cheb_f's, for distances
// outside the fine one), 32 threads to each, and the reciprocals.  Bound by the latency of one evaluation:
// 90 steps of four FP64 operations.
constexpr int FINE_BLOCKS = GEO_FINE_ALL / 8, COARSE_BLOCKS = GEO_CHEB_NI / 4;

__device__ __forceinline__ void fine_build_block(const CovParams &cp, double *tab, double *fine, int pair, int by) {
    __shared__ double val[8][16], cf[8][16];
    __shared__ NodeTabs nt;
    constexpr int n = GEO_FINE_NODES;
    int i = 0, j = pair;
    while (j >= cp.p - i) j -= cp.p - i, ++i;
    const MaternConst &c = cp.m[i * cp.p + i + j];
    const bool coarse = by >= FINE_BLOCKS;
    if (coarse ? (!tab || c.kind != 0 || c.toff < 0) : !fine) return;
    if (c.kind == 0) node_tabs(nt, c, threadIdx.x, 128);
    __syncthreads();
    if (coarse) {
        const int w = threadIdx.x / 32, t = threadIdx.x % 32, iv = (by - FINE_BLOCKS) * 4 + w;
        double *T = tab + c.toff, *hv = &val[2 * w][0];
        const double lo = ldexp(1.0, GEO_CHEB_K0 + iv);
        if (t < GEO_CHEB_N) {
            const double x = 1.5 * lo + 0.5 * lo * cospi((t + 0.5) / GEO_CHEB_N);
            bool scaled;
            const double v = xnu_besselk_node(x, c, nt, &scaled);
            hv[t] = scaled ? v : exp(x) * v;
        }
        __syncwarp();
        if (t < GEO_CHEB_N) {
            const double h0 = hv[GEO_CHEB_N / 2];
            double s = 0.0;
            for (int m = 0; m < GEO_CHEB_N; ++m) s = fma(hv[m] - h0, cospi(t * (m + 0.5) / GEO_CHEB_N), s);
            T[iv * GEO_CHEB_N + t] = fma(s, (t == 0 ? 1.0 : 2.0) / GEO_CHEB_N, t == 0 ? h0 : 0.0);
            if (iv == 0)
                for (int q = 0; q < 4; ++q) T[GEO_CHEB_NI * GEO_CHEB_N + q * GEO_TEMME_K + t] = nt.inv[q][t];
        }
        return;
    }
    const int w = threadIdx.x / 16, k = threadIdx.x % 16, idx = by * 8 + w;
    auto cos22 = [](int q) {   // cos(pi q / 22)
        q %= 44;
        return q <= 22 ? c_cos22[q] : c_cos22[44 - q];
    };
    double mid, half;
    matern_fine_bounds(idx, &mid, &half);
    if (k < n) {
        const double at = fma(half, cos22(2 * k + 1), mid);
        const bool far = idx >= GEO_FINE_N && idx < GEO_FINE_N + GEO_FINE_FAR;
        val[w][k] = far ? matern_far_node(at, c, nt) : matern_fine_node(at, c, nt);
    }
    __syncthreads();
    const double v0 = val[w][n / 2];   // t = 0
    double s = 0.0;
    if (k < n) {
        for (int q = 0; q < n; ++q) s = fma(val[w][q] - v0, cos22(k * (2 * q + 1)), s);
        cf[w][k] = s * ((k == 0 ? 1.0 : 2.0) / n);
    }
    __syncthreads();
    if (k >= n) return;
    s = 0.0;
    for (int m = n - 1; m >= 0; --m) s = fma(cf[w][m], c_cheb_pow[m][k], s);
    if (k == 0) s += v0;
    double *e = fine + c.foff + (long long)idx * GEO_FINE_STRIDE;
    // the floats relative to the value's own power of two: far out both are beyond FP32's range
    const int ex = v0 == 0.0 ? 0 : max(ilogb(v0), -800);
    if (k < 7)
        e[k] = s;
    else
        reinterpret_cast<float *>(e + 7)[k - 7] = (float)ldexp(s, -ex);
    if (k == 0) reinterpret_cast<unsigned *>(e + 9)[0] = (unsigned)((ex + 896) << 20);
}

}  // namespace
