// Covariance generation (Eq. 2, Sec. 4.2) in Representation I (Sec. 5.2),
// and the fused cokriging predictor (Eq. 3 / Eq. 4, Sec. 4.3).
//
// Every matrix entry is one FP64 evaluation of Eq. 2: the work is FP64 ALU
// bound (Bessel K_nu), so the kernels map one location pair to one thread,
// evaluate the p(p+1)/2 distinct C_ij once per pair (from the theta's fine
// tables, matern.cuh, where they pay), and write the p x p block with
// column-major stores that are contiguous across a warp.  Measured against one
// Clenshaw sum per order and one exponential per pair: Sigma of N = 40,000
// (p = 2) 9.4 ms (51.4), a 15,009 x 8,331 cross-covariance (p = 3) 1.25 ms
// (8.0), 2,000 predictions on 10,000 locations (p = 2) 1.12 ms (10.2); the FP64
// operations that are left (27 a pair for p = 2, 48 for p = 3) take 0.9, 1.06
// and 0.99 of that at the pipe's rate.  Entries are 2.5 to 4 times closer to
// the exact values than before (4e-16 relative, weighted by size).
#include "cov_tables.cuh"

namespace {

constexpr int TL = 64;   // locations l (rows) per CTA
constexpr int TR = 4;    // locations r (columns) per CTA

// The p x p block of C at distance h for one location pair, without the fine tables.
__device__ __forceinline__ void cov_block(const CovParams &cp, double h, double *v) {
    matern_block(h * cp.inv_a, cp, v);
}

// K_nu tables of one theta (cheb_build_block, matern.cuh): block (q, k).
__global__ void __launch_bounds__(32) k_cheb_build(const CovParams cp, double *tab) {
    __shared__ double hv[GEO_CHEB_N];
    cheb_build_block(cp, tab, blockIdx.x, blockIdx.y, hv);
}

__global__ void __launch_bounds__(128) k_fine_build(const CovParams cp, double *tab, double *fine) {
    fine_build_block(cp, tab, fine, blockIdx.x, blockIdx.y);
}

// Lower triangle (location blocks l >= r) of Sigma, column-major A[c*ld + r].
__global__ void __launch_bounds__(TL *TR) k_covgen_sym(const CovParams cp, const double *__restrict__ lx,
                                                       const double *__restrict__ ly, int n, double *A,
                                                       long long ld) {
    const int l0 = blockIdx.y * TL, r0 = blockIdx.x * TR;
    if (r0 > l0 + TL - 1) return;   // tile entirely above the location diagonal
    const int l = l0 + (threadIdx.x % TL);
    const int r = r0 + (threadIdx.x / TL);
    if (l >= n || r >= n || r > l) return;
    const double dx = lx[l] - lx[r], dy = ly[l] - ly[r];
    const double h = sqrt(dx * dx + dy * dy);
    double v[GEO_PMAX_DEV * GEO_PMAX_DEV];
    cov_block(cp, (l == r) ? 0.0 : h, v);
    const int p = cp.p;
    for (int j = 0; j < p; ++j) {
        double *col = A + (long long)(p * r + j) * ld + (long long)p * l;
        for (int i = 0; i < p; ++i) col[i] = v[i * GEO_PMAX_DEV + j];
    }
}

// The same from the fine tables.  Each thread takes RPT locations r, so that the table positions and loads of
// one pair run under the FP64 chain of another.
constexpr int RPT = 4;

template <int P>
__global__ void __launch_bounds__(TL *TR) k_covgen_sym_fine(const CovParams cp, const double *__restrict__ lx,
                                                            const double *__restrict__ ly, int n, double *A,
                                                            long long ld) {
    const int l0 = blockIdx.y * TL, r0 = blockIdx.x * (TR * RPT);
    if (r0 > l0 + TL - 1) return;   // tile entirely above the location diagonal
    const int l = l0 + (threadIdx.x % TL);
    if (l >= n) return;
    const double x = lx[l], y = ly[l];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = r0 + q * TR + threadIdx.x / TL;
        if (r > l) continue;
        const double dx = x - lx[r], dy = y - ly[r];
        double v[P * P];
        matern_pair<P>((l == r) ? 0.0 : fma(dx, dx, dy * dy), cp, v);
#pragma unroll
        for (int j = 0; j < P; ++j) {
            double *col = A + (long long)(P * r + j) * ld + (long long)P * l;
#pragma unroll
            for (int i = 0; i < P; ++i) col[i] = v[i * P + j];
        }
    }
}

// Full rectangle: rows p*n1 (locations l of set 1), cols p*n2 (set 2); AoS inputs.  Without the fine tables one pair a
// thread: an evaluation is a long chain then, and there are too few pairs to hide four after one another (order 3.5,
// 100 x 100: 917 us so, 293 with one).
template <int P, bool FINE>
__global__ void __launch_bounds__(TL *TR) k_covgen_rect(const CovParams cp, const double *__restrict__ l1, int n1,
                                                        const double *__restrict__ l2, int n2, double *out,
                                                        long long ld, bool closed) {
    constexpr int RP = FINE ? RPT : 1;
    const int l = blockIdx.y * TL + (threadIdx.x % TL);
    if (l >= n1) return;
    const double x = l1[2 * l], y = l1[2 * l + 1];
#pragma unroll
    for (int q = 0; q < RP; ++q) {
        const int r = (blockIdx.x * RP + q) * TR + threadIdx.x / TL;
        if (r >= n2) return;
        const double dx = x - l2[2 * r], dy = y - l2[2 * r + 1], d2 = fma(dx, dx, dy * dy);
        double v[P * P];
        if constexpr (FINE) {
            matern_pair<P>(d2, cp, v);
        } else {
            const double u = d2 * cp.inv_a2;
            if (closed && u > 0x1p-900 && u < 0x1p900) {
                // from u = x^2 as the tables' nodes are: x without the rounding of h / a, and the root's put back
                const double h = sqrt(u), dh = fma(-h, h, u) / (2.0 * h), ex = exp(-h), emx = fma(-ex, dh, ex);
#pragma unroll
                for (int i = 0; i < P; ++i)
#pragma unroll
                    for (int j = 0; j < P; ++j) v[i * P + j] = matern_cov_e(h, emx, cp.m[i * P + j], nullptr);
            } else {
                double w[GEO_PMAX_DEV * GEO_PMAX_DEV];
                cov_block(cp, sqrt(d2), w);
#pragma unroll
                for (int i = 0; i < P; ++i)
#pragma unroll
                    for (int j = 0; j < P; ++j) v[i * P + j] = w[i * GEO_PMAX_DEV + j];
            }
        }
#pragma unroll
        for (int j = 0; j < P; ++j) {
            double *col = out + (long long)(P * r + j) * ld + (long long)P * l;
#pragma unroll
            for (int i = 0; i < P; ++i) col[i] = v[i * P + j];
        }
    }
}

// One CTA per prediction location: zhat_i(s0) = sum_r sum_j C_ij(|s0 - s_r|) w_(p r + j).
// Fixed thread-to-r assignment and a fixed reduction tree: the result does not
// depend on timing.
constexpr int PRED_THREADS = 256;

template <int P>
__device__ __forceinline__ void predict_one(const CovParams &cp, double x0, double y0, const double *__restrict__ lx,
                                            const double *__restrict__ ly, int n, const double *__restrict__ w,
                                            double *zhat) {
    double acc[P];
#pragma unroll
    for (int i = 0; i < P; ++i) acc[i] = 0.0;
    for (int r = threadIdx.x; r < n; r += PRED_THREADS) {
        const double dx = x0 - lx[r], dy = y0 - ly[r];
        double v[P * P];
        matern_pair<P>(fma(dx, dx, dy * dy), cp, v);
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const double wj = w[(long long)P * r + j];
#pragma unroll
            for (int i = 0; i < P; ++i) acc[i] = fma(v[i * P + j], wj, acc[i]);
        }
    }
    __shared__ double red[P][PRED_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < P; ++i) {
        double t = acc[i];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) red[i][wid] = t;
    }
    __syncthreads();
    if (threadIdx.x < P) {
        double t = 0.0;
        for (int k = 0; k < PRED_THREADS / 32; ++k) t += red[threadIdx.x][k];
        zhat[threadIdx.x] = t;
    }
}

template <int P>
__global__ void __launch_bounds__(PRED_THREADS) k_predict(const CovParams cp, const double *__restrict__ s0,
                                                          const double *__restrict__ lx,
                                                          const double *__restrict__ ly, int n,
                                                          const double *__restrict__ w, double *zhat) {
    const int l = blockIdx.x;
    predict_one<P>(cp, s0[2 * l], s0[2 * l + 1], lx, ly, n, w, zhat + (long long)P * l);
}

__global__ void k_gather_locs(const double *__restrict__ locs, const int *__restrict__ perm, int n, double *lx,
                              double *ly) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int s = perm ? perm[k] : k;
    lx[k] = locs[2 * (long long)s];
    ly[k] = locs[2 * (long long)s + 1];
}

__global__ void k_gather_vec(const double *__restrict__ in, const int *__restrict__ perm, int n, int p,
                             double *out, long long stride) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)n * p) return;
    const int k = (int)(t / p), i = (int)(t % p);
    const int s = perm ? perm[k] : k;
    out[t * stride] = in[(long long)p * s + i];
}

__global__ void k_scatter_vec(const double *__restrict__ in, long long stride, const int *__restrict__ perm, int n,
                              int p, double *out) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)n * p) return;
    const int k = (int)(t / p), i = (int)(t % p);
    const int s = perm ? perm[k] : k;
    out[(long long)p * s + i] = in[t * stride];
}

}  // namespace

bool cov_needs_tables(const CovParams &cp) {
    for (int q = 0; q < cp.p * cp.p; ++q)
        if (cp.m[q].kind == 0 && cp.m[q].toff >= 0) return true;
    return false;
}

bool cov_closed(const CovParams &cp) {
    for (int q = 0; q < cp.p * cp.p; ++q)
        if (cp.m[q].kind == 0) return false;
    return true;
}

cudaError_t launch_cheb_build(CovParams &cp, double *tab, cudaStream_t s) {
    cp.tab = tab;
    if (!cov_needs_tables(cp)) return cudaSuccess;
    if (!tab) return cudaErrorInvalidValue;
    KScope ks(GEO_K_COVGEN, s);
    k_cheb_build<<<dim3(cp.p * cp.p, GEO_CHEB_NI + 1), 32, 0, s>>>(cp, tab);
    return cudaGetLastError();
}

size_t cov_fine_doubles(int p, double pairs) {
    // with fewer location pairs the tables (11,600 evaluations per C_ij) cost more than they save
    return pairs >= 32768.0 ? (size_t)p * (p + 1) / 2 * GEO_FINE_PER_PAIR : 0;
}

size_t cov_fine_doubles(const CovParams &cp, double pairs) {
    // the tables' floats go down to 2^-800 (64 a out, C is 2^-93 of C(0)): covariances smaller than that go without
    for (int q = 0; q < cp.p * cp.p; ++q)
        if (cp.m[q].c0 != 0.0 && fabs(cp.m[q].c0) < 0x1p-700) return 0;
    return cov_fine_doubles(cp.p, pairs);
}

cudaError_t launch_fine_build(CovParams &cp, double *tab, double *fine, cudaStream_t s) {
    KScope ks(GEO_K_COVGEN, s);
    // tab == NULL: cp.tab is there already
    k_fine_build<<<dim3(cp.p * (cp.p + 1) / 2, FINE_BLOCKS + (tab ? COARSE_BLOCKS : 0)), 128, 0, s>>>(cp, tab, fine);
    if (tab) cp.tab = tab;
    cp.fine = fine;
    return cudaGetLastError();
}

cudaError_t launch_covgen_sym(const CovParams &cp, const double *lx, const double *ly, int n, double *A,
                              long long ld, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int per = cp.fine ? TR * RPT : TR;
    dim3 grid((n + per - 1) / per, (n + TL - 1) / TL);
    const double N = (double)cp.p * n;
    KScope ks(GEO_K_COVGEN, s, 0.0, 8.0 * N * (N + cp.p) / 2.0);   // bytes: lower triangle written once
    if (cp.fine)
        cov_by_p(cp.p, [&](auto P) { k_covgen_sym_fine<P.value><<<grid, TL * TR, 0, s>>>(cp, lx, ly, n, A, ld); });
    else
        k_covgen_sym<<<grid, TL * TR, 0, s>>>(cp, lx, ly, n, A, ld);
    return cudaGetLastError();
}

cudaError_t launch_covgen_rect(const CovParams &cp, const double *l1, int n1, const double *l2, int n2,
                               double *out, long long ld, cudaStream_t s) {
    if (n1 <= 0 || n2 <= 0) return cudaSuccess;
    const int per = cp.fine ? TR * RPT : TR;
    dim3 grid((n2 + per - 1) / per, (n1 + TL - 1) / TL);
    KScope ks(GEO_K_COVGEN, s, 0.0, 8.0 * cp.p * (double)n1 * cp.p * (double)n2);
    const bool closed = cov_closed(cp);
    cov_by_p(cp.p, [&](auto P) {
        if (cp.fine)
            k_covgen_rect<P.value, true><<<grid, TL * TR, 0, s>>>(cp, l1, n1, l2, n2, out, ld, closed);
        else
            k_covgen_rect<P.value, false><<<grid, TL * TR, 0, s>>>(cp, l1, n1, l2, n2, out, ld, closed);
    });
    return cudaGetLastError();
}

// Batched predictions: CTA g serves the new location g of the concatenation of
// every entry's locations; it finds its entry by binary search over the
// entries' first indices, copies the entry's theta constants into shared
// memory and computes exactly what k_predict computes for that location (same
// thread-to-r assignment, same reduction tree): bit-identical to one call per
// factor.
__global__ void __launch_bounds__(PRED_THREADS) k_predict_batch(const PredDesc *__restrict__ d, int count) {
    __shared__ CovParams cps;
    __shared__ int ent;
    const int g = blockIdx.x;
    if (threadIdx.x == 0) {
        int lo = 0, hi = count - 1;   // the last entry with first <= g
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (d[mid].first <= g) lo = mid;
            else hi = mid - 1;
        }
        ent = lo;
    }
    __syncthreads();
    const PredDesc &q = d[ent];
    {
        const int words = (int)(sizeof(CovParams) / sizeof(int));
        const int *src = reinterpret_cast<const int *>(&q.cp);
        int *dst = reinterpret_cast<int *>(&cps);
        for (int t = threadIdx.x; t < words; t += PRED_THREADS) dst[t] = src[t];
    }
    __syncthreads();
    const int l = g - q.first, p = cps.p;
    const double x0 = q.s0[2 * l], y0 = q.s0[2 * l + 1];
    double *out = q.zhat + (long long)p * l;
    switch (p) {
        case 1: predict_one<1>(cps, x0, y0, q.lx, q.ly, q.n, q.w, out); break;
        case 2: predict_one<2>(cps, x0, y0, q.lx, q.ly, q.n, q.w, out); break;
        case 3: predict_one<3>(cps, x0, y0, q.lx, q.ly, q.n, q.w, out); break;
        default: predict_one<4>(cps, x0, y0, q.lx, q.ly, q.n, q.w, out); break;
    }
}

cudaError_t launch_predict(const CovParams &cp, const double *new_locs, int m, const double *lx,
                           const double *ly, int n, const double *w, double *zhat, cudaStream_t s) {
    if (m <= 0) return cudaSuccess;
    KScope ks(GEO_K_PREDICT, s, 2.0 * cp.p * (double)m * cp.p * (double)n, 16.0 * n + 24.0 * m);
    cov_by_p(cp.p, [&](auto P) { k_predict<P.value><<<m, PRED_THREADS, 0, s>>>(cp, new_locs, lx, ly, n, w, zhat); });
    return cudaGetLastError();
}

cudaError_t launch_gather_locs(const double *locs, const int *perm, int n, double *lx, double *ly,
                               cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    KScope ks(GEO_K_AUX, s);
    k_gather_locs<<<(n + 255) / 256, 256, 0, s>>>(locs, perm, n, lx, ly);
    return cudaGetLastError();
}

cudaError_t launch_gather_vec(const double *in, const int *perm, int n, int p, double *out, long long stride,
                              cudaStream_t s) {
    const long long t = (long long)n * p;
    if (t <= 0) return cudaSuccess;
    KScope ks(GEO_K_AUX, s);
    k_gather_vec<<<(unsigned)((t + 255) / 256), 256, 0, s>>>(in, perm, n, p, out, stride);
    return cudaGetLastError();
}

cudaError_t launch_scatter_vec(const double *in, long long stride, const int *perm, int n, int p, double *out,
                               cudaStream_t s) {
    const long long t = (long long)n * p;
    if (t <= 0) return cudaSuccess;
    KScope ks(GEO_K_AUX, s);
    k_scatter_vec<<<(unsigned)((t + 255) / 256), 256, 0, s>>>(in, stride, perm, n, p, out);
    return cudaGetLastError();
}

cudaError_t launch_predict_batch(const PredDesc *d, int count, int total, double flops, cudaStream_t s) {
    if (total <= 0) return cudaSuccess;
    KScope ks(GEO_K_PREDICT, s, flops, 0.0);
    k_predict_batch<<<total, PRED_THREADS, 0, s>>>(d, count);
    return cudaGetLastError();
}
