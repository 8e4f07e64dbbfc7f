// Batched FP64 building blocks of the tile-low-rank factorisation (Sec. 5.3):
// variable-size GEMMs, Householder QR of tall-skinny blocks, one-sided Jacobi
// SVD of small square blocks, and the Gaussian test matrices of the
// randomized range finder.  Every problem of a batch is independent; each
// kernel maps one problem (or one 64 x 64 tile of it) to one CTA.
#include <math.h>

#include <algorithm>

#include <cooperative_groups.h>

#include "geo_internal.cuh"

namespace cg = cooperative_groups;

namespace {

// ---- batched GEMM: C = alpha op(A) op(B) + beta C (column-major) ----------
// One CTA per 64 x 64 output tile of one problem, 4 x 4 outputs per thread
// (rows ty + 16 i, columns tx + 16 j).  The FP64 pipe is the limit (a few DFMA
// per clock per SM), so work on padding is the waste to avoid: a tile whose
// rows (columns) end inside it runs only the IM (JM) sixteen-row (-column)
// strips that hold outputs, and the last K slice runs only its valid depth.
// Ranks and sketch widths (the skinny side of most products here) are rarely
// multiples of 64.
constexpr int BT = 64, BKK = 16;

// K range [kbeg, kend); part == NULL: C = alpha acc + beta C, else the raw
// sums go to the tile-local partial part[(c - tn) * pw + (r - tm)].
template <int IM, int JM>
__device__ __forceinline__ void bgemm_tile(const GemmDesc &g, int tm, int tn, double (*As)[BT + 2],
                                           double (*Bs)[BT + 2], int kbeg, int kend, double *part, int pw) {
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    double acc[IM][JM];
#pragma unroll
    for (int i = 0; i < IM; ++i)
#pragma unroll
        for (int j = 0; j < JM; ++j) acc[i][j] = 0.0;
    for (int k0 = kbeg; k0 < kend; k0 += BKK) {
        // consecutive threads walk the operand's contiguous index: rows for a
        // row-contiguous slice, K for a K-contiguous one (transposed A, plain B)
        for (int t = threadIdx.x; t < BKK * 16 * IM; t += 256) {
            const int kk = g.ta ? t % BKK : t / (16 * IM), r = g.ta ? t / BKK : t % (16 * IM);
            const int kg = k0 + kk;
            double a = 0.0;
            if (kg < kend && tm + r < g.m)
                a = g.ta ? g.A[(long long)(tm + r) * g.lda + kg] : g.A[(long long)kg * g.lda + tm + r];
            As[kk][r] = a;
        }
        for (int t = threadIdx.x; t < BKK * 16 * JM; t += 256) {
            const int kk = g.tb ? t / (16 * JM) : t % BKK, r = g.tb ? t % (16 * JM) : t / BKK;
            const int kg = k0 + kk;
            double b = 0.0;
            if (kg < kend && tn + r < g.n)
                b = g.tb ? g.B[(long long)kg * g.ldb + tn + r] : g.B[(long long)(tn + r) * g.ldb + kg];
            Bs[kk][r] = b;
        }
        __syncthreads();
        const int kc = min(BKK, kend - k0);   // uniform over the CTA
        if (kc == BKK) {
#pragma unroll
            for (int kk = 0; kk < BKK; ++kk) {
                double a[IM], b[JM];
#pragma unroll
                for (int i = 0; i < IM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < JM; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < IM; ++i)
#pragma unroll
                    for (int j = 0; j < JM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        } else {
            for (int kk = 0; kk < kc; ++kk) {
                double a[IM], b[JM];
#pragma unroll
                for (int i = 0; i < IM; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < JM; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
                for (int i = 0; i < IM; ++i)
#pragma unroll
                    for (int j = 0; j < JM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < JM; ++j) {
        const int c = tn + tx + 16 * j;
        if (c >= g.n) continue;
#pragma unroll
        for (int i = 0; i < IM; ++i) {
            const int r = tm + ty + 16 * i;
            if (r >= g.m) continue;
            if (part) {
                part[(c - tn) * pw + (r - tm)] = acc[i][j];
                continue;
            }
            double *p = g.C + (long long)c * g.ldc + r;
            *p = g.alpha * acc[i][j] + (g.beta == 0.0 ? 0.0 : g.beta * *p);
        }
    }
}

__global__ void __launch_bounds__(256) k_bgemm(const GemmDesc *__restrict__ d, int count) {
    __shared__ double As[BKK][BT + 2];
    __shared__ double Bs[BKK][BT + 2];
    const int pi = blockIdx.y;
    if (pi >= count) return;
    const GemmDesc g = d[pi];
    const int tiles_m = (g.m + BT - 1) / BT;
    const int tiles_n = (g.n + BT - 1) / BT;
    if ((int)blockIdx.x >= tiles_m * tiles_n) return;
    const int tm = (blockIdx.x % tiles_m) * BT, tn = (blockIdx.x / tiles_m) * BT;
    const int im = min(4, (g.m - tm + 15) / 16), jm = min(4, (g.n - tn + 15) / 16);
    switch ((im - 1) * 4 + (jm - 1)) {
#define GEO_BGEMM_CASE(I, J) \
    case (I - 1) * 4 + (J - 1): bgemm_tile<I, J>(g, tm, tn, As, Bs, 0, g.k, nullptr, 0); break;
        GEO_BGEMM_CASE(1, 1) GEO_BGEMM_CASE(1, 2) GEO_BGEMM_CASE(1, 3) GEO_BGEMM_CASE(1, 4)
        GEO_BGEMM_CASE(2, 1) GEO_BGEMM_CASE(2, 2) GEO_BGEMM_CASE(2, 3) GEO_BGEMM_CASE(2, 4)
        GEO_BGEMM_CASE(3, 1) GEO_BGEMM_CASE(3, 2) GEO_BGEMM_CASE(3, 3) GEO_BGEMM_CASE(3, 4)
        GEO_BGEMM_CASE(4, 1) GEO_BGEMM_CASE(4, 2) GEO_BGEMM_CASE(4, 3) GEO_BGEMM_CASE(4, 4)
#undef GEO_BGEMM_CASE
        default: break;
    }
}

// The same strips on 32 x 32 (S = 2) or 16 x 16 (S = 1) output tiles: for
// launches whose 64 x 64 tiles would leave most SMs idle (few output tiles,
// long K, e.g. the r x r cores V_ik' V_jk with K = nb), 4x or 16x more CTAs
// share the K loops' FP64 work.  Split-K (ws != NULL): blockIdx.z takes one of
// zsplit contiguous K ranges and writes its raw sums to its own partial tile
// ws[((pi zsplit + z) tiles_cap + tile) W^2 ..]; k_bgemm_reduce adds them.
template <int S>
__global__ void __launch_bounds__(256) k_bgemm_small(const GemmDesc *__restrict__ d, int count, int zsplit,
                                                     int tiles_cap, double *ws) {
    __shared__ double As[BKK][BT + 2];
    __shared__ double Bs[BKK][BT + 2];
    const int pi = blockIdx.y;
    if (pi >= count) return;
    const GemmDesc g = d[pi];
    constexpr int W = 16 * S;
    const int tiles_m = (g.m + W - 1) / W;
    const int tiles_n = (g.n + W - 1) / W;
    if ((int)blockIdx.x >= tiles_m * tiles_n) return;
    const int tm = (blockIdx.x % tiles_m) * W, tn = (blockIdx.x / tiles_m) * W;
    const int im = min(S, (g.m - tm + 15) / 16), jm = min(S, (g.n - tn + 15) / 16);
    int kbeg = 0, kend = g.k;
    double *part = nullptr;
    if (ws) {
        const int kc = ((g.k + zsplit - 1) / zsplit + BKK - 1) / BKK * BKK;
        kbeg = min(g.k, (int)blockIdx.z * kc);
        kend = min(g.k, kbeg + kc);
        part = ws + (((long long)pi * zsplit + blockIdx.z) * tiles_cap + blockIdx.x) * (W * W);
    }
    if (S == 1 || (im == 1 && jm == 1))
        bgemm_tile<1, 1>(g, tm, tn, As, Bs, kbeg, kend, part, W);
    else if (im == 1)
        bgemm_tile<1, S == 1 ? 1 : 2>(g, tm, tn, As, Bs, kbeg, kend, part, W);
    else if (jm == 1)
        bgemm_tile<S == 1 ? 1 : 2, 1>(g, tm, tn, As, Bs, kbeg, kend, part, W);
    else
        bgemm_tile<S == 1 ? 1 : 2, S == 1 ? 1 : 2>(g, tm, tn, As, Bs, kbeg, kend, part, W);
}

// C = alpha (sum of the zsplit partial tiles, in order) + beta C: the same
// result on every run.
template <int W>
__global__ void __launch_bounds__(256) k_bgemm_reduce(const GemmDesc *__restrict__ d, int count, int zsplit,
                                                      int tiles_cap, const double *__restrict__ ws) {
    const int pi = blockIdx.y;
    if (pi >= count) return;
    const GemmDesc g = d[pi];
    const int tiles_m = (g.m + W - 1) / W;
    const int tiles_n = (g.n + W - 1) / W;
    if ((int)blockIdx.x >= tiles_m * tiles_n) return;
    const int tm = (blockIdx.x % tiles_m) * W, tn = (blockIdx.x / tiles_m) * W;
    for (int e = threadIdx.x; e < W * W; e += blockDim.x) {
        const int i = e % W, j = e / W;
        if (tm + i >= g.m || tn + j >= g.n) continue;
        double sum = 0.0;
        for (int z = 0; z < zsplit; ++z)
            sum += ws[(((long long)pi * zsplit + z) * tiles_cap + blockIdx.x) * (W * W) + e];
        double *p = g.C + (long long)(tn + j) * g.ldc + tm + i;
        *p = g.alpha * sum + (g.beta == 0.0 ? 0.0 : g.beta * *p);
    }
}

// ---- Householder QR of an m x r block (m >= r), in place -------------------
// Column c: v = x - alpha e1 with alpha = -sign(x_0) |x|, stored below the
// diagonal (v_0 kept in tau-scaled form), R on and above the diagonal; then
// the thin Q (m x r) is formed in Qout by applying the reflectors backwards
// to [I; 0].  One CTA (32 warps) per block; warp w updates columns w, w+32, ...
__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return __shfl_sync(0xffffffffu, v, 0);
}

constexpr int LA_THREADS = 1024, LA_WARPS = LA_THREADS / 32;

__global__ void __launch_bounds__(LA_THREADS) k_house_qr(const QrDesc *__restrict__ d, int count) {
    const int pi = blockIdx.x;
    if (pi >= count) return;
    const QrDesc q = d[pi];
    double *Y = q.Y;
    const long long ld = q.ldy;
    const int m = q.m, r = q.r;
    double *tau = q.tau;   // r entries
    __shared__ double red[LA_WARPS];
    __shared__ double s_alpha, s_tau, s_v0;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int c = 0; c < r; ++c) {
        double *x = Y + (long long)c * ld;
        // norm of x[c:m]
        double s = 0.0;
        for (int i = c + threadIdx.x; i < m; i += LA_THREADS) s += x[i] * x[i];
        s = warp_sum(s);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < LA_WARPS; ++w) t += red[w];
            const double nrm = sqrt(t);
            const double x0 = x[c];
            double alpha = (x0 >= 0.0) ? -nrm : nrm;
            double v0 = x0 - alpha;
            double taue;
            if (nrm == 0.0) {
                alpha = 0.0;
                v0 = 1.0;
                taue = 0.0;
            } else {
                // H = I - tau v v' with v = (v0, x[c+1:]), tau = 2 / (v'v), v'v = 2 nrm (nrm - x0 sign...)
                const double vtv = v0 * v0 + (t - x0 * x0);
                taue = (vtv > 0.0) ? 2.0 / vtv : 0.0;
            }
            s_alpha = alpha;
            s_tau = taue;
            s_v0 = v0;
        }
        __syncthreads();
        const double v0 = s_v0, tauc = s_tau;
        // apply to columns c+1 .. r-1: y -= tau (v'y) v
        for (int j = c + 1 + warp; j < r; j += LA_WARPS) {
            double *y = Y + (long long)j * ld;
            double dot = (lane == 0) ? v0 * y[c] : 0.0;
            for (int i = c + 1 + lane; i < m; i += 32) dot += x[i] * y[i];
            dot = warp_sum(dot) * tauc;
            if (lane == 0) y[c] -= dot * v0;
            for (int i = c + 1 + lane; i < m; i += 32) y[i] -= dot * x[i];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            x[c] = s_alpha;   // R diagonal
            tau[c] = s_tau;
            q.v0[c] = s_v0;
        }
        __syncthreads();
    }
    // thin Q: start from [I; 0] and apply H_c for c = r-1 .. 0
    double *Q = q.Q;
    const long long ldq = q.ldq;
    if (!Q) return;   // only R was wanted
    for (int j = warp; j < r; j += LA_WARPS)
        for (int i = lane; i < m; i += 32) Q[(long long)j * ldq + i] = (i == j) ? 1.0 : 0.0;
    __syncthreads();
    for (int c = r - 1; c >= 0; --c) {
        const double *x = Y + (long long)c * ld;
        const double v0 = q.v0[c], tauc = tau[c];
        for (int j = c + warp; j < r; j += LA_WARPS) {
            double *y = Q + (long long)j * ldq;
            double dot = (lane == 0) ? v0 * y[c] : 0.0;
            for (int i = c + 1 + lane; i < m; i += 32) dot += x[i] * y[i];
            dot = warp_sum(dot) * tauc;
            if (lane == 0) y[c] -= dot * v0;
            for (int i = c + 1 + lane; i < m; i += 32) y[i] -= dot * x[i];
        }
        __syncthreads();
    }
}

// ---- the same Householder QR on a cluster of QC CTAs ------------------------
// Rows are split over the CTAs of a cluster (the block stays in global
// memory, which L2 holds); per column c the CTAs exchange partial norms, then
// partial products v'y_j for the trailing columns, through distributed shared
// memory, every CTA forming alpha, v0, tau and the dots in rank order (so all
// take the same values), and each updates its own rows.  The thin Q is
// accumulated the same way.  r <= QR_MAX.
constexpr int QC = 8, QT = 256, QR_MAX = 256;

size_t house_qr_cl_smem(int m) {
    const int rs = (m + QC - 1) / QC;
    return sizeof(double) * ((size_t)rs + 2 * (QR_MAX + 2) + 2 * QR_MAX);
}

__global__ void __launch_bounds__(QT, 1) k_house_qr_cl(const QrDesc *__restrict__ d, int count) {
    cg::cluster_group cluster = cg::this_cluster();
    const int tile = blockIdx.x / QC;
    if (tile >= count) return;   // uniform over the cluster
    const int rank = (int)cluster.block_rank();
    const QrDesc q = d[tile];
    double *Y = q.Y;
    const long long ld = q.ldy;
    const int m = q.m, r = q.r;
    const int rs = (m + QC - 1) / QC;
    const int row0 = rank * rs, row1 = min(m, row0 + rs);
    extern __shared__ double qsm[];
    double *vloc = qsm;                       // reflector on this CTA's rows (row c holds v0)
    double *P = vloc + rs;                    // [2][QR_MAX + 2]: partial dots, then norm, x_c
    double *taus = P + 2 * (QR_MAX + 2);      // [QR_MAX]
    double *v0s = taus + QR_MAX;              // [QR_MAX]
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = QT / 32;
    int buf = 0;
    for (int c = 0; c < r; ++c) {
        double *Pb = P + buf * (QR_MAX + 2);
        const double *x = Y + (long long)c * ld;
        // (a) partial |x[c:]|^2 over this CTA's rows; the owner of row c also passes x_c
        const int i0 = max(c, row0);
        double t = 0.0;
        for (int i = i0 + threadIdx.x; i < row1; i += QT) t = fma(x[i], x[i], t);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        __shared__ double red[QT / 32];
        if (lane == 0) red[warp] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            double a = 0.0;
            for (int w = 0; w < nw; ++w) a += red[w];
            Pb[QR_MAX] = a;
            Pb[QR_MAX + 1] = (c >= row0 && c < row1) ? x[c] : 0.0;
        }
        cluster.sync();
        // (b) alpha, v0, tau (the same in every CTA)
        double nrm2 = 0.0;
        for (int k = 0; k < QC; ++k) nrm2 += cluster.map_shared_rank(Pb, k)[QR_MAX];
        const double x0 = cluster.map_shared_rank(Pb, c / rs)[QR_MAX + 1];
        const double nrm = sqrt(nrm2);
        double alpha = (x0 >= 0.0) ? -nrm : nrm;
        double v0 = x0 - alpha, tauc;
        if (nrm == 0.0) {
            alpha = 0.0;
            v0 = 1.0;
            tauc = 0.0;
        } else {
            const double vtv = v0 * v0 + (nrm2 - x0 * x0);
            tauc = (vtv > 0.0) ? 2.0 / vtv : 0.0;
        }
        // the reflector on this CTA's rows
        for (int i = i0 + threadIdx.x; i < row1; i += QT) vloc[i - row0] = (i == c) ? v0 : x[i];
        __syncthreads();
        // (c) partial v'y_j for j > c: a warp per pair of columns, lanes over rows
        for (int j = c + 1 + warp; j < r; j += 2 * nw) {
            const int j2 = j + nw;
            const double *y = Y + (long long)j * ld, *y2 = Y + (long long)(j2 < r ? j2 : j) * ld;
            double dot = 0.0, dot2 = 0.0;
#pragma unroll 4
            for (int i = i0 + lane; i < row1; i += 32) {
                const double v = vloc[i - row0];
                dot = fma(v, y[i], dot);
                dot2 = fma(v, y2[i], dot2);
            }
            for (int o = 16; o > 0; o >>= 1) {
                dot += __shfl_down_sync(0xffffffffu, dot, o);
                dot2 += __shfl_down_sync(0xffffffffu, dot2, o);
            }
            if (lane == 0) {
                Pb[j] = dot;
                if (j2 < r) Pb[j2] = dot2;
            }
        }
        cluster.sync();
        // (d) y_j -= tau (v'y_j) v on this CTA's rows
        for (int j = c + 1 + warp; j < r; j += nw) {
            double dot = 0.0;
            for (int k = 0; k < QC; ++k) dot += cluster.map_shared_rank(Pb, k)[j];
            dot *= tauc;
            double *y = Y + (long long)j * ld;
            for (int i = i0 + lane; i < row1; i += 32) y[i] -= dot * vloc[i - row0];
        }
        if (threadIdx.x == 0) {
            taus[c] = tauc;
            v0s[c] = v0;
            if (c >= row0 && c < row1) {
                Y[(long long)c * ld + c] = alpha;   // R diagonal
                q.tau[c] = tauc;
                q.v0[c] = v0;
            }
        }
        __syncthreads();
        buf ^= 1;
    }
    // thin Q: [I; 0] on this CTA's rows, then H_c for c = r-1 .. 0
    double *Q = q.Q;
    const long long ldq = q.ldq;
    if (!Q) {   // only R was wanted
        cluster.sync();
        return;
    }
    for (int j = warp; j < r; j += nw)
        for (int i = row0 + lane; i < row1; i += 32) Q[(long long)j * ldq + i] = (i == j) ? 1.0 : 0.0;
    __syncthreads();
    for (int c = r - 1; c >= 0; --c) {
        double *Pb = P + buf * (QR_MAX + 2);
        const double *x = Y + (long long)c * ld;
        const int i0 = max(c, row0);
        const double v0 = v0s[c], tauc = taus[c];
        for (int j = c + warp; j < r; j += 2 * nw) {
            const int j2 = j + nw;
            const double *y = Q + (long long)j * ldq, *y2 = Q + (long long)(j2 < r ? j2 : j) * ldq;
            double dot = 0.0, dot2 = 0.0;
#pragma unroll 4
            for (int i = i0 + lane; i < row1; i += 32) {
                const double v = (i == c) ? v0 : x[i];
                dot = fma(v, y[i], dot);
                dot2 = fma(v, y2[i], dot2);
            }
            for (int o = 16; o > 0; o >>= 1) {
                dot += __shfl_down_sync(0xffffffffu, dot, o);
                dot2 += __shfl_down_sync(0xffffffffu, dot2, o);
            }
            if (lane == 0) {
                Pb[j] = dot;
                if (j2 < r) Pb[j2] = dot2;
            }
        }
        cluster.sync();
        for (int j = c + warp; j < r; j += nw) {
            double dot = 0.0;
            for (int k = 0; k < QC; ++k) dot += cluster.map_shared_rank(Pb, k)[j];
            dot *= tauc;
            double *y = Q + (long long)j * ldq;
            for (int i = i0 + lane; i < row1; i += 32) y[i] -= dot * ((i == c) ? v0 : x[i]);
        }
        __syncthreads();
        buf ^= 1;
    }
    cluster.sync();   // no CTA leaves while another still reads its shared memory
}

// ---- the same with the whole block in the shared memory of a cluster ---------
// Columns are dealt out to the CTAs in turn (column j to CTA j % QC), all rows
// of each in shared memory: a reflector needs no exchange of partial dots, only
// the reflector itself, which its column's CTA stores into the others' shared
// memory before the step's one cluster barrier.  A warp takes a column, or two
// at once so that their sums share the shuffles; the norm of the next column
// comes out of its update.  The reflectors also go to global memory (in place),
// from where the thin Q, which takes the block's place in shared memory, is
// accumulated without any exchange.  With Rt only R is formed: R' goes to Rt
// and the block is left as it is.  Bound by the FP64 units of eight SMs:
// m = 900, r = 216 3.6 ms, R alone 2.2 (16.5 with the rows split over the CTAs
// and two exchanges a column).
constexpr int QCT = 512, QCW = QCT / 32;

size_t house_qr_col_smem(int m, int r) {
    return sizeof(double) * ((size_t)((r + QC - 1) / QC) * m + 2 * (size_t)(m + 2) + QR_MAX + 4);
}

// 1 / sqrt(d) and 1 / d of a positive normal d: the hardware's approximations (20 bits and more) and one step of
// Halley's iteration.
__device__ __forceinline__ double fast_rsqrt(double d) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-(d * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double fast_rcp(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// y_j -= tau (v'y_j) v for two columns (b2: the second one exists), rows [c, m); v in shared memory, row i at
// v[i].  nrm: receives |y[c1..]|^2 of the first column over the rows from c1 on (NULL: not wanted).
__device__ __forceinline__ void qr_apply(const double *v, double tau, double *y1, double *y2, bool b2, int c, int m, int c1,
                                         double *nrm, int lane) {
    double d1 = 0.0, d2 = 0.0;
    const double *z2 = b2 ? y2 : y1;
    for (int i = c + lane; i < m; i += 32) {
        const double vi = v[i];
        d1 = fma(vi, y1[i], d1);
        d2 = fma(vi, z2[i], d2);
    }
    // lanes 0-15 sum the first column, 16-31 the second
    double a = (lane < 16 ? d1 : d2) + __shfl_xor_sync(0xffffffffu, lane < 16 ? d2 : d1, 16);
    for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    a *= -tau;
    d1 = __shfl_sync(0xffffffffu, a, 0);
    d2 = __shfl_sync(0xffffffffu, a, 16);
    double s = 0.0;
    for (int i = c + lane; i < m; i += 32) {
        const double vi = v[i], n1 = fma(d1, vi, y1[i]);
        y1[i] = n1;
        if (b2) y2[i] = fma(d2, vi, y2[i]);
        if (nrm && i >= c1) s = fma(n1, n1, s);
    }
    if (nrm) {
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) *nrm = s;
    }
}

__global__ void __launch_bounds__(QCT, 1) k_house_qr_col(const QrDesc *__restrict__ d, int count) {
    cg::cluster_group cluster = cg::this_cluster();
    const int tile = blockIdx.x / QC;
    if (tile >= count) return;   // uniform over the cluster
    const int rank = (int)cluster.block_rank();
    const QrDesc q = d[tile];
    const int m = q.m, r = q.r, nloc = (r + QC - 1) / QC;
    extern __shared__ double csm[];
    double *Ys = csm;                          // [nloc][m]
    double *vb = Ys + (size_t)nloc * m;        // [2][m + 2]: reflector (row i at i), then tau at m
    double *taus = vb + 2 * (m + 2);           // [QR_MAX]
    double *sc = taus + QR_MAX;                // norm of the next column; alpha, v0, tau of the current one
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int lj = warp; lj < nloc; lj += QCW) {
        const int j = lj * QC + rank;
        if (j < r)
            for (int i = lane; i < m; i += 32) Ys[(size_t)lj * m + i] = q.Y[(long long)j * q.ldy + i];
    }
    __syncthreads();
    if (rank == 0 && warp == 0) {
        double s = 0.0;
        for (int i = lane; i < m; i += 32) s = fma(Ys[i], Ys[i], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) sc[0] = s;
    }
    cluster.sync();   // every CTA runs (its shared memory may be written); the first norm
    for (int c = 0; c < r; ++c) {
        double *v = vb + (c & 1) * (m + 2);
        if (rank == c % QC) {
            double *x = Ys + (size_t)(c / QC) * m;
            if (warp == 0 && lane == 0) {
                const double nrm2 = sc[0], x0 = x[c];
                double alpha = 0.0, v0 = 1.0, tau = 0.0;
                if (nrm2 > 0.0) {
                    const double nrm = sqrt(nrm2);
                    alpha = (x0 >= 0.0) ? -nrm : nrm;
                    v0 = x0 - alpha;
                    // v'v = v0^2 + (nrm2 - x0^2) = 2 nrm (nrm + |x0|)
                    tau = 1.0 / (nrm * (nrm + fabs(x0)));
                }
                sc[1] = alpha;
                sc[2] = v0;
                sc[3] = tau;
            }
            __syncthreads();
            const double alpha = sc[1], v0 = sc[2], tau = sc[3];
            for (int i = c + threadIdx.x; i < m; i += QCT) {
                const double vi = i == c ? v0 : x[i];
                for (int k = 0; k < QC; ++k) cluster.map_shared_rank(v, k)[i] = vi;
                if (q.Q) q.Y[(long long)c * q.ldy + i] = vi;
            }
            if (threadIdx.x < QC) cluster.map_shared_rank(v, threadIdx.x)[m] = tau;
            __syncthreads();
            if (threadIdx.x == 0) x[c] = alpha;   // R's diagonal
        }
        cluster.sync();
        const double tau = v[m];
        if (threadIdx.x == 0) taus[c] = tau;
        // the columns after c on this CTA; the next column (if it is here) first, alone
        const int l0 = (c + QC - rank) / QC;   // first local column with j > c
        const bool own = rank == (c + 1) % QC && c + 1 < r;
        if (own && warp == 0) qr_apply(v, tau, Ys + (size_t)l0 * m, nullptr, false, c, m, c + 1, sc, lane);
        const int lf = l0 + (own ? 1 : 0), nl = (r - rank + QC - 1) / QC - lf;   // the others
        // one column a warp while there are warps enough, else two
        const int w = own ? warp - 1 : warp, nw = own ? QCW - 1 : QCW;
        if (w >= 0) {
            if (nl <= nw) {
                if (w < nl) qr_apply(v, tau, Ys + (size_t)(lf + w) * m, nullptr, false, c, m, 0, nullptr, lane);
            } else {
                for (int p = w; 2 * p < nl; p += nw)
                    qr_apply(v, tau, Ys + (size_t)(lf + 2 * p) * m, Ys + (size_t)(lf + 2 * p + 1) * m, 2 * p + 1 < nl, c, m, 0,
                             nullptr, lane);
            }
        }
        __syncthreads();
    }
    if (q.Rt) {   // column j of R is row j of the lower triangular R'
        for (int lj = warp; lj < nloc; lj += QCW) {
            const int j = lj * QC + rank;
            if (j < r)
                for (int c = lane; c < r; c += 32) q.Rt[(long long)c * q.ldr + j] = c <= j ? Ys[(size_t)lj * m + c] : 0.0;
        }
    }
    if (!q.Q) {
        cluster.sync();   // no CTA leaves while another may still write its shared memory
        return;
    }
    __threadfence();
    cluster.sync();       // the reflectors in global memory
    for (int lj = warp; lj < nloc; lj += QCW) {
        const int j = lj * QC + rank;
        for (int i = lane; i < m; i += 32) Ys[(size_t)lj * m + i] = (i == j) ? 1.0 : 0.0;
    }
    auto fetch = [&](int c) {
        for (int i = c + threadIdx.x; i < m; i += QCT) vb[(c & 1) * (m + 2) + i] = __ldcg(q.Y + (long long)c * q.ldy + i);
    };
    fetch(r - 1);
    __syncthreads();
    for (int c = r - 1; c >= 0; --c) {
        if (c > 0) fetch(c - 1);
        const double *v = vb + (c & 1) * (m + 2);
        const double tau = taus[c];
        const int lf = (c + QC - 1 - rank) / QC, nl = (r - rank + QC - 1) / QC - lf;   // local columns with j >= c
        if (nl <= QCW) {
            if (warp < nl) qr_apply(v, tau, Ys + (size_t)(lf + warp) * m, nullptr, false, c, m, 0, nullptr, lane);
        } else {
            for (int p = warp; 2 * p < nl; p += QCW)
                qr_apply(v, tau, Ys + (size_t)(lf + 2 * p) * m, Ys + (size_t)(lf + 2 * p + 1) * m, 2 * p + 1 < nl, c, m, 0,
                         nullptr, lane);
        }
        __syncthreads();
    }
    for (int lj = warp; lj < nloc; lj += QCW) {
        const int j = lj * QC + rank;
        if (j < r)
            for (int i = lane; i < m; i += 32) q.Q[(long long)j * q.ldq + i] = Ys[(size_t)lj * m + i];
    }
}

// ---- one-sided Jacobi SVD of an r x r block M (Hestenes) --------------------
// Rotates column pairs of M until every pair is orthogonal to relative 1e-13 or
// the sweep budget is spent (pairs whose columns both have norms below `skip`
// are not rotated); on exit the column norms of M are the singular values
// (unsorted) and the columns over their norms the left singular vectors.
// Pairs are processed in round-robin order, r/2 disjoint pairs per round, one
// warp per pair.
__global__ void __launch_bounds__(LA_THREADS) k_jacobi_svd(const SvdDesc *__restrict__ d, int count, int max_sweeps) {
    const int pi = blockIdx.x;
    if (pi >= count) return;
    const SvdDesc s = d[pi];
    const int r = s.r;
    double *M = s.M;
    const long long ld = s.ld;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    __shared__ int rotated;
    const int rr = r + (r & 1);   // round-robin over an even count (index r = dummy)
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
        if (threadIdx.x == 0) rotated = 0;
        __syncthreads();
        for (int round = 0; round < rr - 1; ++round) {
            for (int pr = warp; pr < rr / 2; pr += LA_WARPS) {
                // pairing of the circle method: position 0 fixed, others rotate
                int a = (pr == 0) ? 0 : 1 + (pr - 1 + round) % (rr - 1);
                int b = 1 + (rr - 2 - pr + round) % (rr - 1);
                if (a >= r || b >= r || a == b) continue;
                if (a > b) {
                    const int t = a;
                    a = b;
                    b = t;
                }
                double *ma = M + (long long)a * ld, *mb = M + (long long)b * ld;
                double al = 0.0, be = 0.0, ga = 0.0;
                for (int i = lane; i < r; i += 32) {
                    const double x = ma[i], y = mb[i];
                    al += x * x;
                    be += y * y;
                    ga += x * y;
                }
                al = warp_sum(al);
                be = warp_sum(be);
                ga = warp_sum(ga);
                // both columns far below the truncation threshold: they are dropped anyway,
                // and any combination of them stays below sqrt(r) * skip
                if (al < s.skip * s.skip && be < s.skip * s.skip) continue;
                if (fabs(ga) <= 1e-13 * sqrt(al * be) || ga == 0.0) continue;
                const double zeta = (be - al) / (2.0 * ga);
                const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                const double cs = 1.0 / sqrt(1.0 + t * t), sn = cs * t;
                for (int i = lane; i < r; i += 32) {
                    const double x = ma[i], y = mb[i];
                    ma[i] = cs * x - sn * y;
                    mb[i] = sn * x + cs * y;
                }
                if (lane == 0) rotated = 1;
            }
            __syncthreads();
        }
        if (!rotated) break;
        __syncthreads();
    }
    // singular values = column norms
    for (int j = warp; j < r; j += LA_WARPS) {
        double t = 0.0;
        for (int i = lane; i < r; i += 32) t += M[(long long)j * ld + i] * M[(long long)j * ld + i];
        t = warp_sum(t);
        if (lane == 0) s.sigma[j] = sqrt(t);
    }
}

// ---- the same on a cluster of JC CTAs, by blocks of columns ------------------
// The columns form 2 JC blocks of at most 16; a CTA holds two, all rows of them
// in shared memory.  A sweep is 2 JC - 1 rounds of the circle method over the
// blocks: in a round a CTA meets every column of its one block with every
// column of the other (b steps of b disjoint pairs; the pairs within the two
// blocks come first in a sweep), then the blocks move on to the neighbours'
// other buffer through distributed shared memory: one cluster barrier a round,
// where rows dealt out to the CTAs need one per step.  Sixteen threads take a
// pair, its columns in registers between the dot product and the rotation; the
// squared norms are carried along (and taken afresh every round and when one
// shrinks much).  A warp-wide FP64 operation holds its scheduler for 64
// clocks, so what counts is their number: five per entry of a pair, and some
// twenty for the angle, from the hardware's approximations refined.
// r = 216: 1.1 ms a sweep where every pair rotates (3.6).  r <= 256.
constexpr int JC = 8, JT = 256, JR_MAX = 256, JBM = JR_MAX / (2 * JC);

size_t jacobi_cl_smem(int b, int rows) { return sizeof(double) * (2 * 2 * (size_t)b * rows + 2 * 2 * JBM); }

template <int NR>   // rows / 16
__global__ void __launch_bounds__(JT, 1) k_jacobi_svd_cl(const SvdDesc *__restrict__ d, int count, int max_sweeps, int bmax) {
    cg::cluster_group cluster = cg::this_cluster();
    const int tile = blockIdx.x / JC;
    if (tile >= count) return;   // uniform over the cluster
    const int rank = (int)cluster.block_rank();
    constexpr int ROWS = 16 * NR;
    extern __shared__ double sm[];
    const SvdDesc s = d[tile];
    const int r = s.r, b = (r + 2 * JC - 1) / (2 * JC);
    const long long ld = s.ld;
    const size_t blk = (size_t)bmax * ROWS;           // doubles of one block buffer
    double *norms = sm + 4 * blk;                     // [2 buffers][2 blocks][JBM]
    __shared__ int flags[2][JC], mine;
    auto col = [&](int buf, int w, int c) { return sm + (buf * 2 + w) * blk + (size_t)c * ROWS; };
    auto nrm = [&](int buf, int w) { return norms + (buf * 2 + w) * JBM; };
    const int g = threadIdx.x / 16, l = threadIdx.x % 16;   // pair slot, lane within it
    const double skip2 = s.skip * s.skip;
    // blocks rank (w = 0) and JC + rank (w = 1)
    for (int w = 0; w < 2; ++w)
        for (int c = g; c < b; c += JT / 16) {
            const int j = (w * JC + rank) * b + c;
            for (int i = l; i < ROWS; i += 16) col(0, w, c)[i] = (j < r && i < r) ? s.M[(long long)j * ld + i] : 0.0;
        }
    cluster.sync();   // every CTA runs: its shared memory may be written
    int buf = 0, sweep = 0, rotated = 0;
    auto sum16 = [](double v) {
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    // one pair per slot: columns xa (squared norm *na) and xb (*nb); act = the slot has a pair.  Every lane of the
    // warp takes part in the shuffles.
    auto pair = [&](double *xa, double *xb, double *na, double *nb, bool act) {
        double al = 0.0, be = 0.0;
        if (act) al = *na, be = *nb;
        act = act && !(al < skip2 && be < skip2);
        if (!__any_sync(0xffffffffu, act)) return;
        double x[NR], y[NR], ga = 0.0;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            x[i] = act ? xa[16 * i + l] : 0.0;
            y[i] = act ? xb[16 * i + l] : 0.0;
            ga = fma(x[i], y[i], ga);
        }
        ga = sum16(ga);
        const bool rot = act && ga * ga > 1e-26 * (al * be);
        if (!__any_sync(0xffffffffu, rot)) return;
        // t = tan of the angle: the smaller root of t^2 + 2 zeta t - 1, zeta = (be - al) / (2 ga)
        double cs = 1.0, sn = 0.0, t = 0.0;
        if (rot) {
            const double dd = be - al, h = fma(dd, dd, 4.0 * (ga * ga));
            t = 2.0 * ga * fast_rcp(fabs(dd) + h * fast_rsqrt(h));
            if (dd < 0.0) t = -t;
            cs = fast_rsqrt(fma(t, t, 1.0));
            sn = cs * t;
        }
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const double xn = fma(cs, x[i], -(sn * y[i]));
            y[i] = fma(sn, x[i], cs * y[i]);
            x[i] = xn;
            if (rot) {
                xa[16 * i + l] = x[i];
                xb[16 * i + l] = y[i];
            }
        }
        double an = fma(-t, ga, al), bn = fma(t, ga, be);
        // a norm that lost most of itself is summed afresh
        const bool fresh = rot && (an < 0.1 * al || bn < 0.1 * be);
        if (__any_sync(0xffffffffu, fresh)) {
            double u = 0.0, v = 0.0;
#pragma unroll
            for (int i = 0; i < NR; ++i) u = fma(x[i], x[i], u), v = fma(y[i], y[i], v);
            u = sum16(u);
            v = sum16(v);
            if (fresh) an = u, bn = v;
        }
        if (rot) {
            rotated = 1;
            if (l == 0) *na = an, *nb = bn;
        }
    };
    __syncthreads();
    for (; sweep < max_sweeps; ++sweep) {
        rotated = 0;
        for (int round = 0; round < 2 * JC - 1; ++round) {
            for (int c = g; c < 2 * JBM; c += JT / 16) {   // norms of the blocks as they are now (32 of 16 slots: two each)
                const int w = c / JBM, cc = c % JBM;
                double u = 0.0;
                if (cc < b)
                    for (int i = 0; i < NR; ++i) u = fma(col(buf, w, cc)[16 * i + l], col(buf, w, cc)[16 * i + l], u);
                u = sum16(u);
                if (cc < b && l == 0) nrm(buf, w)[cc] = u;
            }
            __syncthreads();
            if (round == 0) {
                // pairs within the blocks: slots 0-7 the first block, 8-15 the second
                const int bb = b + (b & 1), w = g / 8, p = g % 8;
                for (int st = 0; st < bb - 1; ++st) {
                    int a = (p == 0) ? 0 : 1 + (p - 1 + st) % (bb - 1);
                    int c = 1 + (bb - 2 - p + st) % (bb - 1);
                    const bool act = p < bb / 2 && a < b && c < b && a != c;
                    if (!act) a = c = 0;
                    pair(col(buf, w, min(a, c)), col(buf, w, max(a, c)), nrm(buf, w) + min(a, c),
                         nrm(buf, w) + max(a, c), act);
                    __syncthreads();
                }
            }
            for (int st = 0; st < b; ++st) {
                const bool act = g < b;
                const int a = act ? g : 0, c = act ? (g + st) % b : 0;
                pair(col(buf, 0, a), col(buf, 1, c), nrm(buf, 0) + a, nrm(buf, 1) + c, act);
                __syncthreads();
            }
            // the circle method's move: first block 0 stays, the first blocks move up, the second ones down
            const int t0 = rank == 0 ? 0 : min(rank + 1, JC - 1), w0 = rank == JC - 1 ? 1 : 0;
            const int t1 = rank == 0 ? 1 : rank - 1, w1 = rank == 0 ? 0 : 1;
            double *to0 = cluster.map_shared_rank(col(buf ^ 1, w0, 0), t0);
            double *to1 = cluster.map_shared_rank(col(buf ^ 1, w1, 0), t1);
            for (int e = threadIdx.x; e < b * ROWS; e += JT) {
                to0[e] = col(buf, 0, 0)[e];
                to1[e] = col(buf, 1, 0)[e];
            }
            if (round == 2 * JC - 2) {   // the sweep's end: did anything rotate anywhere?
                if (threadIdx.x == 0) mine = 0;
                __syncthreads();
                if (rotated) mine = 1;
                __syncthreads();
                if (threadIdx.x < JC) cluster.map_shared_rank(&flags[sweep & 1][0], threadIdx.x)[rank] = mine;
            }
            cluster.sync();
            buf ^= 1;
        }
        int any = 0;
        for (int k = 0; k < JC; ++k) any |= flags[sweep & 1][k];
        if (!any) break;   // the same decision in every CTA
    }
    // after whole sweeps the blocks are where they began
    for (int w = 0; w < 2; ++w)
        for (int c = g; c < JBM; c += JT / 16) {
            const int j = (w * JC + rank) * b + c;
            const bool in = c < b && j < r;
            double u = 0.0;
            if (in)
                for (int i = l; i < ROWS; i += 16) {
                    const double x = col(buf, w, c)[i];
                    u = fma(x, x, u);
                    if (i < r) s.M[(long long)j * ld + i] = x;
                }
            u = sum16(u);
            if (in && l == 0) s.sigma[j] = sqrt(u);
        }
    cluster.sync();   // no CTA leaves while another still writes its shared memory
}

// ---- Gaussian test matrices: counter-based SplitMix64 -> Box-Muller ---------
__device__ __forceinline__ unsigned long long splitmix(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void k_gaussian(double *O, long long n, unsigned long long seed) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (n + 1) / 2) return;
    const unsigned long long h1 = splitmix(seed ^ (2ull * t)), h2 = splitmix(seed ^ (2ull * t + 1));
    const double u1 = 1.0 - (double)(h1 >> 11) * (1.0 / 9007199254740992.0);
    const double u2 = (double)(h2 >> 11) * (1.0 / 9007199254740992.0);
    const double rad = sqrt(-2.0 * log(u1));
    O[2 * t] = rad * cos(6.283185307179586 * u2);
    if (2 * t + 1 < n) O[2 * t + 1] = rad * sin(6.283185307179586 * u2);
}

}  // namespace

static int device_sms() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        n <= 0)
        return 1;
    return n;
}

thread_local double *t_splitk_ws = nullptr;
thread_local size_t t_splitk_doubles = 0;

void bgemm_splitk_scratch(double *ws, size_t bytes) {
    t_splitk_ws = ws;
    t_splitk_doubles = ws ? bytes / sizeof(double) : 0;
}

// max_tiles: the largest number of 64 x 64 output tiles of one problem.  A
// problem has at most 4x (16x) as many 32 x 32 (16 x 16) tiles; the surplus
// CTAs of the smaller-tile grids return at once.  With fewer than two CTAs
// per SM on the small tiles, a K of at least 512 and a split-K scratch
// registered on this thread, the K loop is split over up to 16 CTAs per tile.
cudaError_t launch_bgemm(const GemmDesc *d_desc, int count, int max_tiles, cudaStream_t s, double flops, int kmax) {
    if (count <= 0 || max_tiles <= 0) return cudaSuccess;
    KScope ks(GEO_K_GEMM, s, flops, 0.0);
    const long long ctas = (long long)max_tiles * count;
    const long long sms = device_sms();
    if (ctas >= sms) {
        k_bgemm<<<dim3(max_tiles, count), 256, 0, s>>>(d_desc, count);
        return cudaGetLastError();
    }
    const int S = (4 * ctas >= sms) ? 2 : 1;
    const int W = 16 * S;
    const long long tiles_cap = (long long)(64 / W) * (64 / W) * max_tiles;
    int z = 1;
    if (kmax >= 512 && t_splitk_ws && tiles_cap * count < 2 * sms) {
        const long long want = (2 * sms + tiles_cap * count - 1) / (tiles_cap * count);
        z = (int)std::min<long long>(std::min<long long>(want, 16), kmax / 128);
        while (z >= 2 && (size_t)z * count * tiles_cap * W * W > t_splitk_doubles) --z;
    }
    double *ws = z >= 2 ? t_splitk_ws : nullptr;
    if (z < 2) z = 1;
    const dim3 grid((unsigned)tiles_cap, count, z);
    if (S == 2)
        k_bgemm_small<2><<<grid, 256, 0, s>>>(d_desc, count, z, (int)tiles_cap, ws);
    else
        k_bgemm_small<1><<<grid, 256, 0, s>>>(d_desc, count, z, (int)tiles_cap, ws);
    if (ws) {
        if (S == 2)
            k_bgemm_reduce<32><<<dim3((unsigned)tiles_cap, count), 256, 0, s>>>(d_desc, count, z, (int)tiles_cap, ws);
        else
            k_bgemm_reduce<16><<<dim3((unsigned)tiles_cap, count), 256, 0, s>>>(d_desc, count, z, (int)tiles_cap, ws);
    }
    return cudaGetLastError();
}

template <typename K, typename... A>
static cudaError_t launch_clusters(K kernel, int count, int ctas, int threads, size_t smem, cudaStream_t s, A... args) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)count * ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

bool house_qr_in_smem(int mmax, int rmax) { return rmax <= QR_MAX && house_qr_col_smem(mmax, rmax) <= 226 * 1024; }

cudaError_t launch_house_qr(const QrDesc *d_desc, int count, int mmax, int rmax, cudaStream_t s, double flops) {
    if (count <= 0) return cudaSuccess;
    KScope ks(GEO_K_TLR, s, flops, 0.0);
    // the block in a cluster's shared memory where it fits (m = 900: r = 240); else its rows over a cluster
    if (house_qr_in_smem(mmax, rmax))
        return launch_clusters(k_house_qr_col, count, QC, QCT, house_qr_col_smem(mmax, rmax), s, d_desc, count);
    if (rmax > QR_MAX) {
        k_house_qr<<<count, LA_THREADS, 0, s>>>(d_desc, count);
        return cudaGetLastError();
    }
    return launch_clusters(k_house_qr_cl, count, QC, QT, house_qr_cl_smem(mmax), s, d_desc, count);
}

cudaError_t launch_jacobi_svd(const SvdDesc *d_desc, int count, int max_sweeps, int rmax, cudaStream_t s,
                              double flops) {
    if (count <= 0) return cudaSuccess;
    KScope ks(GEO_K_TLR, s, flops, 0.0);
    if (rmax > JR_MAX) {
        k_jacobi_svd<<<count, LA_THREADS, 0, s>>>(d_desc, count, max_sweeps);
        return cudaGetLastError();
    }
    const int b = (rmax + 2 * JC - 1) / (2 * JC), nr = (rmax + 15) / 16;
    auto go = [&](auto NR) {
        return launch_clusters(k_jacobi_svd_cl<NR.value>, count, JC, JT, jacobi_cl_smem(b, 16 * NR.value), s, d_desc, count,
                               max_sweeps, b);
    };
    if (nr <= 4) return go(std::integral_constant<int, 4>());
    if (nr <= 8) return go(std::integral_constant<int, 8>());
    if (nr <= 12) return go(std::integral_constant<int, 12>());
    if (nr <= 14) return go(std::integral_constant<int, 14>());
    return go(std::integral_constant<int, 16>());
}

cudaError_t launch_gaussian(double *O, long long n, unsigned long long seed, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    KScope ks(GEO_K_AUX, s);
    const long long pairs = (n + 1) / 2;
    k_gaussian<<<(unsigned)((pairs + 255) / 256), 256, 0, s>>>(O, n, seed);
    return cudaGetLastError();
}
