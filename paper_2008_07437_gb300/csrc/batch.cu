// Batched evaluation of many small, uneven Eq. 1 likelihoods (dense FP64).
//
// One launch builds the tables of every problem's theta; ONE persistent launch
// does the rest.  Its unit is a 32 x 32 tile of one problem's matrix (the tile
// code of chol64.cu): generated from Eq. 2 on the spot, brought up to date with
// the finished columns before it in registers, factored or solved, written
// once; the observations ride along as an extra row, and a last unit per
// problem sums up its log-determinant and quadratic form.  Groups of 128
// threads take units from a ticket table and wait on progress words, one per
// tile row of each problem.  The table runs over the columns of all problems
// together, those with most columns left first: between two columns of one
// problem lie the same-numbered columns of all the others, so that a unit's
// inputs are finished long before its turn, and the problems end together.
// Within a problem a unit only waits for units earlier in the table, whose
// groups are running, so the launch cannot deadlock; waits are bounded.  Every
// per-problem quantity lives in a device descriptor array, so the launch
// sequence of a batch shape is captured once as a CUDA graph and replayed with
// new inputs and theta by refreshing the descriptors.  Each problem's result
// depends only on its own data and a fixed operation order: a likelihood is
// bit-identical alone and inside any batch.
//
// Bound by the FP64 pipe: 512 problems of 50 to 1,000 bivariate locations (one draw) take
// 346 ms (461 with 64-wide panels, a barrier between a problem's phases and the
// covariance as units of its own); their N^3 / 3 alone takes about 310.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "chol_tile.cuh"
#include "cov_tables.cuh"

namespace {

struct BatchDesc {
    double *A;            // column-major, ld, N columns; row N receives y'
    long long ld;
    int N, n;
    const double *locs;   // n x 2 (caller order)
    const double *z;      // N
    CovParams cp;
    DevStatus st;         // per-problem status
    DevResults res;
};

constexpr int B_REDUCE = 0xFFFF;   // tile column of a problem's last unit

struct BSmem {
    DfSmem t;
    CovParams cp;                  // the unit's problem
    double red[2][DG / 32];
};

// The 32 x 32 tile of Sigma from row 32 i and column 32 c into S[col][row], by location pairs where the tile's
// edge is a multiple of P, else entry by entry; zeros past the matrix.
template <int P>
__device__ __forceinline__ void b_cov_tile(double (*S)[DLD], const CovParams &cp, const double *__restrict__ locs, int n,
                                           int i, int c, int tid) {
    if constexpr (DT % P == 0) {
        constexpr int LT = DT / P;   // locations along a tile's edge
        for (int e = tid; e < LT * LT; e += DG) {
            const int lr = e % LT, lc = e / LT, l = i * LT + lr, r = c * LT + lc;
            double v[P * P];
            if (l < n && r < n) {
                const double dx = locs[2 * l] - locs[2 * r], dy = locs[2 * l + 1] - locs[2 * r + 1];
                matern_pair<P>(l == r ? 0.0 : fma(dx, dx, dy * dy), cp, v);
            } else {
#pragma unroll
                for (int q = 0; q < P * P; ++q) v[q] = 0.0;
            }
#pragma unroll
            for (int q = 0; q < P * P; ++q) S[P * lc + q % P][P * lr + q / P] = v[q];
        }
    } else {
        for (int e = tid; e < DT * DT; e += DG) {
            const int R = i * DT + e % DT, C = c * DT + e / DT, l = R / P, r = C / P;
            double v = 0.0;
            if (l < n && r < n) {
                const double dx = locs[2 * l] - locs[2 * r], dy = locs[2 * l + 1] - locs[2 * r + 1];
                v = matern_entry(l == r ? 0.0 : fma(dx, dx, dy * dy), cp, R % P, C % P);
            }
            S[e / DT][e % DT] = v;
        }
    }
}

// The tables of every problem's theta.
__global__ void __launch_bounds__(128) k_b_tables(BatchDesc *d) {
    const CovParams &cp = d[blockIdx.z].cp;
    if ((int)blockIdx.x >= cp.p * (cp.p + 1) / 2) return;
    fine_build_block(cp, const_cast<double *>(cp.tab), const_cast<double *>(cp.fine), blockIdx.x, blockIdx.y);
}

// sync: {ticket, abort, timeout, unused}, then `stride` progress words per problem: one per tile row, the
// observations' row last.  units[t] = {problem, tile column << 16 | tile row}.
__global__ void __launch_bounds__(DF_THREADS, 1) k_b_persistent(BatchDesc *d, const int2 *__restrict__ units,
                                                                const int *nunits_p, int *sync, int stride) {
    extern __shared__ __align__(16) unsigned char b_smem[];
    const int grp = threadIdx.x / DG, tid = threadIdx.x % DG;
    BSmem &bs = reinterpret_cast<BSmem *>(b_smem)[grp];
    DfSmem &sm = bs.t;
    const int tx = tid % 16, ty = tid / 16, lr = tid % 32, lc = tid / 32;
    const int nunits = *nunits_p;
    int dr[5], dc[5];
    df_diag_entries(tid, dr, dc);
    for (;;) {
        if (tid == 0) {
            const int t = df_ld_acquire(&sync[1]) ? nunits : atomicAdd(&sync[0], 1);
            const int2 u = t < nunits ? units[t] : make_int2(-1, 0);
            sm.word[0] = u.x;
            sm.word[1] = u.y;
            sm.word[3] = u.x >= 0 && df_ld_acquire(&d[u.x].st.info);
        }
        df_sync(grp);
        const int p = sm.word[0];
        if (p < 0) return;
        const int c = sm.word[1] >> 16 & 0xFFFF, i = sm.word[1] & 0xFFFF;
        BatchDesc &q = d[p];
        const int N = q.N, T = (N + DT - 1) / DT;
        int *prog = sync + 4 + (long long)p * stride;
        if (c == B_REDUCE) {
            if (tid == 0) sm.word[2] = df_wait(&prog[T], &prog[T - 1], T, sync, &sync[2]);
            df_sync(grp);
            if (sm.word[2] < 0) return;
            double a = 0.0, b = 0.0;
            for (int k = tid; k < N; k += DG) {
                a += log(__ldcg(q.A + (long long)k * q.ld + k));
                const double v = __ldcg(q.A + (long long)k * q.ld + N);
                b += v * v;
            }
            for (int o = 16; o > 0; o >>= 1) {
                a += __shfl_down_sync(0xffffffffu, a, o);
                b += __shfl_down_sync(0xffffffffu, b, o);
            }
            if (lr == 0) bs.red[0][lc] = a, bs.red[1][lc] = b;
            df_sync(grp);
            if (tid == 0) {
                double ta = 0.0, tb = 0.0;
                for (int w = 0; w < DG / 32; ++w) ta += bs.red[0][w], tb += bs.red[1][w];
                if (df_ld_acquire(&q.st.info)) {
                    q.res.loglik = q.res.logdet = q.res.quad = nan("");
                } else {
                    q.res.logdet = 2.0 * ta;
                    q.res.quad = tb;
                    q.res.loglik = -0.5 * (double)N * log(2.0 * 3.141592653589793) - 0.5 * q.res.logdet - 0.5 * tb;
                }
            }
            df_sync(grp);
            continue;
        }
        int *prow = &prog[i], *pcol = &prog[c];
        if (sm.word[3]) {   // a pivot of this problem has failed: its units only pass their turn on, in order
            if (tid == 0) {
                sm.word[2] = df_wait(prow, prow, c, sync, &sync[2]);
                if (sm.word[2] >= 0) df_st_release(prow, c + 1);
            }
            df_sync(grp);
            if (sm.word[2] < 0) return;
            continue;
        }
        const bool diag = i == c, obs = i == T;
        const int c0 = DT * c, cb = min(DT, N - c0), r0 = obs ? N : DT * i, nr = obs ? 1 : min(DT, N - r0);
        // the tile as it starts
        if (obs) {
#pragma unroll
            for (int u = 0; u < 8; ++u) sm.Bs[lc + 4 * u][lr] = (lr == 0 && lc + 4 * u < cb) ? q.z[c0 + lc + 4 * u] : 0.0;
        } else {
            const int words = (int)(sizeof(CovParams) / sizeof(int));
            const int *src = reinterpret_cast<const int *>(&q.cp);
            int *dst = reinterpret_cast<int *>(&bs.cp);
            for (int t = tid; t < words; t += DG) dst[t] = src[t];
            df_sync(grp);
            switch (bs.cp.p) {
                case 1: b_cov_tile<1>(sm.Bs, bs.cp, q.locs, q.n, i, c, tid); break;
                case 2: b_cov_tile<2>(sm.Bs, bs.cp, q.locs, q.n, i, c, tid); break;
                case 3: b_cov_tile<3>(sm.Bs, bs.cp, q.locs, q.n, i, c, tid); break;
                default: b_cov_tile<4>(sm.Bs, bs.cp, q.locs, q.n, i, c, tid); break;
            }
        }
        df_sync(grp);
        double acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
            acc[e] = diag ? (e < 5 ? -sm.Bs[dc[e % 5]][dr[e % 5]] : 0.0) : -sm.Bs[tx + 16 * (e % 2)][ty + 8 * (e / 2)];
        df_sync(grp);
        double pa[8], pb[8];
        auto load = [&](int k) {
            const long long kc = DT * k;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const double *col = q.A + (kc + lc + 4 * u) * q.ld + lr;
                pa[u] = lr < nr ? __ldcg(col + r0) : 0.0;
                if (!diag) pb[u] = lr < cb ? __ldcg(col + c0) : 0.0;
            }
        };
        int avail = 0;
        for (int k = 0; k < c; ++k) {
            if (avail <= k) {
                if (tid == 0) sm.word[2] = df_wait(prow, pcol, k + 1, sync, &sync[2]);
                df_sync(grp);
                avail = sm.word[2];
                if (avail < 0) return;
                load(k);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                sm.As[lc + 4 * u][lr] = pa[u];
                if (!diag) sm.Bs[lc + 4 * u][lr] = pb[u];
            }
            df_sync(grp);
            if (k + 1 < c && avail > k + 1) load(k + 1);   // in flight during the products
            if (diag)
                df_mma_diag(acc, sm.As, dr, dc);
            else if (nr <= 8)
                df_mma<1>(acc, sm.As, sm.Bs, tx, ty);
            else
                df_mma<4>(acc, sm.As, sm.Bs, tx, ty);
            df_sync(grp);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (!diag)
                sm.Bs[tx + 16 * (e % 2)][ty + 8 * (e / 2)] = -acc[e];
            else if (e < 5)
                sm.Bs[dc[e % 5]][dr[e % 5]] =
                    (dr[e % 5] < cb && dc[e % 5] < cb) ? -acc[e] : (dr[e % 5] == dc[e % 5] ? 1.0 : 0.0);
        }
        df_sync(grp);
        if (diag) {
            const int bad = df_potrf32(sm.Bs, reinterpret_cast<double (*)[4][DT]>(sm.Ls), sm.dinv, grp, tid);
            // the first failing row stays; units that are under way go on with what they find, nothing reads it
            if (bad < cb && tid == 0) atomicCAS(&q.st.info, 0, c0 + bad + 1);
            df_sync(grp);
        } else {
            if (tid == 0) sm.word[2] = df_wait(pcol, pcol, c + 1, sync, &sync[2]);
            df_sync(grp);
            if (sm.word[2] < 0) return;
            df_load_scaled(sm, q.A + (long long)c0 * q.ld + c0, q.ld, cb, grp, tid);
            df_trsm32_scaled(sm.Bs, sm.Ls, sm.dinv, tid);
            df_sync(grp);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int col = lc + 4 * u;
            if (lr < nr && col < cb && (!diag || lr >= col)) q.A[(long long)(c0 + col) * q.ld + r0 + lr] = sm.Bs[col][lr];
        }
        df_sync(grp);
        if (tid == 0) df_st_release(prow, c + 1);
    }
}

}  // namespace

size_t batch_desc_bytes() { return sizeof(BatchDesc); }

// With the GPU full of problems the tables cost their FP64 operations, 3 million a C_ij, against some 55 saved per
// pair of locations: they pay from about 340 locations on.
size_t batch_fine_doubles(const CovParams &cp, int n) { return n >= 340 ? cov_fine_doubles(cp, 0.5 * n * (n + 1.0)) : 0; }

long long batch_units(const int *N, int count, void *out_v) {
    int2 *out = (int2 *)out_v;
    long long total = 0;
    int Tmax = 0;
    for (int q = 0; q < count; ++q) {
        const long long T = (N[q] + DT - 1) / DT;
        total += T * (T + 1) / 2 + T + 1;   // tiles, the observations' tiles, the reduction
        Tmax = std::max(Tmax, (int)T);
    }
    if (!out) return total;
    // problems by their number of columns, the largest first
    std::vector<int> by(count);
    for (int q = 0; q < count; ++q) by[q] = q;
    std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return (N[a] + DT - 1) / DT > (N[b] + DT - 1) / DT; });
    long long n = 0;
    int active = 0;
    for (int left = Tmax; left >= 1; --left) {   // columns left, this one included
        while (active < count && (N[by[active]] + DT - 1) / DT >= left) ++active;
        for (int a = 0; a < active; ++a) {
            const int q = by[a], T = (N[q] + DT - 1) / DT, c = T - left;
            for (int i = c; i <= T; ++i) out[n++] = make_int2(q, c << 16 | i);
        }
    }
    for (int a = 0; a < count; ++a) out[n++] = make_int2(by[a], B_REDUCE << 16);
    return n;
}

static int batch_stride(int Nmax) { return (Nmax + DT - 1) / DT + 1; }

size_t batch_sync_ints(int count, int Nmax) { return 4 + (size_t)count * batch_stride(Nmax); }

void batch_fill_desc(void *hdesc_v, int k, double *A, long long ld, int N, int n, const double *locs,
                     const double *z, const CovParams &cp) {
    BatchDesc *h = (BatchDesc *)hdesc_v;
    memset(&h[k], 0, sizeof(BatchDesc));
    h[k].A = A;
    h[k].ld = ld;
    h[k].N = N;
    h[k].n = n;
    h[k].locs = locs;
    h[k].z = z;
    h[k].cp = cp;
}

cudaError_t batch_record(void *ddesc_v, const void *units, const int *nunits, int *sync, int count, int pmax, int Nmax,
                         cudaStream_t s) {
    BatchDesc *d = (BatchDesc *)ddesc_v;
    cudaError_t e = cudaMemsetAsync(sync, 0, sizeof(int) * batch_sync_ints(count, Nmax), s);
    if (e != cudaSuccess) return e;
    {
        KScope ks(GEO_K_COVGEN, s);
        k_b_tables<<<dim3(pmax * (pmax + 1) / 2, FINE_BLOCKS + COARSE_BLOCKS, count), 128, 0, s>>>(d);
    }
    {
        KScope ks(GEO_K_GEMM, s);
        constexpr size_t smem = sizeof(BSmem) * DF_GROUPS;
        if ((e = cudaFuncSetAttribute(k_b_persistent, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
            return e;
        k_b_persistent<<<df_sms(), DF_THREADS, smem, s>>>(d, (const int2 *)units, nunits, sync, batch_stride(Nmax));
    }
    return cudaGetLastError();
}

// Results out of the device descriptors into host arrays (after the stream syncs).
cudaError_t batch_results(const void *ddesc_v, void *hdesc_v, int count, double *loglik, int *info, cudaStream_t s) {
    const BatchDesc *d = (const BatchDesc *)ddesc_v;
    BatchDesc *h = (BatchDesc *)hdesc_v;
    cudaError_t e = cudaMemcpyAsync(h, d, sizeof(BatchDesc) * count, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    for (int k = 0; k < count; ++k) {
        if (loglik) loglik[k] = h[k].res.loglik;
        if (info) info[k] = h[k].st.info;
    }
    return cudaSuccess;
}
