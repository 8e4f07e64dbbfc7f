// One 32 x 32 tile of a Cholesky factorisation by a group of 128 threads: products of tile rows, the factor of a
// diagonal tile, the solve against it, and the progress words groups wait on (chol64.cu, batch.cu).
#pragma once

#include "geo_internal.cuh"

namespace {

constexpr int DT = 32;                 // tile edge
constexpr int DG = 128;                // threads per group
constexpr int DF_GROUPS = 4;           // groups per CTA: with one CTA per SM they fill the registers
constexpr int DF_THREADS = DG * DF_GROUPS;
constexpr int DLD = DT + 1;            // operand tiles: conflict-free along rows and columns
constexpr int DLL = DT + 2;            // the solve's copy of L_cc: 16-byte pairs
constexpr long long DF_WAIT_CYCLES = 4000000000LL;   // ~2 s at 2 GHz

struct DfSmem {
    double As[DT][DLD], Bs[DT][DLD];   // operand tiles [k][row]; Bs then holds the tile itself, [col][row]
    double Ls[DT][DLL];                // L_cc, [col][row]; the factorisation's exchange buffer
    double dinv[DT];                   // 1 / diagonal of L_cc
    int word[4];
};

__device__ __forceinline__ int df_ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// (after a barrier: releases what the whole group wrote)
__device__ __forceinline__ void df_st_release(int *p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

// Barrier of one group (named barriers 1 .. DF_GROUPS).
__device__ __forceinline__ void df_sync(int grp) { asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(DG) : "memory"); }

__device__ __forceinline__ void set_info(DevStatus *st, int row1) {
    // keep the smallest failing row
    int old = st->info;
    while (old == 0 || old > row1) {
        const int prev = atomicCAS(&st->info, old, row1);
        if (prev == old) break;
        old = prev;
    }
}

// Wait until min(*p, *q) >= need (one thread).  Returns that minimum, or -1 when the launch was aborted.  It gives up
// when neither these words nor the ticket counter sync[0] has moved for `limit` clocks: as long as tiles are taken the
// launch goes on, however few SMs it has (one tile takes well under a second).
__device__ int df_wait(const int *p, const int *q, int need, int *sync, int *timeout_word,
                       long long limit = DF_WAIT_CYCLES) {
    long long t0 = clock64();
    int last = -1, taken = -1;
    for (;;) {
        int v = df_ld_acquire(p);
        if (q != p) v = min(v, df_ld_acquire(q));
        if (v >= need) return v;
        if (df_ld_acquire(&sync[1])) return -1;
        const int t = df_ld_acquire(&sync[0]);
        if (v != last || t != taken) {
            last = v;
            taken = t;
            t0 = clock64();
        } else if (clock64() - t0 > limit) {
            atomicExch(&sync[1], 1);
            atomicCAS(timeout_word, 0, 8);
            return -1;
        }
        __nanosleep(20);
    }
}

// Half of a normal number well above the smallest one, off the FP64 pipe.
__device__ __forceinline__ double df_half(double x) {
    return __hiloint2double(__double2hiint(x) - (1 << 20), __double2loint(x));
}

// d > 0 and finite (false for a NaN), off the FP64 pipe.
__device__ __forceinline__ bool df_positive(double d) {
    const long long b = __double_as_longlong(d);
    return b > 0 && b < 0x7FF0000000000000LL;
}

// Pivots outside 2^-800 .. 2^900 would come too near the ends of the range for the approximations and residuals below
// (variances of 1e-300, say): a tile with such a diagonal entry (ext, the same in every thread) is factored as D S D
// with powers of two, which is exact.  The scale of a row by its diagonal entry; and one over it.
__device__ __forceinline__ double df_row_scale(double d) {
    const unsigned h = (unsigned)__double2hiint(d);   // (a negative d fails anyway)
    return __hiloint2double((1023 + (h < (1023u - 800u) << 20 ? 500 : h < (1023u + 900u) << 20 ? 0 : -450)) << 20, 0);
}
__device__ __forceinline__ double df_inv_scale(double s) { return __hiloint2double((2046 << 20) - __double2hiint(s), 0); }
__device__ __forceinline__ bool df_extreme(double d) {
    return (unsigned)__double2hiint(d) - ((1023u - 800u) << 20) >= (1700u << 20);
}

// l = sqrt(d) and inv = 1 / l for a d of 2^-960 .. 2^960, both as IEEE rounding gives them, by the method of
// P. Markstein ("Computation of elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34,
// 1990): the hardware's approximation of 1 / sqrt(d) (about 22 bits), one Newton step for the root and its reciprocal,
// and a correction of each by its residual, which an FMA gives exactly.  Before its last rounding each is within 2^-85
// or so of the value, so that only one a hair's breadth from the middle of two doubles could go the other way: none of
// 2^28 did over all those exponents.  The reciprocal's one exception is the method's: a root with a mantissa of ones,
// of a d one or two units below an even power of two, has its reciprocal one unit above the correction's result (which
// is a power of two), and d's bits show that before the chain begins.  A chain of seven
// dependent FP64 operations where sqrt() and a division take some twenty.
__device__ __forceinline__ void df_root(double d, double *l, double *inv) {
    double y0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(d));
    const double t = d * y0, e = fma(-t, df_half(y0), 0.5);   // (1 - d y0^2) / 2
    const double r = fma(t, e, t), y = fma(y0, e, y0);
    const bool below = (__double2hiint(d) & 0x1FFFFF) == 0xFFFFF && (unsigned)__double2loint(d) >= 0xFFFFFFFEu;
    const double root = fma(fma(-r, r, d), df_half(y), r), rec = fma(fma(-root, y, 1.0), y, y);
    *l = root;
    *inv = __hiloint2double(__double2hiint(rec), below ? 1 : __double2loint(rec));
}

// The factor of a scaled tile, and its diagonal's reciprocals, as the tile's own (each warp its columns).
__device__ __noinline__ void df_unscale(double (*S)[DLD], double *dinv, double sc, int lane, int w) {
    const double si = df_inv_scale(sc);
    for (int q = 0; q < 8; ++q) S[4 * q + w][lane] *= si;
    if (w == 0) dinv[lane] *= sc;
}

// Cholesky factor of the 32 x 32 block S[col][row] (lower part) by one group, lane = row, columns w, w + 4, ...
// in the registers of warp w.  Returns the first column without a positive pivot, or 32.  Panels of four
// columns: the warps exchange the panel through shared memory (one barrier), then every warp factors it for
// itself, so that no barrier or shared-memory round trip stands between its pivots, and applies it to its own
// columns, the next panel's first.  A dependent FP64 operation takes 66 clocks and every warp-wide one occupies
// its scheduler's FP64 unit for 64: one warp alone needs 38 us for the block, this 19.
// dinv receives the reciprocals of the factor's diagonal.  Pivots, roots and products are those of the plain
// right-looking algorithm, bit for bit (GEO_CHOL_BLOCK64).
__device__ __forceinline__ int df_potrf32_plain(double (*S)[DLD], double (*buf)[4][DT], double *dinv, int grp, int tid) {
    const int lane = tid & 31, w = tid >> 5;
    double v[8], p[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = S[4 * q + w][lane];
    // (nothing is written before the first barrier)
    const double dg = S[lane][lane];
    const bool ext = __any_sync(0xffffffffu, df_extreme(dg));
    double sc = 1.0;
    if (ext) {
        sc = df_row_scale(dg);
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] *= sc * __shfl_sync(0xffffffffu, sc, 4 * q + w);
    }
    int bad = DT;
#pragma unroll
    for (int P = 0; P < 8; ++P) {
        buf[P & 1][w][lane] = v[P];
        df_sync(grp);
        if (P > 0) {   // the previous panel on this warp's columns beyond this panel
#pragma unroll
            for (int q = P + 1; q < 8; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) v[q] = fma(-p[i], S[4 * (P - 1) + i][4 * q + w], v[q]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = buf[P & 1][i][lane];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = 4 * P + i;
            const double d = __shfl_sync(0xffffffffu, p[i], j);
            if (!df_positive(d) && bad == DT) bad = j;
            double l, inv;
            df_root(d, &l, &inv);
            p[i] = lane == j ? l : p[i] * inv;
            if (tid == j) dinv[j] = inv;
#pragma unroll
            for (int i2 = i + 1; i2 < 4; ++i2) p[i2] = fma(-p[i], __shfl_sync(0xffffffffu, p[i], 4 * P + i2), p[i2]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (w == i) S[4 * P + i][lane] = p[i];
            if (P < 7) v[(P + 1) % 8] = fma(-p[i], __shfl_sync(0xffffffffu, p[i], (4 * P + 4 + w) & 31), v[(P + 1) % 8]);
        }
    }
    if (ext) {
        df_sync(grp);   // every warp has read the columns
        df_unscale(S, dinv, sc, lane, w);
    }
    return bad;
}

// The same as L D L' first: the columns stay unscaled (u = l times the pivot's root) and are applied as
// (u / d) u', so that between two pivots stand a reciprocal approximation and four dependent FP64 operations
// instead of seven and a product; the 32 roots are taken together at the end, one per lane (12.5 us for the block).
__device__ __forceinline__ int df_potrf32(double (*S)[DLD], double (*buf)[4][DT], double *dinv, int grp, int tid) {
    const int lane = tid & 31, w = tid >> 5;
    double v[8], p[4] = {0.0, 0.0, 0.0, 0.0}, m[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = S[4 * q + w][lane];
    // (nothing is written before the first barrier)
    const double dg = S[lane][lane];
    const bool ext = __any_sync(0xffffffffu, df_extreme(dg));
    double sc = 1.0;
    if (ext) {
        sc = df_row_scale(dg);
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] *= sc * __shfl_sync(0xffffffffu, sc, 4 * q + w);
    }
#pragma unroll
    for (int P = 0; P < 8; ++P) {
        buf[P & 1][w][lane] = v[P];
        df_sync(grp);
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i] = buf[P & 1][i][lane];
        double f[4];   // this panel's multipliers
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double d = __shfl_sync(0xffffffffu, p[i], 4 * P + i);
            double r0;
            asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(d));
            const double e = fma(-d, r0, 1.0), f0 = p[i] * r0;
            f[i] = fma(f0, fma(e, e, e), f0);   // u / d: the approximation's error e to the third order
#pragma unroll
            for (int i2 = i + 1; i2 < 4; ++i2) p[i2] = fma(-f[i], __shfl_sync(0xffffffffu, p[i], 4 * P + i2), p[i2]);
            // the previous panel on this warp's columns beyond this one, in the chain's gaps
            if (P > 0)
#pragma unroll
                for (int q = P + 1; q < 8; ++q) v[q] = fma(-m[i], S[4 * (P - 1) + i][4 * q + w], v[q]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            m[i] = f[i];
            if (w == i) S[4 * P + i][lane] = p[i];
            if (P < 7) v[(P + 1) % 8] = fma(-m[i], __shfl_sync(0xffffffffu, p[i], (4 * P + 4 + w) & 31), v[(P + 1) % 8]);
        }
    }
    df_sync(grp);
    // the roots and their reciprocals, in every warp for itself
    const double d = S[lane][lane];
    const unsigned ok = __ballot_sync(0xffffffffu, df_positive(d));
    double l, inv;
    df_root(d, &l, &inv);
    if (w == 0) dinv[lane] = inv;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int col = 4 * q + w;
        const double iv = __shfl_sync(0xffffffffu, inv, col);
        v[q] = lane == col ? l : S[col][lane] * iv;
    }
    df_sync(grp);   // every warp has read the diagonal
#pragma unroll
    for (int q = 0; q < 8; ++q) S[4 * q + w][lane] = v[q];
    if (ext) df_unscale(S, dinv, sc, lane, w);
    return ok == 0xffffffffu ? DT : __ffs(~ok) - 1;
}

// X <- X L^-T for the 32 x 32 tiles X[col][row] and L[col][row] by one group: warp w takes rows 8 w .. 8 w + 7,
// lane = row + 8 g holds the columns g, g + 4, ... of its row; x_m goes from its lane to the row's four lanes
// by shuffle, so the warps never wait for one another.  dinv: 1 / L_mm.
__device__ __forceinline__ void df_trsm32(double (*X)[DLD], const double (*L)[DLL], const double *dinv, int tid) {
    const int lane = tid & 31, g = lane >> 3, row = 8 * (tid >> 5) + (lane & 7);
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = X[4 * i + g][row];
#pragma unroll
    for (int m = 0; m < DT; ++m) {
        const int im = m / 4, gm = m % 4;
        const double xm = __shfl_sync(0xffffffffu, x[im] * dinv[m], (lane & 7) + 8 * gm);
        if (g == gm) X[m][row] = xm;
#pragma unroll
        for (int i = im; i < 8; ++i) {
            if (i == im && gm == 3) continue;
            const double y = fma(-xm, L[m][4 * i + g], x[i]);
            x[i] = (i == im && g <= gm) ? x[i] : y;
        }
    }
}

// The same with the scaled factor H[m][k] = L_km / L_mm in place of L: the unscaled x_m goes out as it is (one
// dependent operation per column instead of two), and the row is scaled once at the end.
__device__ __forceinline__ void df_trsm32_scaled(double (*X)[DLD], const double (*H)[DLL], const double *dinv, int tid) {
    const int lane = tid & 31, g = lane >> 3, row = 8 * (tid >> 5) + (lane & 7);
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = X[4 * i + g][row];
#pragma unroll
    for (int m = 0; m < DT; ++m) {
        const int im = m / 4, gm = m % 4;
        const double xm = __shfl_sync(0xffffffffu, x[im], (lane & 7) + 8 * gm);
#pragma unroll
        for (int i = im; i < 8; ++i) {
            if (i == im && gm == 3) continue;
            const double y = fma(-xm, H[m][4 * i + g], x[i]);
            x[i] = (i == im && g <= gm) ? x[i] : y;
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) X[4 * i + g][row] = x[i] * dinv[4 * i + g];
}

// Products of a 32-deep slice, acc += A-tile times B-tile': rows ty + 8 i, columns tx + 16 j.
template <int IM>
__device__ __forceinline__ void df_mma(double (&acc)[8], const double (*As)[DLD], const double (*Bs)[DLD], int tx,
                                       int ty) {
#pragma unroll 8
    for (int kk = 0; kk < DT; ++kk) {
        double a[IM], b[2];
#pragma unroll
        for (int i = 0; i < IM; ++i) a[i] = As[kk][ty + 8 * i];
#pragma unroll
        for (int j = 0; j < 2; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < IM; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) acc[2 * i + j] = fma(a[i], b[j], acc[2 * i + j]);
    }
}

// The same for a diagonal tile, of which only the ten 8 x 8 blocks at or below the diagonal are formed: five
// entries a thread instead of eight.
__device__ __forceinline__ void df_mma_diag(double (&acc)[8], const double (*As)[DLD], const int (&dr)[5],
                                            const int (&dc)[5]) {
#pragma unroll 8
    for (int kk = 0; kk < DT; ++kk)
#pragma unroll
        for (int i = 0; i < 5; ++i) acc[i] = fma(As[kk][dr[i]], As[kk][dc[i]], acc[i]);
}

// A thread's five entries of a diagonal tile: one of the 64 of every other 8 x 8 block of its lower part.
__device__ __forceinline__ void df_diag_entries(int tid, int (&dr)[5], int (&dc)[5]) {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int b = 2 * i + tid / 64, bi = b < 1 ? 0 : b < 3 ? 1 : b < 6 ? 2 : 3, bj = b - bi * (bi + 1) / 2;
        dr[i] = 8 * bi + tid % 8;
        dc[i] = 8 * bj + tid % 64 / 8;
    }
}

// The finished diagonal tile at L (cb columns) into sm.Ls, columns scaled by the reciprocals of the diagonal
// (also in sm.dinv), as the identity past cb.
__device__ __forceinline__ void df_load_scaled(DfSmem &sm, const double *L, long long ld, int cb, int grp, int tid) {
    const int lr = tid % 32, lc = tid / 32;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int col = lc + 4 * u;
        v[u] = (lr < cb && col < cb && lr >= col) ? __ldcg(L + (long long)col * ld + lr) : (lr == col ? 1.0 : 0.0);
    }
    if (tid < DT) sm.dinv[tid] = tid < cb ? 1.0 / __ldcg(L + (long long)tid * ld + tid) : 1.0;
    df_sync(grp);
#pragma unroll
    for (int u = 0; u < 8; ++u) sm.Ls[lc + 4 * u][lr] = v[u] * sm.dinv[lc + 4 * u];
    df_sync(grp);
}

int df_sms() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
        return 1;
    return n;
}

}  // namespace
