// Dense FP64 tiled Cholesky, Sigma = L L' (Sec. 5.2; the tile algorithm of
// Sec. 5.1 / Fig. 1 / Fig. 2: POTRF on the diagonal tile, TRSM on the panel,
// SYRK / GEMM on the trailing matrix), as one data-flow launch.
//
// On GB300 the FP64 pipe runs at about 1.2 TFLOP/s (two FP64 FMAs per clock
// per SM, a warp-wide FMA every 16 clocks), some 60x below the FP32 pipe.  So
// memory never sets the pace -- a 32 x 32 output tile reads 16 bytes per 32
// FMAs, one byte per clock and SM -- and tiles can be small, which is what the
// latency of the column chain asks for: a 64-wide diagonal block costs one SM
// at least 11 us of FP64 issue, the 64 x 64 solve below it 32 us, while the
// 32-wide ones take 4 and 4.
//
// The matrix is cut into 32 x 32 tiles.  Groups of 128 threads (four to a CTA,
// one CTA per SM) take tiles from a ticket counter, column by column, and do
// everything for a tile at once, left-looking: C_ic = A_ic - sum_k L_ik L_ck'
// in registers over the finished tiles k < c of the two tile rows, then the
// Cholesky factor of the 32 x 32 block (i = c) or the solve with L_cc'
// (i > c).  The tile is written once; only with a column chain (df_chain) the
// diagonal tiles and those below them are written up to date first and
// finished by the chain.  A progress word per tile row counts its finished
// tiles; a group waits on the words of its two rows, so tiles of later columns
// accumulate while the column chain runs (lookahead without streams).
//
// The launch ends whatever the number of resident CTAs, down to one: a group
// waits for tiles whose tickets were taken earlier by groups that are running,
// or for the chain, which takes the first ticket and waits in column order for
// tiles that later tickets bring up to date.  So some other group has to go on
// taking tickets, and the groups that would leave the SM to the chain (or are
// spare) only leave once a second CTA has started: its first group stays to
// the end.  Every wait is bounded: past DF_WAIT_CYCLES without progress the
// waiter raises the abort word, records the timeout and all groups return; a failed
// pivot raises the same word.  Sums run in a fixed order: results do not
// depend on timing.
//
// Rows N .. nrows-1 are extra right-hand-side rows: tiles of their own that
// take part in every product and solve, so row N ends up holding (L^-1 z)'
// when it starts as z' (the forward substitution of Eq. 1 comes out of the
// factorisation).  The inverse of a diagonal tile (for the emulated form's
// panel solves) is the solve of identity rows carried along the same way.
//
// Bounds: small orders by the column chain (34 us per 32 columns: 12.5 the
// block's factorisation, 6.3 the solve below it, 6.6 the product, the rest
// memory and flags), large ones by the FP64 pipe.  Measured, against one
// launch per step of a 64-wide blocked algorithm (POTRF in one CTA 97 us, TRSM
// 65, rank-64 update 100 and more): N = 800 0.85 ms (3.5), N = 8,002 145 ms
// = 0.93 of the pipe (172), a 512-column diagonal tile with its inverse beside
// other work 0.55 ms (1.6), 24 tiles of 256 in the mixed form 10 ms (24).
// Four groups of 128 threads share a CTA because one CTA per SM keeps the
// SMs of a concurrent persistent kernel free, and 128 threads reach all four
// FP64 units of an SM with eight entries each.
#include <algorithm>

#include "chol_tile.cuh"

namespace {

struct DfArgs {
    double *A;
    long long ld;
    int j0, jb;       // columns of the panel (the diagonal tile's rows are the same range)
    double *X;        // extra rows x = 0 .. nx - 1: column j of the matrix at X[j * ldx + x]
    long long ldx;
    int nx;
    int T, E;         // 32-wide column tiles; tiles of extra rows
    int factor;       // 0: the diagonal range already holds L, only the extra rows are solved
    double *W;        // not null: W = -L^-1 of the diagonal range (column-major, ldw, zeros above the diagonal)
    long long ldw;
    int *sync;        // {ticket, abort, CTAs started, progress words: T + E (+ T with W), with chain: ready words 2 T}
    int tickets;
    int chain;        // 1: one group runs the column chain (df_chain)
    int alone;        // chain: the other groups of its CTA leave it the SM (once a second CTA runs)
    int block64;      // GEO_CHOL_BLOCK64: no chain
    int plain;        // GEO_CHOL_BLOCK64 and GEO_CHOL_PLAIN: pivots and solves as the plain algorithm rounds them
    DevStatus *st;
    long long limit;  // clocks without progress after which a wait gives up
};

constexpr int DF_HEAD = 3;   // sync words before the progress words
constexpr int DF_SUM = 2;    // tile columns whose products are summed on their own

// The column chain, by one group: for every column c the last product of the diagonal tile (with L_c,c-1, which
// this group has just solved and still holds), its factorisation, and the solve of the tile below it.  Handing
// these three from group to group costs two trips through L2 (3.5 us each) per 32 columns; the other groups
// bring the two tiles up to date with the columns before and say so in the ready words.
template <bool PLAIN>
__device__ __noinline__ void df_chain(const DfArgs &a, DfSmem &sm, int grp, int tid, const int (&dr)[5],
                                      const int (&dc)[5]) {
    const int lr = tid % 32, lc = tid / 32;
    int *prog = a.sync + DF_HEAD, *ready = prog + a.T + a.E + (a.W ? a.T : 0);
    for (int c = 0; c < a.T; ++c) {
        const int c0 = a.j0 + DT * c, cb = min(DT, a.j0 + a.jb - c0);
        if (c >= 2) {   // the diagonal tile holds the products of the columns before c - 1
            if (tid == 0) sm.word[1] = df_wait(&ready[2 * c], &ready[2 * c], 1, a.sync, &a.st->timeout, a.limit);
            df_sync(grp);
            if (sm.word[1] < 0) return;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int col = lc + 4 * u;
            sm.Bs[col][lr] = (lr < cb && col < cb) ? __ldcg(a.A + (long long)(c0 + col) * a.ld + c0 + lr) : 0.0;
        }
        df_sync(grp);
        double acc[8];
#pragma unroll
        for (int i = 0; i < 5; ++i) acc[i] = c % DF_SUM ? -sm.Bs[dc[i]][dr[i]] : 0.0;
        if (c > 0) df_mma_diag(acc, sm.As, dr, dc);
        if (c % DF_SUM == 0)   // column c - 1 is the end of an earlier block: a sum of its own
#pragma unroll
            for (int i = 0; i < 5; ++i) acc[i] -= sm.Bs[dc[i]][dr[i]];
        df_sync(grp);
#pragma unroll
        for (int i = 0; i < 5; ++i)
            sm.Bs[dc[i]][dr[i]] = (dr[i] < cb && dc[i] < cb) ? -acc[i] : (dr[i] == dc[i] ? 1.0 : 0.0);
        df_sync(grp);
        auto *buf = reinterpret_cast<double (*)[4][DT]>(sm.Ls);
        const int bad = PLAIN ? df_potrf32_plain(sm.Bs, buf, sm.dinv, grp, tid)
                              : df_potrf32(sm.Bs, buf, sm.dinv, grp, tid);
        if (bad < cb) {
            if (tid == 0) {
                set_info(a.st, c0 + bad + 1);
                __threadfence();
                atomicExch(&a.sync[1], 1);
            }
            return;
        }
        df_sync(grp);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int col = lc + 4 * u;
            const double v = sm.Bs[col][lr];
            if (lr < cb && col < cb && lr >= col) a.A[(long long)(c0 + col) * a.ld + c0 + lr] = v;
            sm.Ls[col][lr] = lr >= col ? (PLAIN ? v : v * sm.dinv[col]) : 0.0;
        }
        df_sync(grp);
        if (tid == 0) df_st_release(&prog[c], c + 1);
        if (c + 1 == a.T) return;
        const int r0 = c0 + DT, nr = min(DT, a.j0 + a.jb - r0);
        if (c >= 1) {   // the tile below holds the products of the columns before c
            if (tid == 32) sm.word[1] = df_wait(&ready[2 * c + 1], &ready[2 * c + 1], 1, a.sync, &a.st->timeout, a.limit);
            df_sync(grp);
            if (sm.word[1] < 0) return;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int col = lc + 4 * u;
            sm.As[col][lr] = lr < nr ? __ldcg(a.A + (long long)(c0 + col) * a.ld + r0 + lr) : 0.0;
        }
        df_sync(grp);
        if (PLAIN)
            df_trsm32(sm.As, sm.Ls, sm.dinv, tid);
        else
            df_trsm32_scaled(sm.As, sm.Ls, sm.dinv, tid);
        df_sync(grp);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int col = lc + 4 * u;
            if (lr < nr) a.A[(long long)(c0 + col) * a.ld + r0 + lr] = sm.As[col][lr];
        }
        df_sync(grp);
        if (tid == 0) df_st_release(&prog[c + 1], c + 1);
    }
}

template <bool PLAIN>
__global__ void __launch_bounds__(DF_THREADS, 1) k_chol_df(const DfArgs a) {
    extern __shared__ __align__(16) unsigned char df_smem[];
    const int grp = threadIdx.x / DG, tid = threadIdx.x % DG;
    DfSmem &sm = reinterpret_cast<DfSmem *>(df_smem)[grp];
    const int tx = tid % 16, ty = tid / 16, lr = tid % 32, lc = tid / 32;
    int *prog = a.sync + DF_HEAD;
    int dr[5], dc[5];
    df_diag_entries(tid, dr, dc);
    __shared__ int chain_here;   // this CTA runs the column chain
    if (threadIdx.x == 0) {
        chain_here = 0;
        if (a.chain) atomicAdd(&a.sync[2], 1);
    }
    __syncthreads();
    // with few tiles, fewer groups to an SM share its FP64 pipe
    const bool spare = (long long)grp * gridDim.x >= a.tickets;
    if (spare && !a.chain) return;
    if (spare && tid == 0)   // the other CTAs start within a microsecond, if there is room for them
        for (int i = 0; i < 40 && df_ld_acquire(&a.sync[2]) < 2; ++i) __nanosleep(50);
    for (;;) {
        // stop after a failed pivot (of this launch or an earlier one) or an expired wait
        if (tid == 0) {
            const bool stop = df_ld_acquire(&a.sync[1]) || df_ld_acquire(&a.st->info) ||
                              ((spare || (a.alone && *(volatile int *)&chain_here)) && df_ld_acquire(&a.sync[2]) > 1);
            sm.word[0] = stop ? a.tickets : atomicAdd(&a.sync[0], 1) - a.chain;
            if (sm.word[0] < 0) *(volatile int *)&chain_here = 1;
        }
        df_sync(grp);
        const int t = sm.word[0];
        if (t >= a.tickets) return;
        if (t < 0) {   // the first ticket of a launch with a chain
            df_chain<PLAIN>(a, sm, grp, tid, dr, dc);
            return;
        }
        // tile column c, and tile row: of the diagonal range (kind 0), the extra rows (1) or the identity rows (2)
        int c, q;
        if (!a.factor && a.W) {   // the inverse alone: column c has the identity rows 0 .. c
            c = max(0, (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5) - 1);
            while ((c + 1) * (c + 2) / 2 <= t) ++c;
            q = t - c * (c + 1) / 2 + a.T + a.E;
        } else if (!a.factor) {
            c = t / a.E;
            q = t % a.E + a.T;
        } else if (a.W) {
            c = t / (a.T + a.E + 1);
            q = t % (a.T + a.E + 1) + c;
        } else {
            // column c starts at ticket c (T + E) - c (c - 1) / 2
            const double b = a.T + a.E + 0.5;
            c = max(0, min(a.T - 1, (int)(b - sqrt(b * b - 2.0 * t))));
            auto start = [&](int cc) { return cc * (a.T + a.E) - cc * (cc - 1) / 2; };
            while (c > 0 && start(c) > t) --c;
            while (c + 1 < a.T && start(c + 1) <= t) ++c;
            q = t - start(c) + c;
        }
        const int kind = q < a.T ? 0 : q < a.T + a.E ? 1 : 2;
        const int e = q - (kind == 1 ? a.T : kind == 2 ? a.T + a.E : 0);   // tile row within its kind
        const int c0 = a.j0 + DT * c, cb = min(DT, a.j0 + a.jb - c0);
        const int r0 = kind == 1 ? DT * e : a.j0 + DT * e;   // first row (of X, the matrix, the unit part)
        const int nr = min(DT, (kind == 1 ? a.nx : a.j0 + a.jb) - r0);
        double *R = kind == 1 ? a.X : a.A;
        const long long rld = kind == 1 ? a.ldx : a.ld;
        const bool diag = kind == 0 && e == c;
        // with a chain, the diagonal tile and the one below it are only brought up to date here
        const bool pre = a.chain && kind == 0 && e <= c + 1;
        const int kend = pre && diag ? c - 1 : c;
        if (pre && kend <= 0) {
            df_sync(grp);   // everyone has read the ticket
            continue;
        }
        int *prow = &prog[q], *pcol = a.factor ? &prog[c] : prow;
        // the tile as it starts, through shared memory into the products' layout (eight or, on the diagonal, five
        // entries a thread), negated: acc = -A + sum of products
        double acc[8], cur[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int col = lc + 4 * u;
            double v;
            if (kind == 2)
                v = (e == c && lr == col) ? 1.0 : 0.0;
            else
                v = (lr < nr && col < cb) ? __ldcg(R + (long long)(c0 + col) * rld + r0 + lr) : 0.0;
            sm.Bs[col][lr] = v;
        }
        df_sync(grp);
        // The columns before the tile's own 64 enter as sums of 64 columns, each formed on its own and then taken off
        // the tile, so that the entries are rounded once per 64 columns and not once per column.  Relative errors
        // of the log-determinant (of l) against twice the digits on the same Sigma, rms of 3 to 24 draws, with one
        // sum over all columns, in 960-wide panels of 64-wide steps, and so:
        //   N = 800    4.2e-16 (4.0e-16)   1.6e-16 (3.1e-16)   1.4e-16 (2.8e-16)
        //   N = 1,600  9.2e-16 (9.2e-16)   1.9e-15 (2.1e-15)   2.5e-16 (1.1e-15)
        //   N = 3,200  1.7e-15 (3.6e-15)   3.2e-15 (9.6e-15)   1.6e-16 (3.3e-15)
        //   N = 8,002  2.9e-15 (3.3e-14)   3.8e-15 (2.4e-13)   2.0e-16 (1.4e-14)
        // Sums of 128 come to 1.2 to 3 times the last column.  One more FP64 operation per entry and 64 columns:
        // N = 8,002 142.7 -> 145.1 ms.
        const bool straight = kind == 2 || c < DF_SUM;
        bool based = straight;   // acc holds the tile too, not only a sum
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            cur[i] = diag ? (i < 5 ? -sm.Bs[dc[i % 5]][dr[i % 5]] : 0.0) : -sm.Bs[tx + 16 * (i % 2)][ty + 8 * (i / 2)];
            acc[i] = straight ? cur[i] : 0.0;
        }
        df_sync(grp);
        const int used = diag ? 5 : nr <= 8 ? 2 : 8;   // entries of acc in use
        const int kbeg = kind == 2 ? e : 0;
        int avail = kbeg;
        double pa[8], pb[8];
        auto load = [&](int k) {
            const long long kc = a.j0 + DT * k;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int kk = lc + 4 * u;
                if (kind == 2)   // row r of the identity block's solution is column r of -W; threads walk k
                    pa[u] = (DT * e + kk < a.jb) ? -__ldcg(a.W + (long long)(DT * e + kk) * a.ldw + DT * k + lr) : 0.0;
                else
                    pa[u] = lr < nr ? __ldcg(R + (kc + kk) * rld + r0 + lr) : 0.0;
                if (!diag) pb[u] = lr < cb ? __ldcg(a.A + (kc + kk) * a.ld + c0 + lr) : 0.0;
            }
        };
        bool gone = false;
        for (int k = kbeg; k < kend; ++k) {
            if (avail <= k) {
                if (tid == 0) sm.word[1] = df_wait(prow, pcol, k + 1, a.sync, &a.st->timeout, a.limit);
                df_sync(grp);
                avail = sm.word[1];
                if (avail < 0) {
                    gone = true;
                    break;
                }
                load(k);
            }
            // (the previous slice's products are done: barrier at the end of the loop body)
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (kind == 2)
                    sm.As[lr][lc + 4 * u] = pa[u];
                else
                    sm.As[lc + 4 * u][lr] = pa[u];
                if (!diag) sm.Bs[lc + 4 * u][lr] = pb[u];
            }
            df_sync(grp);
            if (k + 1 < kend && avail > k + 1) load(k + 1);   // in flight during the products
            if (diag)
                df_mma_diag(acc, sm.As, dr, dc);
            else if (nr <= 8)
                df_mma<1>(acc, sm.As, sm.Bs, tx, ty);
            else
                df_mma<4>(acc, sm.As, sm.Bs, tx, ty);
            if (!straight && k % DF_SUM == DF_SUM - 1) {   // a block done: off the tile, and on with the next one
                const bool own = based = k + 1 == c / DF_SUM * DF_SUM;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (i >= used) continue;
                    cur[i] += acc[i];
                    acc[i] = own ? cur[i] : 0.0;
                }
            }
            df_sync(grp);
        }
        if (gone) return;   // uniform over the group
        if (!based) {
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] += cur[i];
        }
        // the tile into shared memory, [col][row]; past the matrix a diagonal block continues as the identity
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (!diag)
                sm.Bs[tx + 16 * (i % 2)][ty + 8 * (i / 2)] = -acc[i];
            else if (i < 5)
                sm.Bs[dc[i % 5]][dr[i % 5]] =
                    (dr[i % 5] < cb && dc[i % 5] < cb) ? -acc[i] : (dr[i % 5] == dc[i % 5] ? 1.0 : 0.0);
        }
        if (pre) {
            df_sync(grp);
        } else if (diag) {
            df_sync(grp);
            // (the tile's part above the diagonal is never set: what the lanes of those rows compute is not used)
            auto *buf = reinterpret_cast<double (*)[4][DT]>(sm.Ls);
            const int bad = PLAIN ? df_potrf32_plain(sm.Bs, buf, sm.dinv, grp, tid)
                                  : df_potrf32(sm.Bs, buf, sm.dinv, grp, tid);
            if (bad < cb) {   // the same in every thread; nothing below this pivot can be finished
                if (tid == 0) {
                    set_info(a.st, c0 + bad + 1);
                    __threadfence();
                    atomicExch(&a.sync[1], 1);
                }
                return;
            }
            df_sync(grp);
        } else {
            // L_cc: wait for its factorisation
            if (tid == 0) sm.word[1] = a.factor ? df_wait(&prog[c], &prog[c], c + 1, a.sync, &a.st->timeout, a.limit) : 0;
            df_sync(grp);
            if (sm.word[1] < 0) return;
            const double *L = a.A + (long long)c0 * a.ld + c0;
            if (PLAIN) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int col = lc + 4 * u;
                    sm.Ls[col][lr] = (lr < cb && col < cb && lr >= col) ? __ldcg(L + (long long)col * a.ld + lr)
                                                                        : (lr == col ? 1.0 : 0.0);
                }
                if (tid < DT) sm.dinv[tid] = tid < cb ? 1.0 / __ldcg(L + (long long)tid * a.ld + tid) : 1.0;
                df_sync(grp);
                df_trsm32(sm.Bs, sm.Ls, sm.dinv, tid);
            } else {
                df_load_scaled(sm, L, a.ld, cb, grp, tid);
                df_trsm32_scaled(sm.Bs, sm.Ls, sm.dinv, tid);
            }
            df_sync(grp);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (kind == 2) {
                // W(column of the solution, row) = -X: threads walk the solution's columns, W's rows
                const int row = lc + 4 * u;   // row of the identity block
                if (lr < cb && row < nr) a.W[(long long)(DT * e + row) * a.ldw + DT * c + lr] = -sm.Bs[lr][row];
            } else {
                const int col = lc + 4 * u;
                if (lr < nr && col < cb && (!diag || lr >= col))
                    R[(long long)(c0 + col) * rld + r0 + lr] = sm.Bs[col][lr];
            }
        }
        df_sync(grp);
        if (tid == 0) {
            if (pre)
                df_st_release(prog + a.T + a.E + (a.W ? a.T : 0) + 2 * c + (diag ? 0 : 1), 1);
            else
                df_st_release(prow, c + 1);
        }
    }
}

// C[r, c] -= sum_k A[r, k] B[c, k] for RR rows r (right-hand sides): a thread per column reads its operand row
// along k, coalesced over columns, sixteen loads in flight.  Bound by the loads' latency and the FP64 FMAs of
// one warp, k of 64 clocks each per row; so the usual single row has its own form (k = 256 on average 31 us a
// launch, 105 with the FMAs of four rows), whose sums are the same.
template <int RR>
__global__ void __launch_bounds__(64) k_rhs_update(double *A, long long ld, int rC, int cC, int m, int n, int kA, int k,
                                                  const DevStatus *st) {
    if (st->info) return;
    const int r0 = blockIdx.y * RR;
    __shared__ double a[RR][256];
    const int c = blockIdx.x * 64 + threadIdx.x;
    double acc[RR] = {};
    for (int k0 = 0; k0 < k; k0 += 256) {
        const int kc = min(256, k - k0);
        __syncthreads();
        for (int t = threadIdx.x; t < RR * kc; t += 64)
            a[t % RR][t / RR] = (r0 + t % RR < m) ? A[(long long)(kA + k0 + t / RR) * ld + rC + r0 + t % RR] : 0.0;
        __syncthreads();
        if (c < n) {
            const double *b = A + (long long)(kA + k0) * ld + cC + c;
#pragma unroll 16
            for (int kk = 0; kk < kc; ++kk) {
                const double bv = b[(long long)kk * ld];
#pragma unroll
                for (int i = 0; i < RR; ++i) acc[i] = fma(a[i][kk], bv, acc[i]);
            }
        }
    }
    if (c < n)
#pragma unroll
        for (int i = 0; i < RR; ++i)
            if (r0 + i < m) A[(long long)(cC + c) * ld + rC + r0 + i] -= acc[i];
}

cudaError_t launch_df(const DfArgs &a0, int sms, int cls, double flops, cudaStream_t s) {
    DfArgs a = a0;
    const long long T = a.T, E = a.E;
    a.chain = a.factor && !a.block64 && T > 1;
    // below about 4,000 columns the chain, not the products, sets the time
    a.alone = a.chain && T < 128;
    const long long fixed = DF_HEAD + T + (a.W ? T : 0) + (a.chain ? 2 * T : 0), room = GEO_CHOL_SYNC_INTS - fixed;
    if (E > room) {   // rows past what the words hold, once the others are done
        if (room <= 0) return cudaErrorInvalidValue;
        DfArgs head = a0, rest = a0;
        head.E = (int)room;
        head.nx = DT * head.E;
        rest.factor = 0;
        rest.W = nullptr;
        rest.X += head.nx;
        rest.nx -= head.nx;
        rest.E -= head.E;
        const cudaError_t e = launch_df(head, sms, cls, flops, s);
        return e != cudaSuccess ? e : launch_df(rest, sms, cls, 0.0, s);
    }
    const long long words = fixed + E;
    const long long tickets = !a.factor ? (a.W ? T * (T + 1) / 2 : T * E)
                              : a.W     ? T * (T + E + 1)
                                        : T * (T + E) - T * (T - 1) / 2;
    if (tickets == 0) return cudaSuccess;
    if (words > GEO_CHOL_SYNC_INTS || tickets > (1LL << 30)) return cudaErrorInvalidValue;
    a.tickets = (int)tickets;
    cudaError_t e = cudaMemsetAsync(a.sync, 0, sizeof(int) * words, s);
    if (e != cudaSuccess) return e;
    constexpr size_t smem = sizeof(DfSmem) * DF_GROUPS;
    auto *kernel = a.plain ? k_chol_df<true> : k_chol_df<false>;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
    const int all = df_sms();
    const int grid = (int)std::min<long long>(sms > 0 ? std::min(sms, all) : all, tickets + a.chain);
    if (grid < 8) a.alone = 0;
    KScope ks(cls, s, flops, 16.0 * ((double)a.jb * a.jb / 2 + (double)a.nx * a.jb));
    kernel<<<grid, DF_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Factor the columns [j0, j0 + jb): the diagonal range, and the rows [x0, x1) below it (x0 >= j0 + jb;
// x0 == x1 = none) solved against it.  factor_diag false: the diagonal range already holds L and only the
// rows are solved (X <- X L^-T), or, without rows, only W is formed.  W (jb x jb, ldw) != NULL: also
// W = -L^-1, its strictly upper part must hold zeros.  sms: at most that many CTAs, one per SM (0 = all).
// sync: GEO_CHOL_SYNC_INTS device ints of scratch.
cudaError_t chol64_panel(double *A, long long ld, int j0, int jb, int x0, int x1, DevStatus *st, int *sync,
                         cudaStream_t s, bool factor_diag, double *W, long long ldw, int sms, int order) {
    if (jb <= 0) return cudaSuccess;
    if (!factor_diag && W && x1 > x0) return cudaErrorInvalidValue;
    const int nx = std::max(0, x1 - x0);
    DfArgs a{A, ld, j0, jb, A + x0, ld, nx, (jb + DT - 1) / DT, (nx + DT - 1) / DT, factor_diag ? 1 : 0, W, ldw, sync,
             0, 0, 0, order == GEO_CHOL_BLOCK64, order != GEO_CHOL_NATIVE, st, DF_WAIT_CYCLES};
    const double j = jb, cubes = (factor_diag ? j * j * j / 3.0 : 0.0) + (W ? j * j * j / 3.0 : 0.0);
    return launch_df(a, sms, factor_diag ? GEO_K_POTRF : GEO_K_TRSM, cubes + nx * j * j, s);
}

// SMs for a diagonal tile of order jb (with its inverse) that runs beside other work of rest_us: the fewest
// with which the tile is done in that time.  A tile takes its column chain, about 0.55 us a column, or its FP64
// FMAs (jb^3 / 6, twice with the inverse) at two per clock and SM, whichever is longer.
int chol64_side_sms(int jb, bool inverse, double rest_us) {
    const double j = jb, chain = 0.55 * j, fma_us = j * j * j / 6.0 * (inverse ? 2.0 : 1.0) / (2.0 * 2000.0);
    int n = 8;
    while (n < 48 && fma_us / n > std::max(chain, rest_us)) n += 8;
    return n;
}

// C[rC.., cC..] (m x n) -= A[rC.., kA..kA+k] A[cC.., kA..kA+k]' in FP64, for the right-hand-side rows of a
// factorisation whose other updates run elsewhere.
cudaError_t chol64_rhs_update(double *A, long long ld, int rC, int cC, int m, int n, int kA, int k, DevStatus *st,
                              cudaStream_t s) {
    if (m <= 0 || n <= 0 || k <= 0) return cudaSuccess;
    KScope ks(GEO_K_GEMM, s, 2.0 * k * (double)m * n, 8.0 * ((double)n * k + 2.0 * m * n));
    if (m == 1)
        k_rhs_update<1><<<(n + 63) / 64, 64, 0, s>>>(A, ld, rC, cC, m, n, kA, k, st);
    else
        k_rhs_update<4><<<dim3((n + 63) / 64, (m + 3) / 4), 64, 0, s>>>(A, ld, rC, cC, m, n, kA, k, st);
    return cudaGetLastError();
}

// In-place lower Cholesky of the leading N x N block of A with the rows N .. nrows-1 carried along: one launch.
cudaError_t chol64_factor(double *A, long long ld, int N, int nrows, DevStatus *st, int *sync, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    const int nx = std::max(0, nrows - N);
    DfArgs a{A, ld, 0, N, A + N, ld, nx, (N + DT - 1) / DT, (nx + DT - 1) / DT, 1, nullptr, 0, sync,
             0, 0, 0, 0, 0, st, DF_WAIT_CYCLES};
    const double n = N;
    return launch_df(a, 0, GEO_K_GEMM, n * n * n / 3.0 + nx * n * n, s);
}

// X <- X L^-T for the rows of X (R x N, column-major, ldx), L the lower N x N factor: one launch.
cudaError_t chol64_solve_rows(double *X, long long ldx, int R, double *L, long long ldl, int N, DevStatus *st, int *sync,
                              cudaStream_t s) {
    if (R <= 0 || N <= 0) return cudaSuccess;
    DfArgs a{L, ldl, 0, N, X, ldx, R, (N + DT - 1) / DT, (R + DT - 1) / DT, 0, nullptr, 0, sync,
             0, 0, 0, 0, 0, st, DF_WAIT_CYCLES};
    return launch_df(a, 0, GEO_K_SOLVE, (double)R * N * N, s);
}
