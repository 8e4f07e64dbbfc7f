// Triangular solves with a column-major lower-triangular L (the factor of
// Sigma): forward L x = b and backward L' x = y, the solves of Eq. 1 and of
// the cokriging weights Sigma^-1 Z in Eq. 3.
//
// The solve is a chain over the 64-row blocks, so all that does not need the
// blocks before is done ahead of a block's turn: its CTA inverts the two 32 x 32
// triangles of the diagonal block while it waits, and the entries of L are
// loaded before the wait.  The chain then carries seven 32 x 32 products, each
// a step over all warps, instead of 64 dependent steps of one warp: two for a
// triangle's inverse and its residual, one more to add the correction (the
// inverse alone has 1.5 to 3.7 times the substitution's error on a smooth
// field's factor, with the correction it is the same), one between the halves.
// The first block has nothing to wait for, and one warp's substitution (20 us)
// is done sooner than the inversion: it is solved that way (N = 64: 21 us, 33
// by inversion).  Backward, with that substitution in every block and now:
// N = 128 41 and 34 us, 512 149 and 87, 2,000 588 and 272, 8,000 2.56 and
// 1.04 ms, 40,500 14.3 and 6.6 ms.  Bound by the chain, about 8 us a block.
//
// One launch per solve.  The rows are cut into blocks of 64; CTAs take the
// blocks in solve order from a ticket counter (forward: top to bottom;
// backward: bottom to top).  The CTA holding block I accumulates the products
// with the blocks already solved, waiting on a `done` counter for the ones
// that are not (a block completes only after its predecessor, so one counter
// suffices), then solves its diagonal block and publishes it.
// A CTA only waits on blocks whose tickets were taken earlier by CTAs that
// are running, so the solve cannot deadlock whatever the number of resident
// CTAs.  Every wait is bounded: past WAIT_CYCLES the CTA raises an abort word
// that makes every other waiter give up too, records the timeout and leaves
// the solve unfinished.  Sums run in a fixed order: the result does not
// depend on timing.  Each pass streams the lower triangle once.
//
// sync: 4 device ints {ticket, done, abort, unused}, zeroed before each launch.
#include "geo_internal.cuh"

namespace {

constexpr int TB = 64;       // rows per block
constexpr int TT = 256;      // threads per CTA
constexpr long long WAIT_CYCLES = 2000000000LL;   // ~1 s at 2 GHz

__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(int *p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}

// Wait until done >= target.  Returns done, or -1 when the solve was aborted
// (here or elsewhere).  limit: the wait's clock budget (0 = WAIT_CYCLES).
__device__ int wait_done(int *sync, int target, int *timeout_word, int code, long long limit) {
    const long long t0 = clock64();
    const long long budget = limit > 0 ? limit : WAIT_CYCLES;
    for (;;) {
        const int d = ld_acquire(&sync[1]);
        if (d >= target) return d;
        if (ld_acquire(&sync[2])) return -1;
        if (clock64() - t0 > budget) {
            atomicExch(&sync[2], 1);
            if (timeout_word) atomicCAS(timeout_word, 0, code);
            return -1;
        }
        __nanosleep(100);
    }
}

constexpr int TH = TB / 2;   // triangles that are inverted

// The diagonal block in shared memory, zeros past ib, columns first: its triangles, their inverses, the square
// below them.
struct Diag {
    double t[2][TH][TH + 1], x[2][TH][TH + 1], m[TH][TH + 1];
    double part[8][TH], rhs[TB], y[TH], e[TH];
};

// Loads the block and the reciprocals of its pivots (the diagonals of x) and, on request, inverts its triangles,
// column by column from the last: below the diagonal, minus the inverse found so far times the column of L, over the
// pivot.  Four warps per triangle share a row's sum.
__device__ __forceinline__ void load_diag(const double *__restrict__ A, long long ld, int i0, int ib, Diag &d,
                                          bool invert) {
    for (int i = threadIdx.x; i < TB * TB; i += TT) {
        const int c = i / TB, r = i % TB, h = c / TH;
        if (r < h * TH) continue;   // above the triangles
        const double v = (r < ib && c < ib && r >= c) ? A[(long long)(i0 + c) * ld + i0 + r] : 0.0;
        if (r / TH == h) {
            d.t[h][c - h * TH][r - h * TH] = v;
            d.x[h][c - h * TH][r - h * TH] = (r == c && r < ib) ? 1.0 / v : 0.0;
        } else
            d.m[c][r - TH] = v;
    }
    __syncthreads();
    if (!invert) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32, q = w % 4;
    double(*T)[TH + 1] = d.t[w / 4], (*X)[TH + 1] = d.x[w / 4];
    for (int j = TH - 2; j >= 0; --j) {
        double s = 0.0;
        for (int k = j + 1 + q; k < TH; k += 4) s = fma(X[k][lane], T[j][k], s);
        d.part[w][lane] = s;
        __syncthreads();
        if (q == 0 && lane > j)
            X[j][lane] = -X[j][j] * ((s + d.part[w + 1][lane]) + (d.part[w + 2][lane] + d.part[w + 3][lane]));
        __syncthreads();
    }
}

// B v for a 32 x 32 block B, columns first (B' v with TR): four of a row's 32 terms per warp.  The sum, in warp 0.
template <bool TR>
__device__ __forceinline__ double mul32(double (*B)[TH + 1], const double *v, Diag &d) {
    const int lane = threadIdx.x & 31, w = threadIdx.x / 32;
    double t[2] = {0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int k = 4 * w + i;
        t[i & 1] = fma(TR ? B[lane][k] : B[k][lane], v[k], t[i & 1]);
    }
    d.part[w][lane] = t[0] + t[1];
    __syncthreads();
    if (w) return 0.0;
    return ((d.part[0][lane] + d.part[1][lane]) + (d.part[2][lane] + d.part[3][lane])) +
           ((d.part[4][lane] + d.part[5][lane]) + (d.part[6][lane] + d.part[7][lane]));
}

// d.y = T^-1 rhs (T'^-1 with TR) for triangle h: by the inverse, then a correction by the residual's.
template <bool TR>
__device__ __forceinline__ void tri32(int h, Diag &d) {
    const int i = threadIdx.x;   // of the first warp's sums
    double v = mul32<TR>(d.x[h], d.rhs + h * TH, d);
    if (i < TH) d.y[i] = v;
    __syncthreads();
    v = mul32<TR>(d.t[h], d.y, d);
    if (i < TH) d.e[i] = d.rhs[h * TH + i] - v;
    __syncthreads();
    v = mul32<TR>(d.x[h], d.e, d);
    if (i < TH) d.y[i] += v;
    __syncthreads();
}

// rhs <- L_II^-1 rhs (L_II'^-1 with TR) by substitution, one warp, rows lane and 32 + lane.
template <bool TR>
__device__ __forceinline__ void substitute(Diag &d, int ib) {
    const int lane = threadIdx.x & 31;
    double v[2] = {d.rhs[lane], d.rhs[TH + lane]};
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int h = TR ? 1 - hh : hh;
        const int n = min(TH, ib - h * TH);
        for (int kk = 0; kk < n; ++kk) {
            const int k = TR ? n - 1 - kk : kk;
            const double vk = __shfl_sync(0xffffffffu, v[h], k) * d.x[h][k][k];
            if (lane == k) v[h] = vk;
            if (TR ? lane < k : lane > k) v[h] = fma(-(TR ? d.t[h][lane][k] : d.t[h][k][lane]), vk, v[h]);
            if (hh == 0) v[1 - h] = fma(-(TR ? d.m[lane][k] : d.m[k][lane]), vk, v[1 - h]);
        }
    }
    d.rhs[lane] = v[0];
    d.rhs[TH + lane] = v[1];
}

__global__ void __launch_bounds__(TT) k_trsv_fwd(const double *__restrict__ A, long long ld, int N, double *x,
                                                 int *sync, int *timeout_word, long long wait_limit) {
    __shared__ Diag d;
    __shared__ int tick, abort_s;
    const int nblk = (N + TB - 1) / TB;
    const int r = threadIdx.x % TB, g = threadIdx.x / TB;   // row of the block, group of 16 columns
    const int lane = threadIdx.x & 31;
    for (;;) {
        if (threadIdx.x == 0) {
            tick = atomicAdd(&sync[0], 1);
            abort_s = 0;
        }
        __syncthreads();
        const int I = tick;
        if (I >= nblk) return;
        const int i0 = I * TB, ib = min(TB, N - i0);
        load_diag(A, ld, i0, ib, d, I > 0);
        // acc = sum_{J < I} L[i0 + r, J block] x[J block], columns g*16 .. g*16+15 of each block
        double acc = (g == 0 && r < ib) ? -x[i0 + r] : 0.0;
        int seen = 0;
        bool aborted = false;
        for (int J = 0; J < I; ++J) {
            double a[16];
            const double *col = A + (long long)(J * TB + g * 16) * ld + i0 + r;
#pragma unroll
            for (int c = 0; c < 16; ++c) a[c] = r < ib ? col[(long long)c * ld] : 0.0;
            if (J >= seen) {   // warp-uniform
                // every lane waits with its own acquire loads before it reads x
                const int done = __reduce_min_sync(0xffffffffu, wait_done(sync, J + 1, timeout_word, 3, wait_limit));
                if (done < 0) {
                    aborted = true;
                    break;
                }
                seen = done;
            }
            const double *xj = x + J * TB + g * 16;
            double s0 = 0.0;   // two chains
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
                acc = fma(a[c], __ldcg(xj + c), acc);
                s0 = fma(a[c + 1], __ldcg(xj + c + 1), s0);
            }
            acc += s0;
        }
        if (aborted && lane == 0) atomicExch(&abort_s, 1);
        d.part[threadIdx.x / 32][lane] = acc;   // warps 2 g and 2 g + 1: the rows' halves
        __syncthreads();
        if (abort_s) return;   // uniform: every thread reads it after the barrier
        if (g == 0) {
            const int h = r / TH;
            d.rhs[r] = -((d.part[h][lane] + d.part[2 + h][lane]) + (d.part[4 + h][lane] + d.part[6 + h][lane]));
        }
        __syncthreads();
        const bool w0 = threadIdx.x < 32;
        if (I == 0) {
            if (w0) {
                substitute<false>(d, ib);
                if (lane < ib) x[lane] = d.rhs[lane];
                if (TH + lane < ib) x[TH + lane] = d.rhs[TH + lane];
            }
        } else {
            tri32<false>(0, d);
            if (w0 && lane < ib) x[i0 + lane] = d.y[lane];
            const double v = mul32<false>(d.m, d.y, d);
            if (w0) d.rhs[TH + lane] -= v;
            __syncthreads();
            tri32<false>(1, d);
            if (w0 && TH + lane < ib) x[i0 + TH + lane] = d.y[lane];
        }
        __syncthreads();
        if (threadIdx.x == 0) st_release(&sync[1], I + 1);   // releases what the CTA wrote before the barrier
    }
}

__global__ void __launch_bounds__(TT) k_trsv_bwd(const double *__restrict__ A, long long ld, int N, double *w,
                                                 int *sync, int *timeout_word) {
    __shared__ Diag d;
    __shared__ int tick, abort_s;
    const int nblk = (N + TB - 1) / TB;
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;   // warp: columns 8 warp .. 8 warp + 7
    for (;;) {
        if (threadIdx.x == 0) {
            tick = atomicAdd(&sync[0], 1);
            abort_s = 0;
        }
        __syncthreads();
        const int t = tick;
        if (t >= nblk) return;
        const int I = nblk - 1 - t;
        const int i0 = I * TB, ib = min(TB, N - i0);
        load_diag(A, ld, i0, ib, d, t > 0);
        // acc[q] = sum_{J > I} sum_{rows k of J} L[k, i0 + 8 warp + q] w[k], lanes over rows
        double acc[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = 0.0;
        int seen = 0;
        bool aborted = false;
        for (int J = nblk - 1; J > I; --J) {
            const int j0 = J * TB, jb = min(TB, N - j0);
            double a0[8], a1[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int c = 8 * warp + q;
                const double *col = A + (long long)(i0 + c) * ld + j0;
                a0[q] = (c < ib && lane < jb) ? col[lane] : 0.0;
                a1[q] = (c < ib && lane + 32 < jb) ? col[lane + 32] : 0.0;
            }
            const int need = nblk - J;   // tickets 0 .. need-1 done
            if (need > seen) {   // warp-uniform
                // every lane waits with its own acquire loads before it reads w
                const int done = __reduce_min_sync(0xffffffffu, wait_done(sync, need, timeout_word, 4, 0));
                if (done < 0) {
                    aborted = true;
                    break;
                }
                seen = done;
            }
            const double w0 = (lane < jb) ? __ldcg(w + j0 + lane) : 0.0;
            const double w1 = (lane + 32 < jb) ? __ldcg(w + j0 + lane + 32) : 0.0;
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] = fma(a1[q], w1, fma(a0[q], w0, acc[q]));
        }
        if (aborted && lane == 0) atomicExch(&abort_s, 1);
        // the eight sums over the warp: each halving of the lanes halves the number of sums a lane carries
#pragma unroll
        for (int h = 4, o = 16; h >= 1; h >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int q = 0; q < h; ++q)
                acc[q] = (up ? acc[q + h] : acc[q]) + __shfl_xor_sync(0xffffffffu, up ? acc[q] : acc[q + h], o);
        }
        double v = acc[0];   // of column 4 [lane & 16] + 2 [lane & 8] + [lane & 4]
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        if ((lane & 3) == 0) {
            const int c = 8 * warp + (lane >> 2 & 1) + (lane >> 3 & 1) * 2 + (lane >> 4 & 1) * 4;
            d.rhs[c] = c < ib ? w[i0 + c] - v : 0.0;
        }
        __syncthreads();
        if (abort_s) return;
        if (t == 0) {
            if (warp == 0) {
                substitute<true>(d, ib);
                if (lane < ib) w[i0 + lane] = d.rhs[lane];
                if (TH + lane < ib) w[i0 + TH + lane] = d.rhs[TH + lane];
            }
        } else {
            tri32<true>(1, d);
            if (warp == 0 && TH + lane < ib) w[i0 + TH + lane] = d.y[lane];
            v = mul32<true>(d.m, d.y, d);
            if (warp == 0) d.rhs[lane] -= v;
            __syncthreads();
            tri32<true>(0, d);
            if (warp == 0 && lane < ib) w[i0 + lane] = d.y[lane];
        }
        __syncthreads();
        if (threadIdx.x == 0) st_release(&sync[1], t + 1);   // releases what the CTA wrote before the barrier
    }
}

__global__ void k_copy_strided(const double *__restrict__ in, long long stride, int N, double *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < N) out[k] = in[(long long)k * stride];
}

// sync[0] = v (the ticket counter) before a launch
__global__ void k_set_ticket(int *sync, int v) { sync[0] = v; }

int solve_grid(int N) {
    const int nblk = (N + TB - 1) / TB;
    return nblk < 152 * 4 ? nblk : 152 * 4;
}

}  // namespace

cudaError_t forward_solve(const double *A, long long ld, int N, double *x, int *sync, int *timeout_word,
                          cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(sync, 0, 4 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    KScope ks(GEO_K_SOLVE, s, (double)N * N, 8.0 * (double)N * N / 2.0);
    k_trsv_fwd<<<solve_grid(N), TT, 0, s>>>(A, ld, N, x, sync, timeout_word, 0);
    return cudaGetLastError();
}

// The forward solve with its first block withheld: the ticket counter starts
// at 1, so no CTA ever solves block 0 and publishes it, and the CTA of block 1
// waits for a completion that never comes.  With a wait budget of
// wait_limit cycles that wait gives up, raises the abort word (every other
// waiter returns too), records code 3 in *timeout_word and the launch ends.
cudaError_t forward_solve_withheld(const double *A, long long ld, int N, double *x, int *sync, int *timeout_word,
                                   long long wait_limit, cudaStream_t s) {
    if (N <= TB || wait_limit <= 0) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(sync, 0, 4 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_set_ticket<<<1, 1, 0, s>>>(sync, 1);
    k_trsv_fwd<<<solve_grid(N), TT, 0, s>>>(A, ld, N, x, sync, timeout_word, wait_limit);
    return cudaGetLastError();
}

// w = L^-T y (y strided; w may be y's storage when ystride == 1).
cudaError_t backward_solve(const double *A, long long ld, int N, const double *y, long long ystride, double *w,
                           int *sync, int *timeout_word, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    if (y != w || ystride != 1) {
        KScope ks(GEO_K_AUX, s);
        k_copy_strided<<<(N + 255) / 256, 256, 0, s>>>(y, ystride, N, w);
    }
    cudaError_t e = cudaMemsetAsync(sync, 0, 4 * sizeof(int), s);
    if (e != cudaSuccess) return e;
    KScope ks(GEO_K_SOLVE, s, (double)N * N, 8.0 * (double)N * N / 2.0);
    k_trsv_bwd<<<solve_grid(N), TT, 0, s>>>(A, ld, N, w, sync, timeout_word);
    return cudaGetLastError();
}
