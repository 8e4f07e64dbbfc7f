// FP64-accurate matrix products on the BF16 tensor cores (the Ozaki scheme:
// error-free splitting into short integer digits), and the dense Cholesky
// factorisation of Sec. 5.2 with its trailing updates (the SYRK / GEMM tile
// tasks of Sec. 5.1) computed that way.
//
// GB300 runs FP64 at about 1.26 TFLOP/s but BF16 MMAs at ~1,900 TFLOP/s.
// Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012) split each
// operand into slices whose pairwise products a lower-precision unit computes
// without rounding error; summing the products in high precision recovers the
// FP64 product.  Here:
//
//   row scale   every operand row r gets e_r with max_k |x_rk| < 2^e_r;
//   digits      X = rint(x 2^(7S - 1 - e_r)) is an integer of at most 7S bits;
//               its balanced base-128 digits d_1 .. d_S (d_1 the most
//               significant, |d_1| <= 64, -64 <= d_t < 64 after it) give
//               x ~= 2^e_r sum_t d_t 2^(1 - 7t), with |error| <= 2^(e_r - 7S);
//   products    level l = t + u collects d_t(a) d_u(b), scale 2^(2 - 7l); the
//               levels l <= S + 1 are kept (S(S+1)/2 products), the rest
//               would change the result by about 2^-7S relative;
//   exactness   each digit is an integer in [-64, 64], exact in BF16, each
//               product is an integer of magnitude <= 2^12, and a level holds
//               at most S products: over a depth K with S K 2^12 <= 2^24 every
//               partial sum in the FP32 tensor-memory accumulator is an
//               integer below 2^24, so the tensor cores add without rounding
//               (the depth of one launch is capped at kmax = 4096 / S);
//   recombine   the epilogue converts each level to an integer and folds
//               groups of four levels (2..5, 6..9) into 64-bit integers
//               (exact: below 2^46), then applies
//               C -= 2^(e_r + e_c) sum_w W_w 2^(2 - 7 hi_w), hi_w the last
//               level of group w, with one FP64 FMA per group.
//
//   level cut  (optional, trailing updates of the factorisation) the levels
//               kept for an output tile follow its operands' magnitudes: with
//               E the largest row exponent of the launch's A rows plus that of
//               its B rows, and e_i + e_j the same over the tile's own rows,
//               the tile keeps the levels l <= S + 1 - q, q = floor((E - e_i - e_j) / 7).
//               A level-l term is at most 2^(e_i + e_j + 14 - 7 l), so the
//               first level such a tile drops, S + 2 - q, is at most
//               2^(e_i + e_j + 7 q - 7 S) <= 2^(E - 7 S): no larger than the
//               first level the launch's largest tile drops without the cut.
//               Every entry's error thus stays within the bound of the
//               launch's largest products; tiles whose operands are tiny
//               against the largest (far from the diagonal in a spatially
//               ordered covariance) skip levels or vanish entirely.
//
// The digits lie interleaved: per operand row and 16 columns (the K of one MMA)
// the 16 digits of every slice in turn, 32 bytes a slice.  A TMA box of 128
// lines of 128 bytes brings four slices at once (the last one of a chunk may
// reach into the next chunk's, which no MMA reads, so that S need not be a
// multiple of 4), and a slice is a 32-byte step of the
// operand descriptor within the 128-byte swizzle, the step that usually
// advances K.  With the slices apart a chunk of 8 slices took 24 boxes of
// 32-byte lines a tile, with almost no MMAs 0.73 ms for the product below; now
// 6 boxes, 0.61 ms.
//
// The kernel is persistent (one CTA per SM) over 128 x 128 output tiles, the
// K range in chunks of 16.  TMEM (512 columns) holds four level accumulators
// of 128 x 128 FP32, so the levels run as passes of four over K, each loading
// only the slices its levels use and writing its part of C.  (64-column tiles
// would hold eight levels, but the 128-row A operand read per MMA then keeps
// shared memory twice as busy as the math: 4 slices 0.56 ms against 0.34 for
// C 8192 x 4096, K = 512, 5 slices 0.76 against 0.57.)
//   warp 0, one lane: TMA producer, ring of slots, each with four digit slices
//     of a K chunk of the A rows (128 lines of 128 bytes) and of the B rows
//     (128 lines); a pass that reads at most four takes one slot per chunk;
//   warp 1: allocates the 512 TMEM columns; one lane issues tcgen05.mma
//     kind::f16 (M 128, N 128, K 16) level by level from precomputed shared
//     memory descriptors and commits chunks back to the producer;
//   warps 2-9: epilogue; tcgen05.ld of each level, releasing that
//     accumulator slot as soon as it is read (the MMAs of the next pass or
//     tile may start into it while the epilogue folds the values in
//     registers), then the FP64 read-modify-write of C, which comes through
//     shared memory by cp.async twelve columns ahead, the first of them
//     before the tile's MMAs are done.
// What bounds it: without the cut the MMAs (77 of 64 ideal cycles each: two
// 4 KB operands per MMA take all of shared memory's bandwidth), 8 slices 67 us
// a tile of K = 512; with few levels left the epilogue's FP64 work and loads of
// C, 7 us a pass (28 before the loads ran ahead).  The single-thread roles count
// along where they stand in the ring: a 64-bit division per chunk there took as
// long as ten MMAs.  C 8192 x 4096, K = 512: 8 slices 1.02 -> 0.93 ms, 6 slices
// 0.91 -> 0.64, 4 slices 0.56 -> 0.34; the updates of N = 40,000 with the level cut
// 343 -> 305 ms.
// With the level cut each CTA first computes the cut of all its tiles into a
// shared-memory table, and the MMA thread counts the products it issues
// (the device-side tensor work of the profile).
// Every mbarrier wait is bounded; on expiry the thread records a code in the
// status word, the CTA drains what it has in flight, frees TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "geo_internal.cuh"
#include "tcgen05_ptx.cuh"

namespace {

using namespace tc;

constexpr int OZ_BM = 128;        // output rows per tile (MMA M, TMEM lanes)
constexpr int OZ_BN = 128;        // output columns per tile (MMA N)
constexpr int OZ_KALIGN = 32;     // slice arrays: K padded to a multiple of 32 (64-byte rows)
constexpr int OZ_EPI_WARPS = 8;
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;
constexpr int OZ_TMEM_COLS = 512;
constexpr int OZ_A_BYTES = OZ_BM * 128, OZ_SLOT_BYTES = (OZ_BM + OZ_BN) * 128;   // one group of one K chunk
constexpr int OZ_SLOTS = 6;               // ring of K chunks
constexpr int OZ_CPT = OZ_BN / 2;         // columns per epilogue thread
constexpr int OZ_CD = 12, OZ_CQ = 4;      // C columns in flight per epilogue thread, columns per copy group
constexpr size_t OZ_SMEM = (size_t)OZ_SLOTS * OZ_SLOT_BYTES + sizeof(double) * OZ_EPI_WARPS * OZ_CD * 32 + 1024;
constexpr int OZ_LC_CAP = 8192;           // tiles per CTA whose level cut is computed up front
constexpr int OZ_GROUP = 8;       // row blocks swept together (operand reuse in L2)
constexpr int OZ_LPW = 4;         // levels folded into one 64-bit word
constexpr int OZ_E_NONE = -4096;  // block exponent of rows that are all zero (or absent)

// TMEM holds 512 / OZ_BN = 4 level accumulators, one word of levels, so the S levels are processed in passes of a
// word over the whole K range; each pass loads only the groups of four slices its levels use.
template <int S>
struct OzCfg {
    static constexpr int PASSES = (S + OZ_LPW - 1) / OZ_LPW;   // words of <= 4 levels (levels 2 .. S+1)
    static constexpr int NG = (S + 3) / 4;                     // groups of four slices
    // levels of pass g: [lev_lo, lev_hi]; slices it reads: 1 .. tmax
    __host__ __device__ static constexpr int lev_lo(int g) { return 2 + OZ_LPW * g; }
    // (also the word's unit, 2^(2 - 7 lev_hi))
    __host__ __device__ static constexpr int lev_hi(int g) { return (5 + OZ_LPW * g) < (S + 1) ? (5 + OZ_LPW * g) : (S + 1); }
    __host__ __device__ static constexpr int tmax(int g) { return lev_hi(g) - 1; }
};

struct OzArgs {
    double *C;
    long long ldc;
    int r0, c0;          // global row / col of the region's first output
    int m_end, n_end;    // outputs with global row >= m_end or col >= n_end are not written
    int mt, nt;          // 128 x 128 tiles of the region
    int tri;             // write only global row >= global col; skip tiles entirely above the diagonal
    int overwrite;       // 1: C = -A B' (C is not read)
    int a_off, b_off;    // slice row of the region's first row (A) / first column (B)
    int nk;              // K chunks of 16
    int split;           // CTAs per tile, each of which forms it and updates 1 / split of its columns (1, 2 or 4)
    const int *ea, *eb;  // per-row exponents of the A / B slices
    // level cut: per 32-row block maxima of the row exponents over every row (ba, bb) and over the
    // reference rows (ra, rb) of the A / B slices, nba / nbb blocks; cut = 0 keeps every level
    const int *ba, *bb, *ra, *rb;
    int nba, nbb, cut;
    unsigned long long *tc_flops;   // tensor-core flops issued, summed over CTAs (may be NULL)
    DevStatus *st;
};

__device__ __forceinline__ int ntiles_all(const OzArgs &a) { return a.mt * a.nt; }

__device__ __forceinline__ void cp_async8(double *dst, const double *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Highest level an output tile keeps (< 2: the tile is skipped); eref = E_A + E_B.
template <int S>
__device__ __forceinline__ int oz_lcut(const OzArgs &a, int ar, int br, int eref) {
    if (!a.cut) return S + 1;
    int ei = OZ_E_NONE, ej = OZ_E_NONE;
    const int a1 = min((ar + OZ_BM - 1) >> 5, a.nba - 1), b1 = min((br + OZ_BN - 1) >> 5, a.nbb - 1);
    for (int b = ar >> 5; b <= a1; ++b) ei = max(ei, a.ba[b]);
    for (int b = br >> 5; b <= b1; ++b) ej = max(ej, a.bb[b]);
    if (ei == OZ_E_NONE || ej == OZ_E_NONE) return 1;   // every row of one side is zero: nothing to add
    return S + 1 - max(0, eref - ei - ej) / 7;
}

__device__ __forceinline__ bool oz_tile(const OzArgs &a, int L, int *gr, int *gc, int *ar, int *br) {
    const unsigned per_band = (unsigned)OZ_GROUP * a.nt;
    const unsigned band = (unsigned)L / per_band;
    const int i0 = (int)band * OZ_GROUP;
    const unsigned gm = min(OZ_GROUP, a.mt - i0);
    const unsigned w = (unsigned)L - band * per_band;
    const int j = (int)(w / gm), i = i0 + (int)(w % gm);
    *gr = a.r0 + i * OZ_BM;
    *gc = a.c0 + j * OZ_BN;
    *ar = a.a_off + i * OZ_BM;
    *br = a.b_off + j * OZ_BN;
    return !(a.tri && *gr + OZ_BM - 1 < *gc);
}

// A CTA's first tile and the step to its next one; SPLIT: args.split CTAs to a tile.
template <bool SPLIT>
__device__ __forceinline__ unsigned oz_first(const OzArgs &a) { return SPLIT ? blockIdx.x / (unsigned)a.split : blockIdx.x; }
template <bool SPLIT>
__device__ __forceinline__ unsigned oz_step(const OzArgs &a) { return SPLIT ? gridDim.x / (unsigned)a.split : gridDim.x; }

// 2^e as a double (0 below the normal range, where the scaled terms are
// below 2^-1000 and vanish against any entry of C that matters).
__device__ __forceinline__ double pow2i(int e) {
    if (e < -1022) return 0.0;
    if (e > 1023) e = 1024;   // infinity: only reachable from non-finite operands
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// LOW_FIRST: the passes from the last levels up instead of down to them (without the level cut).  SPLIT: args.split
// CTAs to a tile (a form of its own: the columns' bounds cost registers that large products need).
template <int S, bool LOW_FIRST, bool SPLIT>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_update(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const OzArgs args) {
    using Cfg = OzCfg<S>;
    constexpr int ST = OZ_SLOTS, NG = Cfg::NG, PASSES = Cfg::PASSES, CPT = OZ_CPT;
    extern __shared__ uint8_t smem_raw[];
    constexpr int NSLOT = OZ_TMEM_COLS / OZ_BN;   // accumulator slots
    __shared__ uint64_t full_bar[ST], empty_bar[ST], acc_full, slot_empty[NSLOT], drain_bar;
    __shared__ uint32_t tmem_slot;
    __shared__ int skip, emax_a, emax_b;

    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    // one read for the whole CTA: a factorisation step on another stream may set it meanwhile
    if (threadIdx.x == 0) {
        skip = *(volatile const int *)&args.st->info;
        emax_a = emax_b = OZ_E_NONE;
    }
    __syncthreads();
    if (skip) return;   // an earlier step failed
    if (args.cut) {   // the launch's reference exponents E_A, E_B
        int ma = OZ_E_NONE, mb = OZ_E_NONE;
        for (int b = threadIdx.x; b < args.nba; b += OZ_THREADS) ma = max(ma, args.ra[b]);
        for (int b = threadIdx.x; b < args.nbb; b += OZ_THREADS) mb = max(mb, args.rb[b]);
        for (int o = 16; o > 0; o >>= 1) {
            ma = max(ma, __shfl_xor_sync(0xffffffffu, ma, o));
            mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        }
        if (lane == 0) {
            atomicMax(&emax_a, ma);
            atomicMax(&emax_b, mb);
        }
        __syncthreads();
    }
    const int eref = emax_a + emax_b;
    // the level cut of this CTA's tiles (the i-th tile it visits is L = blockIdx.x + i gridDim.x),
    // computed once here so that no role waits on the exponent loads inside its tile loop
    __shared__ uint8_t lc_tab[OZ_LC_CAP];
    if (args.cut) {
        const int mine = (int)((ntiles_all(args) - oz_first<SPLIT>(args) + oz_step<SPLIT>(args) - 1) / oz_step<SPLIT>(args));
        for (int i = threadIdx.x; i < OZ_LC_CAP && i < mine; i += OZ_THREADS) {
            int gr, gc, ar, br;
            const int L = (int)(oz_first<SPLIT>(args) + (unsigned)i * oz_step<SPLIT>(args));
            lc_tab[i] = oz_tile(args, L, &gr, &gc, &ar, &br) ? (uint8_t)max(0, oz_lcut<S>(args, ar, br, eref))
                                                                 : (uint8_t)0;
        }
        __syncthreads();
    }
    double *c_stage = reinterpret_cast<double *>((((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023) + ST * OZ_SLOT_BYTES);
    auto tile_lc = [&](int i, int ar, int br) -> int {
        if (!args.cut) return S + 1;
        return i < OZ_LC_CAP ? (int)lc_tab[i] : oz_lcut<S>(args, ar, br, eref);
    };
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int ntiles = ntiles_all(args);

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&acc_full, 1);
        for (int j = 0; j < NSLOT; ++j) mbar_init(&slot_empty[j], OZ_EPI_WARPS);
        mbar_init(&drain_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(OZ_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_slot;
    int *tword = &args.st->timeout;

    if (warp == 0) {
        if (lane == 0) {
            // the ring's position and phase are counted along: a division per chunk in this one thread costs more
            // than the chunk's MMAs
            int s = 0, filled = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int L = oz_first<SPLIT>(args), it = 0; L < ntiles && ok; L += oz_step<SPLIT>(args), ++it) {
                int gr, gc, ar, br;
                if (!oz_tile(args, L, &gr, &gc, &ar, &br)) continue;
                const int lc = tile_lc(it, ar, br);
#pragma unroll
                for (int pi = 0; pi < PASSES; ++pi) {
                    const int ps = LOW_FIRST ? PASSES - 1 - pi : pi;
                    if (Cfg::lev_lo(ps) > lc) break;   // every level of this pass (and later ones) is cut
                    const int ng = (min(Cfg::tmax(ps), lc - 1) + 3) / 4;   // groups of slices the pass reads
                    for (int kb = 0; kb < args.nk && ok; ++kb)
                        for (int gi = 0; gi < ng; ++gi) {
                            // (a fresh barrier counts as past its odd phase: the first round does not wait)
                            if (!mbar_wait(&empty_bar[s], ph ^ 1, tword, 21)) {
                                ok = false;
                                break;
                            }
                            uint8_t *base = smem + (size_t)s * OZ_SLOT_BYTES;
                            mbar_arrive_expect_tx(&full_bar[s], (uint32_t)OZ_SLOT_BYTES);
                            tma_load_2d(&mapA, &full_bar[s], base, (kb * S + 4 * gi) * 16, ar);
                            tma_load_2d(&mapB, &full_bar[s], base + OZ_A_BYTES, (kb * S + 4 * gi) * 16, br);
                            if (filled < ST) ++filled;
                            if (++s == ST) s = 0, ph ^= 1;
                        }
                }
            }
            if (!ok)   // the copies in flight, newest first
                for (int q = 0; q < filled; ++q) {
                    if (s == 0) s = ST, ph ^= 1;
                    --s;
                    mbar_wait(&full_bar[s], ph, tword, 22);
                }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = instr_desc_f16(1, OZ_BM, OZ_BN);
            int s = 0;
            uint32_t ph = 0;
            uint32_t used = 0, uph = 0;   // per accumulator slot: used before; parity of its last release
            unsigned long long nmma = 0;
            bool ok = true;
            for (int L = oz_first<SPLIT>(args), it = 0; L < ntiles && ok; L += oz_step<SPLIT>(args), ++it) {
                int gr, gc, ar, br;
                if (!oz_tile(args, L, &gr, &gc, &ar, &br)) continue;
                const int lc = tile_lc(it, ar, br);
#pragma unroll
                for (int pi = 0; pi < PASSES; ++pi) {
                    const int ps = LOW_FIRST ? PASSES - 1 - pi : pi;
                    if (!ok || Cfg::lev_lo(ps) > lc) break;
                    // every slot of the pass takes part in the release protocol; only levels <= lc get MMAs
                    const int llo = Cfg::lev_lo(ps), lhi = Cfg::lev_hi(ps);
                    const int ng = (min(Cfg::tmax(ps), lc - 1) + 3) / 4;
                    for (int kb = 0; kb < args.nk; ++kb) {
                        uint64_t da[NG], db[NG];
                        uint64_t *done[NG];
#pragma unroll
                        for (int gi = 0; gi < NG; ++gi) {
                            if (gi >= ng) continue;
                            if (!mbar_wait(&full_bar[s], ph, tword, 23)) {
                                ok = false;
                                break;
                            }
                            const uint32_t a0 = smem_u32(smem + (size_t)s * OZ_SLOT_BYTES);
                            da[gi] = smem_desc_sw128(a0);
                            db[gi] = smem_desc_sw128(a0 + OZ_A_BYTES);
                            done[gi] = &empty_bar[s];
                            if (++s == ST) s = 0, ph ^= 1;
                        }
                        if (!ok) break;
                        fence_after_sync();
#pragma unroll
                        for (int l = 2; l <= S + 1; ++l) {
                            if (l < llo || l > lhi) continue;
                            const int tlo = (l - S > 1) ? l - S : 1, thi = (l - 1 < S) ? l - 1 : S;
                            const int slot = l - llo;
                            if (kb == 0) {
                                if (used >> slot & 1) {
                                    // the epilogue has read this slot's previous contents (per-slot release)
                                    if (!mbar_wait(&slot_empty[slot], uph >> slot & 1, tword, 25)) {
                                        ok = false;
                                        break;
                                    }
                                    fence_after_sync();
                                    uph ^= 1u << slot;
                                }
                                used |= 1u << slot;
                            }
                            if (l > lc) continue;
                            nmma += (unsigned long long)(thi - tlo + 1);
#pragma unroll
                            for (int t = tlo; t <= thi; ++t) {
                                const int u = l - t;
                                // slice t: group (t - 1) / 4, 32-byte step (t - 1) % 4 (the start-address field
                                // counts 16 bytes; no carry: smem addresses < 2^18)
                                mma_f16(tmem + (uint32_t)(slot * OZ_BN), da[(t - 1) / 4] + (uint64_t)(((t - 1) % 4) * 2),
                                        db[(u - 1) / 4] + (uint64_t)(((u - 1) % 4) * 2), idesc,
                                        (kb != 0 || t != tlo) ? 1u : 0u);
                            }
                        }
                        if (!ok) break;
#pragma unroll
                        for (int gi = 0; gi < NG; ++gi)
                            if (gi < ng) mma_commit(done[gi]);
                    }
                    if (!ok) break;
                    mma_commit(&acc_full);
                }
            }
            // every MMA issued so far has completed before TMEM can be freed
            mma_commit(&drain_bar);
            mbar_wait(&drain_bar, 0, tword, 26);
            if (args.tc_flops && (!SPLIT || blockIdx.x % args.split == 0))   // (a shared tile counts once)
                atomicAdd(args.tc_flops, nmma * (unsigned long long)(2 * OZ_BM * OZ_BN * 16));
        }
        __syncwarp();
    } else {
        // epilogue: warps 2..9; TMEM lane quarter q = warp % 4 (tile rows 32q..), column half h
        const int q = warp % 4, h = (warp - 2) / 4;
        const int row = q * 32 + lane;
        int job = 0;
        bool ok = true;
        // C entries of this thread's row come through shared memory by cp.async, OZ_CD columns ahead, the first of
        // them while the tile's MMAs still run: a load of C takes about a microsecond, and with four columns in
        // flight these waits were 28 us a pass
        double *cbuf = c_stage + (warp - 2) * OZ_CD * 32 + lane;
        for (int L = oz_first<SPLIT>(args), it = 0; L < ntiles && ok; L += oz_step<SPLIT>(args), ++it) {
            int gr, gc, ar, br;
            if (!oz_tile(args, L, &gr, &gc, &ar, &br)) continue;
            const int lc = tile_lc(it, ar, br);
            const int grow = gr + row;
            const int er = (grow < args.m_end) ? args.ea[ar + row] : 0;
            double *cp = args.C + (long long)(gc + h * CPT) * args.ldc + grow;
            const int *eb = args.eb + br + h * CPT;
            const int c_all = min(CPT, args.n_end - (gc + h * CPT));
            const int eb0 = lane < c_all ? eb[lane] : 0, eb1 = 32 + lane < c_all ? eb[32 + lane] : 0;
            int c_end = c_all;   // this thread's columns, in a triangle up to its row
            if (args.tri) c_end = min(c_end, grow - (gc + h * CPT) + 1);
            if (grow >= args.m_end) c_end = 0;
            int c_begin = 0;
            if constexpr (SPLIT) {
                c_begin = (int)(blockIdx.x % args.split) * (CPT / args.split);
                c_end = min(c_end, c_begin + CPT / args.split);
            }
            // the warp's columns: what lies past them is not converted or stored (a product of few columns or rows
            // would pay for a whole tile's FP64 operations, 8 us a pass)
            const int c_warp = __reduce_max_sync(0xffffffffu, max(c_end, 0));
#pragma unroll
            for (int pi = 0; pi < PASSES; ++pi) {
                const int ps = LOW_FIRST ? PASSES - 1 - pi : pi;
                if (Cfg::lev_lo(ps) > lc) break;
                const bool over = args.overwrite && pi == 0;
                const int c_load = over ? 0 : c_end;
                const double *cs = cp;   // the next column to stage
                auto stage = [&](int j0) {
#pragma unroll
                    for (int jj = 0; jj < OZ_CQ; ++jj, cs += args.ldc)
                        if ((!SPLIT || j0 + jj >= c_begin) && j0 + jj < c_load) cp_async8(&cbuf[(j0 + jj) % OZ_CD * 32], cs);
                    cp_async_commit();
                };
#pragma unroll
                for (int j0 = 0; j0 < OZ_CD; j0 += OZ_CQ) stage(j0);
                ok = mbar_wait(&acc_full, (uint32_t)(job & 1), tword, 24);
                ok = __all_sync(0xffffffffu, ok);   // every lane takes part in tcgen05.ld
                if (!ok) break;
                fence_after_sync();
                const int llo = Cfg::lev_lo(ps), lhi = Cfg::lev_hi(ps);
                long long acc[CPT];
#pragma unroll
                for (int l = 2; l <= S + 1; ++l) {
                    if (l < llo || l > lhi) continue;
                    const bool first = ((l - 2) % OZ_LPW) == 0;
                    const bool live = l <= lc;   // a cut level's slot holds stale values: taken as 0
#pragma unroll
                    for (int c32 = 0; c32 < CPT / 32; ++c32) {
                        float v[32];
                        tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((l - llo) * OZ_BN + h * CPT + c32 * 32),
                                  v);
                        if (c32 == CPT / 32 - 1) {
                            // this warp has read the slot: the MMAs of the next job may overwrite it
                            fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&slot_empty[l - llo]);
                        }
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const long long d = live ? (long long)__float2int_rn(v[j]) : 0;   // exact, below 2^24
                            acc[c32 * 32 + j] = first ? d : acc[c32 * 32 + j] * 128 + d;
                        }
                    }
                }
                ++job;
                double *cw = cp;
#pragma unroll
                for (int j0 = 0; j0 < CPT; j0 += OZ_CQ) {
                    if (j0 >= c_warp) break;
                    if (SPLIT && j0 < c_begin) {   // another CTA's
                        cw += OZ_CQ * args.ldc;
                        stage(j0 + OZ_CD);
                        continue;
                    }
                    cp_async_wait<OZ_CD / OZ_CQ - 1>();
#pragma unroll
                    for (int jj = 0; jj < OZ_CQ; ++jj, cw += args.ldc) {
                        const int j = j0 + jj;
                        // the columns' exponents sit in the warp's lanes
                        const int e = er + __shfl_sync(0xffffffffu, j < 32 ? eb0 : eb1, j % 32);
                        double c = over ? 0.0 : cbuf[j % OZ_CD * 32];
                        c = fma(-(double)acc[j], pow2i(e + 2 - 7 * lhi), c);
                        if (j < c_end) *cw = c;
                    }
                    if (j0 + OZ_CD < CPT)
                        stage(j0 + OZ_CD);
                    else
                        cp_async_commit();   // an empty group keeps the count
                }
            }
        }
        cp_async_wait<0>();
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        fence_after_sync();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS)
                     : "memory");
    }
}

// Digit slices of rows [0, R) of the column-major FP64 panel P (ld), columns
// [k0, k0 + kc) for the K chunk blockIdx.y (kc = kchunk, the last one
// shorter): digit t (from 0) of row r, column k at out[(r Kp + k / 16 * 16) S + 16 t + k % 16]
// (BF16, zero for k beyond the panel), the row exponent at exps[chunk * exp_stride + r].
// Per 32-row block b the largest exponent of its non-zero rows goes to
// bexps[2 chunk bstride + b], and that of its non-zero rows below ref_rows to
// bexps[(2 chunk + 1) bstride + b] (OZ_E_NONE where there is none).
// One CTA per 32 rows: a column sweep for the row maxima, then 32 x 32
// tiles through shared memory so that each slice row is written along K, four
// digits (8 bytes) per store.  Everything runs on the integer pipes: the
// maxima compare the magnitudes' bit patterns (ordered like the values), and
// X = rint(x 2^(7S - 1 - e)) is the 53-bit significand shifted by the
// difference of exponents with round-to-nearest-even, the same integer the
// FP64 product and conversion would give.  64 in every digit is added first, so
// that the balanced digits come out as plain bit fields instead of one after
// the other with their borrows; two at a time become BF16 by one subtraction,
// and the next tile is loaded meanwhile.  Bound by the integer pipes and the
// loads' latency: 12,290 rows of 512 to 8 slices 165 -> 65 us (200 MB: 30).
__device__ __forceinline__ long long oz_scaled_int(unsigned long long b, int k) {
    // rint(x 2^k) for the double with bits b (|x 2^k| < 2^62)
    const int E = (int)((b >> 52) & 0x7FF);
    if (E == 0) return 0;   // zero or subnormal: below 2^-1022, far below 1/2 after any scaling used here
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = 1075 - E - k;   // x 2^k = m 2^-sh
    unsigned long long q;
    if (sh <= 0) {
        q = m << (-sh);
    } else if (sh >= 64) {
        q = 0;
    } else {
        q = (m + ((1ull << (sh - 1)) - 1) + ((m >> sh) & 1)) >> sh;   // to nearest, ties to even
    }
    return (b >> 63) ? -(long long)q : (long long)q;
}

// Two digits d = u - 64 as BF16 (exact) from u in 0 .. 128: the bits 0x4300 + u are 128 + u, less 192.
__device__ __forceinline__ unsigned int oz_digit_pair(unsigned int u0, unsigned int u1) {
    const unsigned int b = 0x43004300u + u0 + (u1 << 16);
    const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162 *>(&b), __float2bfloat162_rn(192.0f));
    return *reinterpret_cast<const unsigned int *>(&d);
}

__global__ void __launch_bounds__(256) k_oz_slice(const double *P, long long ld, int R, int K, int kchunk, int S,
                                                  __nv_bfloat16 *out, int Kp, int *exps,
                                                  long long exp_stride, int *bexps, long long bstride, int ref_rows,
                                                  const DevStatus *st) {
    __shared__ unsigned long long tile[32][33];
    __shared__ unsigned long long red[8][32];
    __shared__ int ex[32];
    __shared__ int skip;
    if (threadIdx.x == 0) skip = *(volatile const int *)&st->info;
    __syncthreads();
    if (skip) return;
    const int r0 = blockIdx.x * 32;
    const int kbeg = blockIdx.y * kchunk, kend = min(K, kbeg + kchunk);
    const int kpad_end = min(Kp, kbeg + (kchunk + OZ_KALIGN - 1) / OZ_KALIGN * OZ_KALIGN);
    const int rr = threadIdx.x % 32, g = threadIdx.x / 32;
    const unsigned long long *Pb = reinterpret_cast<const unsigned long long *>(P);
    constexpr unsigned long long MAG = 0x7FFFFFFFFFFFFFFFull;
    unsigned long long mx = 0;
    if (r0 + rr < R)
#pragma unroll 8
        for (int k = kbeg + g; k < kend; k += 8) mx = max(mx, Pb[(long long)k * ld + r0 + rr] & MAG);
    red[g][rr] = mx;
    __syncthreads();
    if (threadIdx.x < 32) {
        unsigned long long m = red[0][rr];
        for (int q = 1; q < 8; ++q) m = max(m, red[q][rr]);
        // max |x| = f 2^e with f in [1/2, 1): |x| < 2^e on the row (e = biased exponent - 1022)
        int e = 0;
        if (m > 0) e = max((int)(m >> 52) - 1022, -960);
        ex[rr] = e;
        if (r0 + rr < R) exps[(long long)blockIdx.y * exp_stride + r0 + rr] = e;
        const bool live = r0 + rr < R && m > 0;
        int eall = live ? e : OZ_E_NONE, eref = (live && r0 + rr < ref_rows) ? e : OZ_E_NONE;
        for (int o = 16; o > 0; o >>= 1) {
            eall = max(eall, __shfl_xor_sync(0xffffffffu, eall, o));
            eref = max(eref, __shfl_xor_sync(0xffffffffu, eref, o));
        }
        if (rr == 0) {
            bexps[2LL * blockIdx.y * bstride + blockIdx.x] = eall;
            bexps[(2LL * blockIdx.y + 1) * bstride + blockIdx.x] = eref;
        }
    }
    __syncthreads();
    // this thread's row and four consecutive columns of each 32 x 32 tile
    const int r = threadIdx.x / 8, cq = (threadIdx.x % 8) * 4;
    const int kshift = 7 * S - 1 - ex[r];
    unsigned long long bias = 0;   // 64 in every digit: the digits of X + bias are those of X plus 64, none negative
    for (int t = 0; t < S; ++t) bias = bias * 128 + 64;
    unsigned long long nx[4];   // the next tile, loaded during this one's digits
    auto fetch = [&](int c0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = c0 + g + 8 * i;
            nx[i] = (r0 + rr < R && c < kend) ? Pb[(long long)c * ld + r0 + rr] : 0ull;
        }
    };
    fetch(kbeg);
    for (int c0 = kbeg; c0 < kpad_end; c0 += 32) {
#pragma unroll
        for (int i = 0; i < 4; ++i) tile[g + 8 * i][rr] = nx[i];
        __syncthreads();
        if (c0 + 32 < kpad_end) fetch(c0 + 32);
        if (r0 + r < R) {
            unsigned int lo[4], hi[4], lead[4];   // digits 0 .. 3 and 4 .. 7 from the least one, the leading one
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const unsigned long long y = (unsigned long long)oz_scaled_int(tile[cq + i][r], kshift) + bias;
                lo[i] = (unsigned int)y;
                hi[i] = (unsigned int)(y >> 28);
                lead[i] = (unsigned int)(y >> (7 * (S - 1)));
            }
            const long long at = ((long long)(r0 + r) * Kp + (c0 + cq) / 16 * 16) * S + cq % 16;
            unsigned int *o = reinterpret_cast<unsigned int *>(out + at);
#pragma unroll
            for (int t = 0; t < 7; ++t)
                if (t < S - 1) {
                    unsigned int u[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) u[i] = ((t < 4 ? lo[i] : hi[i]) >> (7 * (t % 4))) & 127;
                    *reinterpret_cast<uint2 *>(o + (S - 1 - t) * 8) =
                        make_uint2(oz_digit_pair(u[0], u[1]), oz_digit_pair(u[2], u[3]));
                }
            *reinterpret_cast<uint2 *>(o) = make_uint2(oz_digit_pair(lead[0], lead[1]), oz_digit_pair(lead[2], lead[3]));
        }
        __syncthreads();
    }
}

template <int S, bool LOW_FIRST = false>
cudaError_t launch_oz_kernel(const CUtensorMap &ma, const CUtensorMap &mb, const OzArgs &a, int grid,
                             cudaStream_t s) {
    static_assert(OZ_SLOTS >= 2 * OzCfg<S>::NG, "shared memory holds fewer than two chunks");
    auto *kernel = a.split > 1 ? k_oz_update<S, LOW_FIRST, true> : k_oz_update<S, LOW_FIRST, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM);
    if (e != cudaSuccess) return e;
    kernel<<<grid, OZ_THREADS, OZ_SMEM, s>>>(ma, mb, a);
    return cudaGetLastError();
}

// 2-D tensor map over the digits of a K chunk: (interleaved columns, row), box 64 (four slices of 16 columns:
// one 128-byte line; past the chunk's end zeros) x rows_box, swizzled by lines.  Every box starts at a multiple of
// 16 columns, 32 bytes.
cudaError_t slice_map(CUtensorMap *map, const OzSlices &sl, int chunk, int rows_box) {
    tc::EncodeTiledFn enc = tc::encode_fn();
    if (!enc) return cudaErrorNotSupported;
    void *base = (__nv_bfloat16 *)sl.d + (size_t)chunk * sl.kchunk * sl.S;   // kchunk is a multiple of 32
    cuuint64_t dims[2] = {(cuuint64_t)std::min(sl.kchunk, sl.Kp - chunk * sl.kchunk) * sl.S, (cuuint64_t)sl.valid};
    cuuint64_t strides[1] = {(cuuint64_t)sl.Kp * sl.S * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)rows_box};
    cuuint32_t es[2] = {1, 1};
    CUresult cr = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return cr == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

int oz_kmax(int S) { return (4096 / S) / OZ_KALIGN * OZ_KALIGN; }

size_t oz_slices_bytes(long long rows, int K, int S) {
    const long long Kp = (K + OZ_KALIGN - 1) / OZ_KALIGN * OZ_KALIGN;
    const int nchunk = (K + oz_kmax(S) - 1) / oz_kmax(S);
    return (size_t)S * (size_t)rows * (size_t)Kp * 2 + sizeof(int) * (size_t)rows * nchunk +
           sizeof(int) * 2 * (size_t)((rows + 31) / 32) * nchunk + 768;
}

OzSlices oz_slices_carve(void *ws, long long rows, int K, int S) {
    OzSlices o;
    o.S = S;
    o.rows = rows;
    o.K = K;
    o.kchunk = oz_kmax(S);
    o.Kp = (K + OZ_KALIGN - 1) / OZ_KALIGN * OZ_KALIGN;
    o.nchunk = (K + o.kchunk - 1) / o.kchunk;
    o.valid = rows;
    o.d = ws;
    uintptr_t e = (uintptr_t)ws + (size_t)o.S * rows * o.Kp * 2;
    o.e = (int *)((e + 255) & ~(uintptr_t)255);
    o.bstride = (rows + 31) / 32;
    o.be = (int *)(((uintptr_t)(o.e + rows * o.nchunk) + 255) & ~(uintptr_t)255);
    o.ref_rows = -1;
    return o;
}

cudaError_t oz_slice(const double *P, long long ld, int R, const OzSlices &o, const DevStatus *st, cudaStream_t s) {
    if (R <= 0) return cudaSuccess;
    if (R > o.rows || R > o.valid) return cudaErrorInvalidValue;
    dim3 grid((R + 31) / 32, o.nchunk);
    KScope ks(GEO_K_AUX, s, 0.0, (double)R * o.K * (16.0 + 2.0 * o.S));
    k_oz_slice<<<grid, 256, 0, s>>>(P, ld, R, o.K, o.kchunk, o.S, (__nv_bfloat16 *)o.d, o.Kp, o.e,
                                    o.rows, o.be, o.bstride, o.ref_rows < 0 ? R : (int)std::min<long long>(o.ref_rows, R),
                                    st);
    return cudaGetLastError();
}

cudaError_t oz_update(const OzSlices &A, const OzSlices &B, double *C, long long ldc, int r0, int c0, int rows,
                      int cols, int m_end, int n_end, int a_off, int b_off, int tri, int grid_cap, DevStatus *st,
                      cudaStream_t s, int overwrite, int cut) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    if (A.S != B.S || A.K != B.K || A.S < 3 || A.S > 8) return cudaErrorInvalidValue;
    if (cut && overwrite) return cudaErrorInvalidValue;   // a skipped tile would leave C unwritten
    const int S = A.S;
    OzArgs a;
    a.C = C;
    a.ldc = ldc;
    a.r0 = r0;
    a.c0 = c0;
    a.m_end = m_end;
    a.n_end = n_end;
    a.mt = (rows + OZ_BM - 1) / OZ_BM;
    a.nt = (cols + OZ_BN - 1) / OZ_BN;
    a.tri = tri;
    a.a_off = a_off;
    a.overwrite = 0;
    a.b_off = b_off;
    a.st = st;
    a.cut = cut ? 1 : 0;
    a.nba = (int)((A.valid + 31) / 32);
    a.nbb = (int)((B.valid + 31) / 32);
    a.tc_flops = t_prof ? t_prof->d_tc_flops : nullptr;
    const long long ntiles = (long long)a.mt * a.nt;
    if (ntiles > (1LL << 30)) return cudaErrorInvalidValue;   // the kernel counts tiles in 32 bits
    const int ctas = std::max(1, std::min(grid_cap, tc::num_sms()));
    // few tiles: the epilogue's FP64 operations, 8 us a pass over a tile, on two or four SMs each (the MMAs are done in
    // every one of them; C 100 x 1000, K = 32, 5 slices 76 -> 62 us a call, 64
    // with 64-column tiles)
    a.split = 1;
    while (a.split < 4 && ntiles * a.split * 2 <= ctas) a.split *= 2;
    const int grid = (int)std::min<long long>(ntiles * a.split, ctas);
    // algorithmic work: 2 K flops per output written (lower triangle when tri)
    const double rr = rows, cc = cols;
    const double outs = tri ? std::max(0.0, rr * cc - cc * (cc - 1.0) / 2.0) : rr * cc;
    for (int ch = 0; ch < A.nchunk; ++ch) {
        const int kc = std::min(A.kchunk, A.K - ch * A.kchunk);
        a.nk = (kc + 15) / 16;
        a.ea = A.e + (long long)ch * A.rows;
        a.eb = B.e + (long long)ch * B.rows;
        a.ba = A.be + 2LL * ch * A.bstride;
        a.ra = a.ba + A.bstride;
        a.bb = B.be + 2LL * ch * B.bstride;
        a.rb = a.bb + B.bstride;
        CUtensorMap ma, mb;
        cudaError_t e;
        if ((e = slice_map(&ma, A, ch, OZ_BM)) != cudaSuccess ||
            (e = slice_map(&mb, B, ch, OZ_BN)) != cudaSuccess)
            return e;
        a.overwrite = (overwrite && ch == 0) ? 1 : 0;   // later K chunks accumulate onto the first
        KScope ks(GEO_K_TCGEMM, s, 2.0 * kc * outs, 16.0 * outs + 2.0 * S * kc * (rr + cc));
        switch (S) {
            case 3: e = launch_oz_kernel<3>(ma, mb, a, grid, s); break;
            case 4: e = launch_oz_kernel<4>(ma, mb, a, grid, s); break;
            // five slices without the cut add their last level first (the sums' rounding is part of the form's result)
            case 5: e = cut ? launch_oz_kernel<5>(ma, mb, a, grid, s) : launch_oz_kernel<5, true>(ma, mb, a, grid, s); break;
            case 6: e = launch_oz_kernel<6>(ma, mb, a, grid, s); break;
            case 7: e = launch_oz_kernel<7>(ma, mb, a, grid, s); break;
            default: e = launch_oz_kernel<8>(ma, mb, a, grid, s); break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

constexpr int OZ_TILE_IB = 64;   // inner block of the diagonal tiles (the rank of their updates)

size_t oz_chol_workspace_bytes(int nrows, int nb, int S) {
    return oz_slices_bytes((long long)nrows + 128, nb, S) + oz_slices_bytes(nb, nb, S) + sizeof(double) * (size_t)nb * nb +
           oz_slices_bytes(nb, OZ_TILE_IB, S) + 1280;
}

namespace {
// The rank-64 updates inside a diagonal tile as emulated products: the rows
// below the inner block (their columns kA .. kA + k) as digit slices, then the
// lower triangle of the rest of the tile.  Runs on the side stream with at most
// `sms` CTAs, beside the trailing update.
struct TileUpdate {
    OzSlices sl;
    int sms;
};

cudaError_t tile_update(const TileUpdate &t, double *A, long long ld, int rC, int m, int kA, int k, DevStatus *st,
                        cudaStream_t s) {
    if (m <= 0 || k <= 0) return cudaSuccess;
    if (k > t.sl.K || m > t.sl.rows) return cudaErrorInvalidValue;
    OzSlices p = t.sl;
    p.K = k;
    p.nchunk = (k + p.kchunk - 1) / p.kchunk;
    p.valid = m;
    cudaError_t e = oz_slice(A + (long long)kA * ld + rC, ld, m, p, st, s);
    if (e != cudaSuccess) return e;
    return oz_update(p, p, A, ld, rC, rC, m, m, rC + m, rC + m, 0, 0, 1, t.sms, st, s, 0, 0);
}
}  // namespace

// Right-looking over panels of width nb with a lookahead of one (as the mixed
// form).  Step j slices its solved panel (the rows below the diagonal tile,
// right-hand-side rows included) and updates the next panel's tile column
// first; on a high-priority second stream the next diagonal tile is factored
// and inverted, W = -L_kk^-1, in one native FP64 launch while the rest of the
// trailing update runs (its persistent launch leaves it the SMs it needs).
// After the join the rows below the new diagonal tile are solved as one
// emulated product, L_ik = A_ik L_kk^-T = -(A_ik W'), written over A_ik.
// Every trailing update and panel solve is emulated; POTRF of the diagonal
// tiles and their inversion are native FP64, and so is the last panel.
constexpr double OZ_REST_RATE = 1.2e9;   // BF16 flops per us of a trailing update, for the split of the SMs

cudaError_t chol_oz_factor(double *A, long long ld, int N, int nrows, int nb, int S, int cut, void *ws,
                           size_t ws_bytes, DevStatus *st, int *sync, cudaStream_t s) {
    if (nb < 64 || nb % 64 != 0 || nb > 1024 || S < 3 || S > 8) return cudaErrorInvalidValue;
    if (ws_bytes < oz_chol_workspace_bytes(nrows, nb, S)) return cudaErrorInvalidValue;
    const OzSlices sl = oz_slices_carve(ws, (long long)nrows + 128, nb, S);
    uintptr_t wp = ((uintptr_t)ws + oz_slices_bytes((long long)nrows + 128, nb, S) + 255) & ~(uintptr_t)255;
    const OzSlices slw0 = oz_slices_carve((void *)wp, nb, nb, S);
    wp = (wp + oz_slices_bytes(nb, nb, S) + 255) & ~(uintptr_t)255;
    double *W = (double *)wp;   // nb x nb, ld nb
    wp = (wp + sizeof(double) * (size_t)nb * nb + 255) & ~(uintptr_t)255;
    const OzSlices tile_sl = oz_slices_carve((void *)wp, nb, OZ_TILE_IB, S);
    // with FP64-class slices a diagonal tile is one native launch; with fewer its own rank-64 updates
    // are emulated like every other update (their rounding is part of that form's result)
    const bool fused = S >= 7;
    const int order = fused ? GEO_CHOL_NATIVE : GEO_CHOL_BLOCK64;
    int prio_lo = 0, prio_hi = 0;
    cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi);
    cudaStream_t s2 = nullptr;
    cudaEvent_t e_upd = nullptr, e_pan = nullptr;
    cudaError_t e;
    if ((e = cudaStreamCreateWithPriority(&s2, cudaStreamNonBlocking, prio_hi)) != cudaSuccess) return e;
    if ((e = cudaEventCreateWithFlags(&e_upd, cudaEventDisableTiming)) != cudaSuccess ||
        (e = cudaEventCreateWithFlags(&e_pan, cudaEventDisableTiming)) != cudaSuccess) {
        cudaStreamDestroy(s2);
        if (e_upd) cudaEventDestroy(e_upd);
        return e;
    }
    const int all = tc::num_sms();
    // rows [x0, x1) of panel [t0, t0 + jb) <- A L^-T with W = -L^-1 already in place
    auto panel_solve = [&](int t0, int jb, int x0, int x1, cudaStream_t st_) -> cudaError_t {
        if (x0 >= x1) return cudaSuccess;
        OzSlices p = sl, q = slw0;
        p.K = q.K = jb;
        p.nchunk = q.nchunk = (jb + p.kchunk - 1) / p.kchunk;
        p.valid = x1 - x0;
        q.valid = jb;
        cudaError_t r;
        if ((r = oz_slice(A + (long long)t0 * ld + x0, ld, x1 - x0, p, st, st_)) != cudaSuccess ||
            (r = oz_slice(W, nb, jb, q, st, st_)) != cudaSuccess)
            return r;
        return oz_update(p, q, A, ld, x0, t0, x1 - x0, jb, x1, t0 + jb, 0, 0, 0, all, st, st_, 1, 0);
    };
    // factorisation of the diagonal tile [t0, t0 + jb) and its inverse on at most sms SMs
    auto diag = [&](int t0, int jb, int sms, cudaStream_t st_) -> cudaError_t {
        if (fused) return chol64_panel(A, ld, t0, jb, t0 + jb, t0 + jb, st, sync, st_, true, W, nb, sms);
        cudaError_t r;
        for (int c0 = t0; c0 < t0 + jb; c0 += OZ_TILE_IB) {
            const int cb = std::min(OZ_TILE_IB, t0 + jb - c0);
            if ((r = chol64_panel(A, ld, c0, cb, c0 + cb, t0 + jb, st, sync, st_, true, nullptr, 0, sms,
                                  GEO_CHOL_PLAIN)) != cudaSuccess ||
                (r = tile_update(TileUpdate{tile_sl, sms > 0 ? sms : all}, A, ld, c0 + cb, t0 + jb - c0 - cb, c0, cb, st,
                                 st_)) != cudaSuccess)
                return r;
        }
        return chol64_panel(A, ld, t0, jb, t0 + jb, t0 + jb, st, sync, st_, false, W, nb, sms, GEO_CHOL_PLAIN);
    };
    auto run = [&]() -> cudaError_t {
        cudaError_t r;
        const int jb0 = std::min(nb, N);
        if (jb0 == N)   // one tile: native
            return chol64_panel(A, ld, 0, N, N, nrows, st, sync, s, true, nullptr, 0, 0, order);
        // the launches below write W's lower part only
        if ((r = cudaMemsetAsync(W, 0, sizeof(double) * (size_t)nb * nb, s)) != cudaSuccess) return r;
        if ((r = diag(0, jb0, 0, s)) != cudaSuccess || (r = panel_solve(0, jb0, jb0, nrows, s)) != cudaSuccess)
            return r;
        for (int j0 = 0;;) {
            const int jb = std::min(nb, N - j0);
            const int t0 = j0 + jb;
            if (t0 >= N) break;
            // the solved panel's rows below the diagonal tile as digit slices
            OzSlices p = sl;
            p.K = jb;
            p.nchunk = (jb + p.kchunk - 1) / p.kchunk;
            p.valid = nrows - t0;
            p.ref_rows = N - t0;   // the reference scale is the matrix's, not the right-hand side rows'
            if ((r = oz_slice(A + (long long)j0 * ld + t0, ld, nrows - t0, p, st, s)) != cudaSuccess) return r;
            const int n1 = std::min(N, t0 + nb);
            // the next panel's tile column: rows [t0, nrows), cols [t0, n1)
            if ((r = oz_update(p, p, A, ld, t0, t0, nrows - t0, n1 - t0, nrows, n1, 0, 0, 1, all, st, s, 0, cut)) !=
                cudaSuccess)
                return r;
            if (n1 >= N) {
                // last panel: diagonal tile + RHS rows
                r = chol64_panel(A, ld, t0, N - t0, N, nrows, st, sync, s, true, nullptr, 0, 0, order);
                if (r != cudaSuccess) return r;
                j0 = t0;
                continue;
            }
            if ((r = cudaEventRecord(e_upd, s)) != cudaSuccess) return r;
            if ((r = cudaStreamWaitEvent(s2, e_upd, 0)) != cudaSuccess) return r;
            const double left = N - n1;
            const double rest_us = left * left * jb * S * (S + 1) / 2.0 / OZ_REST_RATE;
            // with its updates emulated the diagonal tile is a longer chain (about 1.3 ms for 512 columns): the
            // update's rest is the shorter side below that, and gives up SMs
            const int side = !fused && rest_us < 5.0 * (n1 - t0) ? 48 : chol64_side_sms(n1 - t0, true, rest_us);
            if ((r = diag(t0, n1 - t0, side, s2)) != cudaSuccess) return r;
            if ((r = cudaEventRecord(e_pan, s2)) != cudaSuccess) return r;
            // the rest of the trailing update meanwhile: rows [n1, nrows), cols [n1, N)
            if ((r = oz_update(p, p, A, ld, n1, n1, nrows - n1, N - n1, nrows, N, n1 - t0, n1 - t0, 1,
                               all - side, st, s, 0, cut)) != cudaSuccess)
                return r;
            if ((r = cudaStreamWaitEvent(s, e_pan, 0)) != cudaSuccess) return r;
            if ((r = panel_solve(t0, n1 - t0, n1, nrows, s)) != cudaSuccess) return r;
            j0 = t0;
        }
        return cudaSuccess;
    };
    e = run();
    if (e != cudaSuccess) cudaStreamSynchronize(s2);
    cudaEventDestroy(e_upd);
    cudaEventDestroy(e_pan);
    cudaStreamDestroy(s2);
    return e;
}

// C (m x n) -= A (m x k) B (n x k)' for column-major FP64 operands, through
// the digit slices of A's rows and B's rows (workspace ws of
// oz_gemm_workspace_bytes).
size_t oz_gemm_workspace_bytes(int m, int n, int k, int S) {
    return oz_slices_bytes(m, k, S) + oz_slices_bytes(n, k, S) + 256;
}

cudaError_t oz_gemm(int m, int n, int k, const double *A, long long lda, const double *B, long long ldb, double *C,
                    long long ldc, int S, void *ws, DevStatus *st, cudaStream_t s) {
    if (m <= 0 || n <= 0 || k <= 0) return cudaSuccess;
    const OzSlices sa = oz_slices_carve(ws, m, k, S);
    uintptr_t wb = (uintptr_t)ws + oz_slices_bytes(m, k, S);
    wb = (wb + 255) & ~(uintptr_t)255;
    const OzSlices sb = oz_slices_carve((void *)wb, n, k, S);
    cudaError_t e;
    if ((e = oz_slice(A, lda, m, sa, st, s)) != cudaSuccess || (e = oz_slice(B, ldb, n, sb, st, s)) != cudaSuccess)
        return e;
    return oz_update(sa, sb, C, ldc, 0, 0, m, n, m, n, 0, 0, 0, tc::num_sms(), st, s, 0, 0);
}
