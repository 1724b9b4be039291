// FP64 GEMM emulated on tcgen05 BF16 tensor cores (exact slicing in the
// manner of Ozaki, Ogita and Oishi's error-free splitting), used by the plain
// FP64 path for its large contractions.
//
// Each row i of op(A) (and each column j of op(B)) is scaled by a power of
// two 2^-e so that its entries lie in (-1, 1), then cut into NS balanced
// base-256 digits q_s in [-128, 128], every one exact in BF16:
//     a = 2^e * sum_s q_s 2^(-7 - 8s),   rounded at 2^(e - 8 NS).
// Products of digits are integers of magnitude <= 2^14.  Pairs (s, t) with
// s + t < NS are grouped by g = s + t (weight 2^(-14 - 8g)); group g holds
// g + 1 pairs, so over a K chunk of 256 the sums of groups 0-3 are at most
// 4 * 256 * 2^14 = 2^24, over one of 128 those of the groups above at most
// 8 * 128 * 2^14 = 2^24, and the tensor core's FP32 accumulation is exact.
// After each chunk the epilogue warps read the group
// sums from TMEM as integers and add them to two int64 accumulators per
// entry (groups 0-3 in units of 2^-38, the others in units of the last
// group's), which hold the sums exactly; the two are combined and rounded
// once, in integer arithmetic, at the end.  What is lost is the rounding of
// the last digits and the pairs with s + t >= NS: about 2^(1 - 8 NS) of the
// row x column scale per term.
//   NS = 7 (28 products): the factorisation's products; 2^-56 per term, the
//   level of an FP64 dot product.
//   NS = 4 (10 products): FP32 data and results; 2^-31 per term, below FP32's
//   own rounding.  Its 4 x 64 accumulator columns fit TMEM twice, so a chunk is
//   drained while the next is multiplied; with more tiles than SMs a CTA takes
//   several, its products running ahead of its epilogues.
//   NS = 8 (36 products): A_hat = U D V^T in FP64.
// These errors are relative to the largest entry of the row times that of the
// column, not to the entry computed: where an entry's own terms are far smaller
// (operands graded along k, zeros against the large ones) FMAs are the more
// accurate.  The factorisations' results are accurate in norm only, so there it
// is enough; A_hat is checked entry by entry (oz_decode).
//
// CTA tile 128 x 64; a K block of 64 stages all NS B slices and streams the
// NS A slices through a ring; TMEM holds NS x 64 FP32 group accumulators.  An
// A slice s meets all its B slices t in MMAs of up to 256 columns: the B slices
// lie one after another in shared memory and the groups s + t in TMEM, so the A
// rows are read once for up to four slices.  For NS > 4 the products of groups
// 0-3 come first in every K block, then the others, and the two halves of TMEM
// are handed over apart: the lower every four K blocks, drained while their last
// upper products run, the upper every two, drained while the next block's lower
// ones do.
// Warp 0: TMA producer, warp 1: MMA issuer, warps 2-17: drain and epilogue
// (four per TMEM lane quarter, 16 columns each).  All waits are bounded
// (EOD_ETIMEOUT on expiry).
//
// Measured (the kernel alone): 2048^3 391 us = 44 TFLOP/s of FP64, 4000 x 1600
// x 1600 479 us, 4000 x 1600 x 4000 1053 us; with both halves handed over every
// 256 terms, where the upper groups' sums could pass 2^24, 373, 459 and 999.  In
// that form, with one MMA of 64 columns per slice pair (72 cycles each instead
// of 32: shared-memory reads, 6 KB per MMA), eight drain warps and one hand-over
// per chunk: 634, 776 and 1750 us; wide MMAs alone 452, 563 and 1209; with
// sixteen drain warps 429, 530 and 1173.  What bounds it: shared-memory reads
// (4.4 thousand cycles of a K block's about 5, the MMAs alone 3.6), the drains
// that the next products wait for, the first and last chunk's, and the last wave
// of tiles.  Slicing a 2048^2 operand and its transpose: 57 us.
#include "common.cuh"
#include "instrument.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cstring>
#include <type_traits>

namespace eod {
namespace oz {

using namespace eod::tc;

constexpr int BM = 128, BN = 64, BK = 64;
constexpr int KCH = 4;                // K blocks per chunk of groups 0-3 (256 terms)
constexpr int KCH_UPPER = 2;          // and of the groups above (128), which hold up to eight pairs
static_assert(4 * KCH * BK * 16384 <= 1 << 24 && kOzSlicesFine * KCH_UPPER * BK * 16384 <= 1 << 24 && KCH == 2 * KCH_UPPER,
              "the group sums stay exact in FP32");
constexpr int UMMA_K = 16;            // K per tcgen05.mma kind::f16
constexpr int A_TILE = BM * BK * 2;   // 16 KB: one slice
constexpr int B_TILE = BN * BK * 2;   // 8 KB
constexpr int BSTAGES = 2;            // K blocks of B in flight (NS slices each)
template <int NS> struct Cfg {
    static constexpr int ASTAGES = NS == 4 ? 4 : NS == 7 ? 7 : 5;   // A slices in flight (at least 5 for NS > 4)
    static constexpr int NBUF = NS <= 4 ? 2 : 1;                     // accumulator sets in TMEM
    static constexpr int HALVES = NS <= 4 ? 1 : 2;                   // groups 0-3 and the rest, handed over apart
    static constexpr int B_SET = NS * B_TILE;
    // the sums staged for the epilogue: with NS = 4 (one accumulator, products
    // of the next tile under way) in a place of their own
    static constexpr int STAGING = NS == 4 ? 256 * 32 * 8 : 0;
    static constexpr int SMEM = BSTAGES * B_SET + ASTAGES * A_TILE + STAGING + 1024 + 256;
    static_assert(NS == 4 || BSTAGES * B_SET + ASTAGES * A_TILE >= 256 * 32 * 16, "the epilogue's staging");
};
constexpr int kMaxSlices = kOzSlicesFine;
constexpr uint32_t TMEM_COLS = 512;   // NS x 64 used
constexpr int DRAIN = 16 * 32;            // drain threads
constexpr int NTHREADS = 64 + DRAIN;      // producer, MMA issuer, drain warps
constexpr int ECOLS = BN * 128 / DRAIN;   // columns per drain warp

struct Maps {
    CUtensorMap a[kMaxSlices];
    CUtensorMap b[kMaxSlices];
};

struct Params {
    int64_t M, N;
    int64_t kblocks, kb_per_split;
    const int *ea, *eb;       // row exponents of op(A), column exponents of op(B) (or null:
    int ea_fixed, eb_fixed;   // then every row / column uses the fixed exponent)
    double alpha, beta;
    double *C;                // output (or split partials when split_stride > 0)
    float *Cf;                // FP32 output instead of C (EPI_STORE without split partials)
    int64_t ldc, split_stride;
    const double *R;          // EPI_ERR reference
    int64_t ldr;
    double *errp;
    int *err_flag;
    const int *skip;          // nothing is done where this is set (null: always done)
    int upper_only;           // store only entries with row <= col
    int a_tri, b_tri;         // op(A) / op(B) upper triangular: skip their zero K blocks
    int64_t gm, tiles;        // NS = 4: tile rows, and the tiles a CTA strides over (0: one tile per CTA)
};

// The tile and K blocks of step t of this CTA; false past its last one.
template <bool MANY>
struct Tile {
    int64_t m0, n0, kb0, kb1;
    __device__ __forceinline__ bool at(const Params &p, int64_t t) {
        if (MANY && p.tiles > 0) {
            const int64_t i = blockIdx.x + t * gridDim.x;
            if (i >= p.tiles) return false;
            n0 = i / p.gm;
            m0 = (i - n0 * p.gm) * BM;
            n0 *= BN;
        } else {
            if (t > 0) return false;
            m0 = (int64_t)blockIdx.x * BM;
            n0 = (int64_t)blockIdx.y * BN;
        }
        kb0 = (int64_t)blockIdx.z * p.kb_per_split;
        kb1 = kb0 + p.kb_per_split;
        if (kb1 > p.kblocks) kb1 = p.kblocks;
        if (p.a_tri && kb0 < m0 / BK) kb0 = m0 / BK;              // op(A)(i, k) = 0 for k < i
        if (p.b_tri && kb1 > (n0 + BN + BK - 1) / BK) kb1 = (n0 + BN + BK - 1) / BK;   // op(B)(k, j) = 0 for k > j
        if (kb1 < kb0 || (p.upper_only && m0 >= n0 + BN)) kb1 = kb0;
        return true;
    }
};

// m 2^e for a result outside the normal range's middle (kept out of line: its
// FP64 instructions would otherwise be issued, predicated, for every entry)
__device__ __noinline__ double far_scale(unsigned long long m, int e) { return ldexp((double)m, e); }

// (hi 2^SH + lo) 2^e as a double, rounded once to nearest (ties to even), in
// integer arithmetic: an FP64 instruction costs a warp 64 cycles here, and a
// tile has 8192 entries.  |hi| < 2^62.
template <int SH>
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int e) {
    // magnitude: h 2^SH + r, 0 <= r < 2^SH
    long long h = hi + (lo >> SH);
    unsigned long long r = (unsigned long long)lo & ((1ull << SH) - 1);
    const unsigned long long sign = (unsigned long long)h & (1ull << 63);
    if (h < 0) {
        h = -h - (r ? 1 : 0);
        r = r ? (1ull << SH) - r : 0ull;
    }
    if (h == 0) {   // all of it in r (< 2^SH <= 2^32): exact
        h = (long long)r;
        r = 0;
        e -= SH;
        if (h == 0) return 0.0;
    }
    // normalise to a leading one at bit 63; what r holds below goes in behind h
    const int lz = __clzll(h);
    unsigned long long m = ((unsigned long long)h << lz) | (lz >= SH ? r << (lz - SH) : r >> (SH - lz));
    if (lz < SH && (r & ((1ull << (SH - lz)) - 1)) != 0ull) m |= 1ull;   // sticky
    const int ex = 63 - lz + SH + e;                                     // value = m 2^(ex - 63)
    const unsigned long long q = (m + 0x3ffull + ((m >> 11) & 1ull)) >> 11;
    const bool carried = m >= 0xfffffffffffffc00ull;                    // the rounding wrapped past bit 63
    if (ex >= -1022 && ex <= 1022) {
        const unsigned long long bits = ((unsigned long long)(ex + 1022) << 52) + (carried ? 1ull << 53 : q);
        return __longlong_as_double((long long)(bits | sign));           // (q's leading bit adds one to the exponent)
    }
    const double v = far_scale(carried ? 1ull << 53 : q, ex - 52);   // overflow or subnormal
    return sign ? -v : v;
}

// h 2^e as a float, rounded once to nearest (ties to even); |h| < 2^63
__device__ __forceinline__ float fixed_to_float(long long h, int e) {
    if (h == 0) return 0.f;
    const unsigned int sign = h < 0 ? 0x80000000u : 0u;
    const unsigned long long a = h < 0 ? (unsigned long long)-h : (unsigned long long)h;
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << lz;
    const int ex = 63 - lz + e;                                             // value = m 2^(ex - 63)
    // the upper 32 bits with the rest sticky, then to 24 bits
    const unsigned int u = (unsigned int)(m >> 32) | ((unsigned int)m ? 1u : 0u);
    const unsigned int q = (u >> 8) + ((u & 0x80u) && (u & 0x17fu) ? 1u : 0u);   // may carry to 2^24
    if (ex >= -126 && ex <= 126) return __uint_as_float((((unsigned int)(ex + 126) << 23) + q) | sign);
    const float v = (float)far_scale(m, ex - 63);                           // overflow or subnormal
    return sign ? -v : v;
}

// acc + v 2^k (exact), one wide multiply-add
__device__ __forceinline__ long long mad_wide(int v, int pow2, long long acc) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(v), "r"(pow2), "l"(acc));
    return d;
}

template <int NS, int EPI>
__global__ void __launch_bounds__(NTHREADS, 1) oz_gemm_kernel(const __grid_constant__ Maps maps, Params p) {
    constexpr int NG = NS, ASTAGES = Cfg<NS>::ASTAGES, B_SET = Cfg<NS>::B_SET, NBUF = Cfg<NS>::NBUF;
    constexpr int HALVES = Cfg<NS>::HALVES, NACC = NBUF * HALVES;
    constexpr uint32_t BUF_COLS = TMEM_COLS / NBUF;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *bbuf = smem;                                 // BSTAGES x NS B slices
    uint8_t *abuf = smem + BSTAGES * B_SET;                // ring of A slices
    uint64_t *fullB = (uint64_t *)(abuf + ASTAGES * A_TILE + Cfg<NS>::STAGING);
    uint64_t *emptyB = fullB + BSTAGES;
    uint64_t *fullA = emptyB + BSTAGES;
    uint64_t *emptyA = fullA + ASTAGES;
    uint64_t *tmem_full = emptyA + ASTAGES;
    uint64_t *tmem_empty = tmem_full + NACC;
    uint32_t *tmem_slot = (uint32_t *)(tmem_empty + NACC);
    int *abort_sh = (int *)(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (p.skip && *p.skip) return;   // set by earlier kernels of the stream: the same for every thread
    Tile<NS == kOzSlicesF32> w;
    if (!(NS == kOzSlicesF32 && p.tiles > 0) && p.upper_only) {   // every entry of the tile is below the diagonal
        w.at(p, 0);
        if (w.m0 >= w.n0 + BN) return;
    }

    if (threadIdx.x == 0) {
        for (int i = 0; i < BSTAGES; ++i) { mbar_init(&fullB[i], 1); mbar_init(&emptyB[i], 1); }
        for (int i = 0; i < ASTAGES; ++i) { mbar_init(&fullA[i], 1); mbar_init(&emptyA[i], 1); }
        for (int i = 0; i < NACC; ++i) { mbar_init(&tmem_full[i], 1); mbar_init(&tmem_empty[i], DRAIN); }
        *abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        // The whole warp runs the loop (waits and control flow stay
        // warp-uniform); one elected lane issues the copies.
        const bool leader = elect_one();
        int64_t ib = 0, ia = 0;
        bool ok = true;
        for (int64_t t = 0; ok && w.at(p, t); ++t)
        for (int64_t kb = w.kb0; kb < w.kb1 && ok; ++kb) {
            const int sb = (int)(ib % BSTAGES);
            if (ib >= BSTAGES) ok = warp_wait(&emptyB[sb], (uint32_t)((ib / BSTAGES - 1) & 1));
            if (ok && __any_sync(0xffffffffu, *(volatile int *)abort_sh != 0)) ok = false;
            if (!ok) break;
            if (leader) {
                mbar_expect_tx(&fullB[sb], B_SET);
                for (int q = 0; q < NS; ++q)
                    tma_load_2d(bbuf + sb * B_SET + q * B_TILE, &maps.b[q], &fullB[sb], (int)(kb * BK), (int)w.n0);
            }
            ++ib;
            for (int s = 0; s < NS && ok; ++s) {
                const int sa = (int)(ia % ASTAGES);
                if (ia >= ASTAGES) ok = warp_wait(&emptyA[sa], (uint32_t)((ia / ASTAGES - 1) & 1));
                if (!ok) break;
                if (leader) {
                    mbar_expect_tx(&fullA[sa], A_TILE);
                    tma_load_2d(abuf + sa * A_TILE, &maps.a[s], &fullA[sa], (int)(kb * BK), (int)w.m0);
                }
                ++ia;
            }
            __syncwarp();
        }
        if (!ok && leader) { atomicExch(p.err_flag, 1); *abort_sh = 1; }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // Warp-uniform loop, one elected lane issues: single-thread divergent
        // control flow around tcgen05 instructions slows their issue.
        // Fully unrolled over the slice pairs and the 4 K steps of a
        // block: descriptors are a base plus constant offsets (the 16-byte
        // unit field advances by 2 per 32-byte K step and by 512 per 8 KB B
        // slice).
        const bool leader = elect_one();
        int64_t ib = 0, ia = 0;
        bool ok = true;
        int64_t chunk0 = 0;   // chunks of the tiles before
        for (int64_t step = 0; ok && w.at(p, step); ++step) {
        const int64_t nkb = w.kb1 - w.kb0;
        for (int64_t q = 0; q < nkb && ok; ++q) {
            const int sb = (int)(ib % BSTAGES);
            ok = warp_wait(&fullB[sb], (uint32_t)((ib / BSTAGES) & 1));
            if (!ok) break;
            const uint64_t bd0 = sdesc(smem_u32(bbuf + sb * B_SET), 16, 1024);
            if (__any_sync(0xffffffffu, *(volatile int *)abort_sh != 0)) ok = false;
#pragma unroll
            for (int h = 0; h < HALVES; ++h) {
                const int len = h == 0 ? KCH : KCH_UPPER;
                const bool first = q % len == 0, last = q % len == len - 1 || q == nkb - 1;
                const int64_t chunk = chunk0 + q / len;   // (chunk0 = 0 with two halves: one tile per CTA)
                const int buf = NBUF > 1 ? (int)(chunk % NBUF) : 0;
                const uint32_t tacc = tmem + (uint32_t)buf * BUF_COLS;
                // the accumulators of this half, once the chunk before has been drained
                if (first && ok && chunk >= NBUF)
                    ok = warp_wait(&tmem_empty[buf + h], (uint32_t)((chunk / NBUF - 1) & 1));
                if (ok) tc_fence_after();
                const int s1 = h == 0 ? 4 : NS;
#pragma unroll
                for (int s = 0; s < s1; ++s) {
                    const int64_t at = ia + s;
                    const int sa = (int)(at % ASTAGES);
                    if (ok && (h == 0 || s >= 4)) ok = warp_wait(&fullA[sa], (uint32_t)((at / ASTAGES) & 1));
                    if (ok) {
                        tc_fence_after();
                        if (leader) {
                            const uint64_t ad0 = sdesc(smem_u32(abuf + sa * A_TILE), 16, 1024);
                            // groups g0 .. g0 + n - 1: one MMA over the n B slices that belong to them
                            const int t0 = h == 0 || s >= 4 ? 0 : 4 - s, n = (h == 0 ? 4 : NG) - s - t0;
#pragma unroll
                            for (int kk = 0; kk < BK / UMMA_K; ++kk) {
                                // the first MMA of a group in a chunk overwrites it
                                const uint32_t accum = (first && s == 0 && kk == 0) ? 0u : 1u;
                                umma_bf16(tacc + (uint32_t)((s + t0) * BN), ad0 + (uint64_t)(2 * kk),
                                          bd0 + (uint64_t)(512 * t0 + 2 * kk), idesc_bf16(BM, BN * n, false, false), accum);
                            }
                            if (h == HALVES - 1) umma_commit(&emptyA[sa]);
                        }
                        __syncwarp();
                    }
                }
                if (!ok) break;
                if (leader && last) umma_commit(&tmem_full[buf + h]);
            }
            if (!ok) break;
            if (leader) umma_commit(&emptyB[sb]);
            __syncwarp();
            ia += NS;
            ++ib;
        }
        chunk0 += (nkb + KCH - 1) / KCH;
        }
        if (!ok && leader) {
            atomicExch(p.err_flag, 1);
            *abort_sh = 1;
            for (int i = 0; i < NACC; ++i) umma_commit(&tmem_full[i]);   // release the epilogue once the MMAs already issued finish
        }
    } else if (warp >= 2) {
        // ---------------- drain + epilogue ----------------
        const int qtr = warp & 3;                 // TMEM lane quarter this warp may read
        const int c0 = ((warp - 2) >> 2) * ECOLS; // its columns of the 64
        constexpr int SH = 8 * (NS - 4);          // from the high unit to the low one
        constexpr int EC = 4;
        bool ok = true;
        double local = 0.0;
        int64_t chunk0 = 0;                       // chunks of the tiles before
        for (int64_t step = 0; ok && w.at(p, step); ++step) {
        const int64_t m0 = w.m0, n0 = w.n0, nchunks = (w.kb1 - w.kb0 + KCH - 1) / KCH;
        const int64_t row = m0 + 32 * qtr + lane;
        // this lane's row exponent and the exponent of column c0 + lane, both
        // read before the products are ready
        const int erow = p.ea && row < p.M ? max(p.ea[row], -1100) : p.ea_fixed;
        const int ecol = p.eb && n0 + c0 + lane < p.N ? max(p.eb[n0 + c0 + lane], -1100) : p.eb_fixed;
        // Per chunk the FP32 group sums (integers) are added to two int64
        // accumulators, groups 0-3 in base 256 (unit 2^-38 of the row x column
        // scale, |per chunk| < 2^47) and the others (unit 2^(-14 - 8 (NS - 1)),
        // < 2^49): exact, with no FP64 instruction in the drain.
        // (NS = 4: the first accumulator alone.)
        long long acch[ECOLS], accl[ECOLS];
#pragma unroll
        for (int j = 0; j < ECOLS; ++j) acch[j] = accl[j] = 0;
        // chunk c of half h from TMEM into the accumulators; false once a wait ran out
        auto drain = [&](auto half, int64_t c) -> bool {
            constexpr int h = decltype(half)::value, g0 = h == 0 ? 0 : 4, ng = h == 0 ? 4 : NG - 4;
            const int buf = NBUF > 1 ? (int)(c % NBUF) : 0;
            const bool full =
                __all_sync(0xffffffffu, mbar_wait(&tmem_full[buf + h], (uint32_t)((c / NBUF) & 1)) ? 1 : 0) != 0;
            if (!full || *(volatile int *)abort_sh) return false;
            tc_fence_after();
            // 4 columns at a time: the groups' loads are in flight together
#pragma unroll
            for (int cc = 0; cc < ECOLS; cc += 4) {
                uint32_t r[4][4];
#pragma unroll
                for (int g = 0; g < ng; ++g)
                    tmem_ld4_nowait(tmem + ((uint32_t)(32 * qtr) << 16) + (uint32_t)buf * BUF_COLS +
                                        (uint32_t)((g0 + g) * BN + c0 + cc),
                                    r[g]);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
#pragma unroll
                    for (int g = 0; g < ng; ++g) {
                        const int iv = __float2int_rn(__uint_as_float(r[g][j]));
                        if (h == 0) acch[cc + j] = mad_wide(iv, 1 << (8 * (3 - g)), acch[cc + j]);
                        else accl[cc + j] = mad_wide(iv, 1 << (8 * (NG - 5 - g)), accl[cc + j]);
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&tmem_empty[buf + h]);
            return true;
        };
        // in the order in which the issuer hands them over
        using Lower = std::integral_constant<int, 0>;
        using Upper = std::integral_constant<int, HALVES - 1>;
        if constexpr (HALVES == 1) {
            for (int64_t c = 0; c < nchunks && ok; ++c) ok = drain(Lower(), chunk0 + c);
            chunk0 += nchunks;
        } else {
            const int64_t nupper = (w.kb1 - w.kb0 + KCH_UPPER - 1) / KCH_UPPER;
            for (int64_t u = 0; u < nupper && ok; ++u) {
                if ((u & 1) || u == nupper - 1) ok = drain(Lower(), u >> 1);
                if (ok) ok = drain(Upper(), u);
            }
        }
        if (!ok) {
            atomicExch(p.err_flag, 1);
            break;
        }
        // The sums go through shared memory (for NS > 4 the pipeline's, free by
        // now: every product of this CTA has been read) so that the epilogue is
        // a short loop; unrolled over the registers its code alone, fetched once
        // per CTA, took 30 us.
        longlong2 *st = (longlong2 *)smem + (threadIdx.x - 64);
        long long *st1 = (long long *)(smem + BSTAGES * B_SET + ASTAGES * A_TILE) + (threadIdx.x - 64);
#pragma unroll
        for (int j = 0; j < ECOLS; ++j) {
            if (NS == 4) st1[j * DRAIN] = acch[j];
            else st[j * DRAIN] = make_longlong2(acch[j], accl[j]);
        }
        const bool split = EPI == EPI_STORE && p.split_stride > 0;
        const bool unit_alpha = p.alpha == 1.0;
        // four columns at a time: what the epilogue reads (C or the reference)
        // is loaded for all of them before the first is used
        const int64_t left = p.N - (n0 + c0);
#pragma unroll 1
        for (int cc = 0; cc < ECOLS && cc < left; cc += EC) {
            double old[EC];
            float oldf[EC];   // NS = 4
#pragma unroll
            for (int j = 0; j < EC; ++j) {
                const int64_t col = n0 + c0 + cc + j;
                const bool in = row < p.M && cc + j < left && !(p.upper_only && row > col);
                if (NS == 4) {
                    oldf[j] = EPI == EPI_STORE && !split && p.beta != 0.0 && in ? p.Cf[row + col * p.ldc] : 0.f;
                    continue;
                }
                old[j] = 0.0;
                if (EPI == EPI_ERR) {
                    if (in) old[j] = __ldcs(p.R + row + col * p.ldr);
                } else if (!split && p.beta != 0.0 && in) {
                    old[j] = p.C[row + col * p.ldc];
                }
            }
#pragma unroll
            for (int j = 0; j < EC; ++j) {
                const int64_t col = n0 + c0 + cc + j;
                const int ec = __shfl_sync(0xffffffffu, ecol, cc + j);
                const longlong2 v = NS == 4 ? make_longlong2(st1[(cc + j) * DRAIN], 0) : st[(cc + j) * DRAIN];
                const int ev = erow + ec - 14 - 8 * (NS - 1);
                if (NS == 4 && EPI == EPI_STORE && !split) {   // an FP32 result, in FP32
                    if (row < p.M && cc + j < left && !(p.upper_only && row > col)) {
                        float out = fixed_to_float(v.x, ev);
                        if (!unit_alpha) out *= (float)p.alpha;
                        if (p.beta != 0.0) out = fmaf((float)p.beta, oldf[j], out);
                        p.Cf[row + col * p.ldc] = out;
                    }
                    continue;
                }
                const double val = fixed_to_double<SH>(v.x, v.y, ev);
                if (row < p.M && cc + j < left && !(p.upper_only && row > col)) {
                    if (EPI == EPI_STORE) {
                        if (split) {
                            p.C[(int64_t)blockIdx.z * p.split_stride + row + col * p.M] = val;
                        } else {
                            double out = unit_alpha ? val : p.alpha * val;
                            if (p.beta != 0.0) out = fma(p.beta, old[j], out);
                            p.C[row + col * p.ldc] = out;
                        }
                    } else {
                        const double d = fma(-p.alpha, val, old[j]);
                        local = fma(d, d, local);
                    }
                }
            }
        }
        }
        if (EPI == EPI_ERR) {
            local = warp_sum(local);
            __shared__ double red[DRAIN / 32];
            if (lane == 0) red[warp - 2] = local;
            asm volatile("bar.sync 1, %0;" ::"n"(DRAIN) : "memory");
            if (warp == 2 && lane == 0) {
                double t = 0.0;
                for (int i = 0; i < DRAIN / 32; ++i) t += red[i];
                p.errp[blockIdx.x + (int64_t)blockIdx.y * gridDim.x] = t;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Triangular operands (the SIMT kernel's a_upper / b_upper): with tri == 1
// op(A) is upper triangular, X(r, k) = op(A)(r, k) is zero for r > k; with
// tri == 2 op(B) is, and X(r, k) = op(B)(k, r) is zero for k > r.  Those
// entries are never read.
__device__ __forceinline__ bool tri_zero(int tri, int64_t r, int64_t k) {
    return (tri == 1 && r > k) || (tri == 2 && k > r);
}

// |x| as its bit pattern (orders like the value for non-negative numbers);
// non-finite entries count as zero (the contraction expects finite data).
// FP32 data stays on the integer units: a conversion to FP64 costs a warp as
// much as an FP64 operation.
__device__ __forceinline__ unsigned int abs_bits(float x) {
    const unsigned int a = __float_as_uint(x) & 0x7fffffffu;
    return (a >> 23) == 0xff ? 0u : a;
}
__device__ __forceinline__ int exp_of_bits(unsigned int a) {
    const int E = (int)(a >> 23);
    return E > 0 ? E - 126 : -117 - __clz(a);   // subnormal: a 2^-149 < 2^(32 - clz - 149)
}
template <typename TX> struct AbsKey { using type = unsigned long long; };
template <> struct AbsKey<float> { using type = unsigned int; };
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    const unsigned long long a = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    return (a >> 52) == 0x7ff ? 0ull : a;
}

// frexp exponent of the double with bit pattern a > 0 (a < 2^e)
__device__ __forceinline__ int exp_of_bits(unsigned long long a) {
    const int E = (int)(a >> 52);
    if (E > 0) return E - 1022;
    int ex;
    frexp(__longlong_as_double((long long)a), &ex);   // subnormal
    return ex;
}

constexpr int kExpZero = -2000000000;   // exponent of an all-zero row (< -1100)
constexpr int kMaxExpSplit = 16;        // K ranges of the row-exponent pass

// ep[z][r] = exponent of max |X(r, k)| over the z-th K range (frexp
// convention: max < 2^e), kExpZero if that range of the row is zero; blocks
// cover 32 rows x one K range, so every entry is written once (no atomics,
// no initialisation pass).  Integer compares of the bit patterns: no FP64
// arithmetic.
template <typename TX>
__global__ void rowexp_kernel(const TX *__restrict__ X, int64_t R, int64_t K, int64_t sr, int64_t sk,
                              int64_t kper, int tri, int *ep) {
    int *e = ep + (int64_t)blockIdx.y * R;
    using Key = typename AbsKey<TX>::type;
    __shared__ Key red[8][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;      // 32 x 8
    const int64_t r0 = (int64_t)blockIdx.x * 32;
    const int64_t kb = (int64_t)blockIdx.y * kper;
    int64_t ke = kb + kper;
    if (ke > K) ke = K;
    if (sk == 1) {
        // K contiguous: lanes along k, warps over rows
        for (int rr = ty; rr < 32; rr += 8) {
            const int64_t r = r0 + rr;
            Key m = 0;
            if (r < R)
                for (int64_t k = kb + tx; k < ke; k += 32)
                    if (!tri_zero(tri, r, k)) m = max(m, abs_bits(X[r * sr + k]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (tx == 0 && r < R) e[r] = m > 0 ? exp_of_bits(m) : kExpZero;
        }
        return;
    }
    // rows contiguous: lanes along rows, warps split the K range
    const int64_t r = r0 + tx;
    Key mx = 0;
    if (r < R)
        for (int64_t k = kb + ty; k < ke; k += 8)
            if (!tri_zero(tri, r, k)) mx = max(mx, abs_bits(X[r + k * sk]));
    red[ty][tx] = mx;
    __syncthreads();
    if (ty == 0 && r < R) {
        Key m = red[0][tx];
#pragma unroll
        for (int i = 1; i < 8; ++i) m = max(m, red[i][tx]);
        e[r] = m > 0 ? exp_of_bits(m) : kExpZero;
    }
}

// v (below 2^(8 NS - 1)) in NS balanced base-256 digits
template <int NS>
__device__ __forceinline__ void cut(unsigned long long v, bool neg, __nv_bfloat16 q[NS]) {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const int w = 8 * (NS - 1 - s);
        int d;                           // balanced digit, |d| <= 128; carries in two's complement
        if (s == 0) d = (int)((v + (1ull << (w - 1))) >> w);
        else if (w > 0) d = (int)((long long)(v + (1ull << (w - 1))) >> w);
        else d = (int)(long long)v;
        v -= (unsigned long long)(long long)d << w;
        q[s] = __float2bfloat16_rn((float)(neg ? -d : d));
    }
}

// The NS BF16 digits of x 2^-er (|x| < 2^er) in q: v = round(|x| 2^(8 NS - 1 - er))
// in balanced base-256 digits, integer arithmetic on the bit pattern.
template <int NS>
__device__ __forceinline__ void digits(double x, int er, __nv_bfloat16 q[NS], bool &nonfinite) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    int E = (int)((bits >> 52) & 0x7ff);
    unsigned long long M = bits & 0xfffffffffffffull;
    if (E == 0x7ff) {                    // non-finite: not representable, taken as zero
        M = 0;
        nonfinite = true;
    } else if (E == 0) E = 1;            // subnormal: M 2^(1 - 1075)
    else M |= 1ull << 52;                // |x| = M 2^(E - 1075)
    unsigned long long v = 0;
    const int sh = E - 1075 + 8 * NS - 1 - er;   // v = M 2^sh; sh <= 8 NS - 54 since |x| < 2^er
    if (er >= -1100 && M != 0) {
        if (sh >= 0) v = M << sh;
        else if (sh > -63) v = (M >> (-sh)) + ((M >> (-sh - 1)) & 1ull);
    }
    cut<NS>(v, (bits >> 63) != 0, q);
}
template <int NS>
__device__ __forceinline__ void digits(float x, int er, __nv_bfloat16 q[NS], bool &nonfinite) {
    const unsigned int bits = __float_as_uint(x);
    int E = (int)((bits >> 23) & 0xff);
    unsigned int M = bits & 0x7fffffu;
    if (E == 0xff) {
        M = 0;
        nonfinite = true;
    } else if (E == 0) E = 1;            // |x| = M 2^(E - 150)
    else M |= 1u << 23;
    unsigned long long v = 0;
    const int sh = E - 150 + 8 * NS - 1 - er;    // sh <= 8 NS - 25
    if (er >= -1100 && M != 0) {
        if (sh >= 0) v = (unsigned long long)M << sh;
        else if (sh > -31) v = (M >> (-sh)) + ((M >> (-sh - 1)) & 1u);
    }
    cut<NS>(v, (bits >> 31) != 0, q);
}

// out[s][r * ldk + k] = slice s of X(r, k) 2^-e[r], tiles of 32 rows x 64 k
// through shared memory so reads follow X's contiguous axis and writes follow
// k (two neighbouring k per lane, one 4-byte store per slice).
// The row exponents come from the nsplit partial ones of rowexp_kernel (the
// blocks of the first K column also store them in e_out for the product), or
// every row takes fixed_e when ep is null.  The tiles are numbered along
// grid.x, k first: rows or k alone may need more than the 65535 blocks that the
// other grid dimensions hold (2.1 million rows, 4.2 million k).
template <typename TX, int NS>
__global__ void __launch_bounds__(256) slice_kernel(const TX *__restrict__ X, int64_t R, int64_t K, int64_t sr, int64_t sk,
                             int tri, const int *__restrict__ ep, int nsplit, int *__restrict__ e_out, int fixed_e,
                             __nv_bfloat16 *__restrict__ out, int64_t ldk, int64_t slice_stride, int *nonfinite) {
    __shared__ TX tile[32][65];
    __shared__ int erow[32];
    const unsigned kt = (unsigned)((K + 63) / 64);
    const int64_t r0 = (int64_t)(blockIdx.x / kt) * 32, k0 = (int64_t)(blockIdx.x % kt) * 64;
    const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
    if (ty == 0) {
        const int64_t r = r0 + tx;
        int er = fixed_e;
        if (ep && r < R) {
            er = kExpZero;
            for (int z = 0; z < nsplit; ++z) er = max(er, ep[(int64_t)z * R + r]);
            if (k0 == 0 && e_out) e_out[r] = er;
        }
        erow[tx] = er;
    }
    if (sk == 1) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = ty + 8 * (u >> 1), kk = tx + 32 * (u & 1);
            const int64_t r = r0 + i, k = k0 + kk;
            tile[i][kk] = (r < R && k < K && !tri_zero(tri, r, k)) ? X[r * sr + k] : TX(0);
        }
    } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int kk = ty + 8 * u;
            const int64_t r = r0 + tx, k = k0 + kk;
            tile[tx][kk] = (r < R && k < K && !tri_zero(tri, r, k)) ? X[r * sr + k * sk] : TX(0);
        }
    }
    __syncthreads();
    bool bad = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int i = ty + 8 * u;
        const int64_t r = r0 + i, k = k0 + 2 * tx;
        if (r >= R || k >= K) continue;
        __nv_bfloat16 a[NS], b[NS];
        digits<NS>(tile[i][2 * tx], erow[i], a, bad);
        digits<NS>(tile[i][2 * tx + 1], erow[i], b, bad);
        __nv_bfloat16 *o = out + r * ldk + k;
        if (k + 1 < K && (((uintptr_t)o | (uintptr_t)(slice_stride * 2)) & 3) == 0) {
#pragma unroll
            for (int s = 0; s < NS; ++s) *(__nv_bfloat162 *)(o + s * slice_stride) = __nv_bfloat162(a[s], b[s]);
        } else {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                o[s * slice_stride] = a[s];
                if (k + 1 < K) o[s * slice_stride + 1] = b[s];
            }
        }
    }
    if (bad && nonfinite) *nonfinite = 1;
}

// Rows with K contiguous (sk == 1) and their own exponents, one CTA per row:
// the row maximum (as in rowexp_kernel) and then the slices (as in
// slice_kernel), in one launch.  A thread takes pairs of neighbouring k; the
// first RU pairs stay in registers between the two, the rest are read again.
template <typename TX, int NS>
__global__ void __launch_bounds__(256) slice_rows_kernel(const TX *__restrict__ X, int64_t K, int64_t sr,
                                                         int tri, int *__restrict__ e_out,
                                                         __nv_bfloat16 *__restrict__ out, int64_t ldk,
                                                         int64_t slice_stride, int *nonfinite) {
    constexpr int RU = 4;
    using Key = typename AbsKey<TX>::type;
    __shared__ Key red[8];
    __shared__ int er_sh;
    const int64_t r = blockIdx.x;
    const TX *x = X + r * sr;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t k0 = 2 * tid;
    auto load = [&](int64_t k) -> TX { return k < K && !tri_zero(tri, r, k) ? x[k] : TX(0); };
    TX va[RU], vb[RU];
#pragma unroll
    for (int u = 0; u < RU; ++u) {
        va[u] = load(k0 + 512 * u);
        vb[u] = load(k0 + 512 * u + 1);
    }
    Key m = 0;
#pragma unroll
    for (int u = 0; u < RU; ++u) m = max(m, max(abs_bits(va[u]), abs_bits(vb[u])));
    for (int64_t k = k0 + 512 * RU; k < K; k += 512) m = max(m, max(abs_bits(load(k)), abs_bits(load(k + 1))));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red[warp] = m;
    __syncthreads();
    if (tid == 0) {
        Key t = red[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) t = max(t, red[i]);
        const int er = t > 0 ? exp_of_bits(t) : kExpZero;
        er_sh = er;
        e_out[r] = er;
    }
    __syncthreads();
    const int er = er_sh;
    __nv_bfloat16 *row = out + r * ldk;
    const bool pairs = (((uintptr_t)row | (uintptr_t)(slice_stride * 2)) & 3) == 0;
    bool bad = false;
    auto store = [&](int64_t k, TX p, TX q) {
        __nv_bfloat16 a[NS], b[NS];
        digits<NS>(p, er, a, bad);
        digits<NS>(q, er, b, bad);
        __nv_bfloat16 *o = row + k;
        if (pairs && k + 1 < K) {
#pragma unroll
            for (int s = 0; s < NS; ++s) *(__nv_bfloat162 *)(o + s * slice_stride) = __nv_bfloat162(a[s], b[s]);
        } else {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                o[s * slice_stride] = a[s];
                if (k + 1 < K) o[s * slice_stride + 1] = b[s];
            }
        }
    };
#pragma unroll
    for (int u = 0; u < RU; ++u)
        if (k0 + 512 * u < K) store(k0 + 512 * u, va[u], vb[u]);
    for (int64_t k = k0 + 512 * RU; k < K; k += 512) store(k, load(k), load(k + 1));
    if (bad && nonfinite) *nonfinite = 1;
}

template <typename TC>
__global__ void split_sum_kernel(const double *__restrict__ part, int S, int64_t M, int64_t N, double alpha,
                                 double beta, TC *C, int64_t ldc, int upper_only) {
    const int64_t total = M * N;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e % M, j = e / M;
        if (upper_only && i > j) continue;
        double sum = 0.0;
        for (int z = 0; z < S; ++z) sum += part[(int64_t)z * total + e];
        double out = alpha * sum;
        if (beta != 0.0) out = fma(beta, (double)C[i + j * ldc], out);
        C[i + j * ldc] = (TC)out;
    }
}

// The emulation's own buffers: without room for them the caller takes the FMA
// kernels (nothing has been written to C by then).
cudaError_t room(void **p, size_t bytes, cudaStream_t s) {
    return fail_this_alloc() ? cudaErrorMemoryAllocation : lib_malloc_async(p, bytes, s);
}

struct Slices {
    __nv_bfloat16 *q = nullptr;
    int *e = nullptr;
    int64_t R = 0, ldk = 0;
};

template <int NS, typename TX>
cudaError_t slice_into(const TX *X, int64_t R, int64_t K, int64_t sr, int64_t sk, __nv_bfloat16 *q, int *e,
                       int fixed_e, int64_t ldk, int64_t slice_stride, cudaStream_t s, int tri = 0,
                       int *nonfinite = nullptr) {
    if (R <= 0 || K <= 0) return cudaSuccess;
    ProfScope prof(PROF_OZ_SLICE, 0.0, (double)sizeof(TX) * R * K + 2.0 * NS * (double)R * K, s);
    if (e && sk == 1 && (R >= kNumSMs || K <= 8192)) {
        count_launch();
        slice_rows_kernel<TX, NS><<<(unsigned)R, 256, 0, s>>>(X, K, sr, tri, e, q, ldk, slice_stride, nonfinite);
        return cudaGetLastError();
    }
    int *ep = nullptr;
    int64_t ksplit = 1;
    if (e) {
        const int64_t rblocks = (R + 31) / 32;
        ksplit = (4 * kNumSMs + rblocks - 1) / rblocks;
        const int64_t kmax = (K + 255) / 256;
        if (ksplit > kmax) ksplit = kmax;
        if (ksplit > kMaxExpSplit) ksplit = kMaxExpSplit;
        if (ksplit < 1) ksplit = 1;
        const int64_t kper = (K + ksplit - 1) / ksplit;
        ksplit = (K + kper - 1) / kper;
        ep = e;   // one range: the partial exponents are the exponents
        if (ksplit > 1) EOD_CUDA_TRY(room((void **)&ep, sizeof(int) * (size_t)ksplit * R, s));
        count_launch();
        rowexp_kernel<<<dim3((unsigned)rblocks, (unsigned)ksplit), 256, 0, s>>>(X, R, K, sr, sk, kper, tri, ep);
        cudaError_t le = cudaGetLastError();
        if (le != cudaSuccess) {
            if (ep != e) cudaFreeAsync(ep, s);
            return le;
        }
    }
    count_launch();
    const int64_t tiles = ((K + 63) / 64) * ((R + 31) / 32);
    slice_kernel<TX, NS><<<(unsigned)tiles, dim3(32, 8), 0, s>>>(X, R, K, sr, sk, tri, ep, (int)ksplit,
                                                       (ep && ep != e) ? e : nullptr, fixed_e, q, ldk, slice_stride,
                                                       nonfinite);
    cudaError_t le = cudaGetLastError();
    if (ep && ep != e) cudaFreeAsync(ep, s);
    return le;
}

template <int NS, typename TX>
cudaError_t make_slices(const TX *X, int64_t R, int64_t K, int64_t sr, int64_t sk, Slices &sl, cudaStream_t s,
                        int tri = 0, int *nonfinite = nullptr) {
    sl.R = R;
    sl.ldk = round_up(K, 8);
    EOD_CUDA_TRY(room((void **)&sl.q, sizeof(__nv_bfloat16) * (size_t)NS * R * sl.ldk, s));
    EOD_CUDA_TRY(room((void **)&sl.e, sizeof(int) * (size_t)R, s));
    return slice_into<NS>(X, R, K, sr, sk, sl.q, sl.e, 0, sl.ldk, R * sl.ldk, s, tri, nonfinite);
}

void free_slices(Slices &sl, cudaStream_t s) {
    if (sl.q) cudaFreeAsync(sl.q, s);
    if (sl.e) cudaFreeAsync(sl.e, s);
    sl.q = nullptr;
    sl.e = nullptr;
}

}  // namespace oz

// Slices of op(X) as `rows` x K with K contiguous (see oz_gemm.cu header).
cudaError_t oz_slice(const double *X, int64_t rows, int64_t K, int64_t sr, int64_t sk, void *q, int *e,
                     int fixed_e, int64_t ldk, int64_t slice_stride, cudaStream_t s) {
    return oz::slice_into<kOzSlices>(X, rows, K, sr, sk, (__nv_bfloat16 *)q, e, fixed_e, ldk, slice_stride, s);
}

namespace oz {
template <int NS>
cudaError_t run_ops(const OzOperand &A, const OzOperand &B, int64_t M, int64_t N, int64_t K, double alpha, double beta,
                    double *C, int64_t ldc, const GemmExtra &x, int *err_flag, cudaStream_t s, float *Cf) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if ((NS == kOzSlicesF32) != (Cf != nullptr) || (NS != kOzSlices && x.epilogue != EPI_STORE)) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    Maps maps;
    std::memset(&maps, 0, sizeof(maps));
    for (int i = 0; i < NS; ++i) {
        const __nv_bfloat16 *qa = (const __nv_bfloat16 *)A.q, *qb = (const __nv_bfloat16 *)B.q;
        if (!make_map(&maps.a[i], qa + (size_t)i * A.slice_stride, K, M, A.ldk, BK, BM) ||
            !make_map(&maps.b[i], qb + (size_t)i * B.slice_stride, K, N, B.ldk, BK, BN))
            return cudaErrorInvalidValue;
    }
    // exponents: a fixed exponent is passed as a one-entry array by the caller
    Params p;
    std::memset(&p, 0, sizeof(p));
    p.M = M;
    p.N = N;
    p.kblocks = (K + BK - 1) / BK;
    p.ea = A.e;
    p.eb = B.e;
    p.alpha = alpha;
    p.beta = beta;
    p.err_flag = err_flag;
    p.skip = x.skip;
    p.R = (const double *)x.ref;
    p.ldr = x.ldref;
    p.errp = x.err_partials;
    p.ea_fixed = A.e_fixed;
    p.eb_fixed = B.e_fixed;
    p.upper_only = x.upper_only ? 1 : 0;
    p.a_tri = x.a_upper ? 1 : 0;
    p.b_tri = x.b_upper ? 1 : 0;
    const int64_t tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
    // K split until the grid covers the SMs, at least two K blocks per split
    // (a split's exact chunks start at its own first block)
    int64_t splits = 1;
    if (x.epilogue == EPI_STORE && tiles < kNumSMs) {
        splits = (kNumSMs + tiles - 1) / tiles;
        const int64_t smax = p.kblocks / 2;
        if (splits > smax) splits = smax;
        if (splits < 1) splits = 1;
    }
    p.kb_per_split = (p.kblocks + splits - 1) / splits;
    if (p.kb_per_split < 1) p.kb_per_split = 1;
    splits = (p.kblocks + p.kb_per_split - 1) / p.kb_per_split;
    if (splits < 1) splits = 1;
    double *part = nullptr;
    constexpr int SMEM = Cfg<NS>::SMEM;
    e = set_smem_once(oz_gemm_kernel<NS, EPI_STORE>, SMEM);
    if constexpr (NS == kOzSlices)
        if (e == cudaSuccess) e = set_smem_once(oz_gemm_kernel<NS, EPI_ERR>, SMEM);
    if (e == cudaSuccess && splits > 1) {
        e = room((void **)&part, sizeof(double) * (size_t)splits * M * N, s);
        p.C = part;
        p.ldc = M;
        p.split_stride = M * N;
    } else {
        p.C = C;
        p.Cf = Cf;
        p.ldc = ldc;
        p.split_stride = 0;
    }
    // the method's flops: an upper-only output or a triangular operand halves
    // the multiply-adds (both triangular: a sixth), as the kernel skips them
    double frac = 1.0;
    if (x.upper_only) frac *= 0.5;
    if (x.a_upper && x.b_upper) frac /= 6.0;
    else if (x.a_upper || x.b_upper) frac *= 0.5;
    ProfScope prof(PROF_OZ_GEMM, 2.0 * M * N * K * frac,
                   2.0 * NS * ((double)M * K + (double)K * N) + 8.0 * 2 * M * N, s);
    if (e == cudaSuccess) {
        dim3 grid((unsigned)((M + BM - 1) / BM), (unsigned)((N + BN - 1) / BN), (unsigned)splits);
        p.gm = grid.x;
        if (NS == kOzSlicesF32 && splits == 1 && tiles > kNumSMs) {
            p.tiles = tiles;
            grid = dim3(kNumSMs);
        }
        count_launch();
        if constexpr (NS != kOzSlices) {
            oz_gemm_kernel<NS, EPI_STORE><<<grid, NTHREADS, SMEM, s>>>(maps, p);
        } else {
            if (x.epilogue == EPI_ERR) oz_gemm_kernel<NS, EPI_ERR><<<grid, NTHREADS, SMEM, s>>>(maps, p);
            else oz_gemm_kernel<NS, EPI_STORE><<<grid, NTHREADS, SMEM, s>>>(maps, p);
        }
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && splits > 1) {
        count_launch();
        const int blocks = (int)std::min<int64_t>((M * N + 255) / 256, 4LL * kNumSMs * 8);
        if (Cf) split_sum_kernel<float><<<blocks, 256, 0, s>>>(part, (int)splits, M, N, alpha, beta, Cf, ldc,
                                                                 p.upper_only);
        else split_sum_kernel<double><<<blocks, 256, 0, s>>>(part, (int)splits, M, N, alpha, beta, C, ldc,
                                                              p.upper_only);
        e = cudaGetLastError();
    }
    if (part) cudaFreeAsync(part, s);
    return e;
}
}  // namespace oz

cudaError_t oz_gemm_ops(const OzOperand &A, const OzOperand &B, int64_t M, int64_t N, int64_t K, double alpha,
                        double beta, double *C, int64_t ldc, const GemmExtra &x, int *err_flag, cudaStream_t s) {
    return oz::run_ops<kOzSlices>(A, B, M, N, K, alpha, beta, C, ldc, x, err_flag, s, nullptr);
}

namespace oz {
template <int NS, typename T>
cudaError_t gemm_any(bool ta, bool tb, int64_t M, int64_t N, int64_t K, double alpha, const T *A, int64_t lda,
                     const T *B, int64_t ldb, double beta, double *C, float *Cf, int64_t ldc, const GemmExtra &x,
                     int *err_flag, cudaStream_t s) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    Slices sa, sb;
    // op(A)(i, k): rows i, reduction k; op(B)(k, j) seen as rows j
    // a_upper / b_upper: op(A) / op(B) is upper triangular and its zero part
    // is not read, as in the SIMT kernel
    cudaError_t e = make_slices<NS>(A, M, K, ta ? lda : 1, ta ? 1 : lda, sa, s, x.a_upper ? 1 : 0);
    const bool same = (A == B) && (ta != tb) && (lda == ldb) && (M == N) && !x.a_upper && !x.b_upper;
    if (e == cudaSuccess && !same) e = make_slices<NS>(B, N, K, tb ? 1 : ldb, tb ? ldb : 1, sb, s, x.b_upper ? 2 : 0);
    const Slices &SB = same ? sa : sb;
    if (e == cudaSuccess) {
        OzOperand oa{sa.q, sa.e, 0, sa.ldk, (int64_t)M * sa.ldk};
        OzOperand ob{SB.q, SB.e, 0, SB.ldk, (int64_t)N * SB.ldk};
        e = run_ops<NS>(oa, ob, M, N, K, alpha, beta, C, ldc, x, err_flag, s, Cf);
    }
    free_slices(sa, s);
    if (!same) free_slices(sb, s);
    return e;
}
}  // namespace oz

// C = alpha op(A) op(B) + beta C (EPI_STORE) or the squared error against
// x.ref (EPI_ERR), FP64, through the sliced tensor-core product.
cudaError_t oz_gemm(bool ta, bool tb, int64_t M, int64_t N, int64_t K, double alpha, const double *A, int64_t lda,
                    const double *B, int64_t ldb, double beta, double *C, int64_t ldc, const GemmExtra &x,
                    int *err_flag, cudaStream_t s) {
    return oz::gemm_any<kOzSlices, double>(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, nullptr, ldc, x, err_flag, s);
}

// The same product of FP32 data (exact in FP64, so sliced the same way) with
// an FP32 result: C = alpha op(A) op(B) + beta C rounded once to FP32.
cudaError_t oz_gemm_f32(bool ta, bool tb, int64_t M, int64_t N, int64_t K, double alpha, const float *A, int64_t lda,
                        const float *B, int64_t ldb, double beta, float *C, int64_t ldc, const GemmExtra &x,
                        int *err_flag, cudaStream_t s) {
    if (x.epilogue != EPI_STORE) return cudaErrorInvalidValue;
    return oz::gemm_any<kOzSlicesF32, float>(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, nullptr, C, ldc, x, err_flag, s);
}

namespace oz {

// What the check of oz_decode takes of the sliced operands W (R_w rows, then V's),
// one warp per row: the entries' magnitudes in BF16, rounded towards zero from
// |256 q_0 + q_1| - 1 <= 2^15 |x| / 2^e, and the row's part of what each entry of
// A_hat needs (oz_decode): rows of W scale (1, 2^(eu + E - e)), eu the exponent
// of U's row, E the largest of D's nd columns' ed; rows of V (1, sum over l of
// 2^(ed_l - E) |x_l| / 2^e).  With nd = 0 (W given) the second part is zero.  A
// row of zeros needs nothing, unless W's came out of a U that is not zero: then
// no entry is vouched for.  (Reads and writes 6 bytes an entry; 2 x 8192 rows of
// 455: 15 us.)
__global__ void __launch_bounds__(256) cover_rows_kernel(const __nv_bfloat16 *__restrict__ qw,
                                                         const __nv_bfloat16 *__restrict__ qv, int64_t R_w, int64_t R,
                                                         int64_t K, int64_t ldk, const int *__restrict__ ew,
                                                         const int *__restrict__ ev, const int *__restrict__ eu,
                                                         const int *__restrict__ ed, int64_t nd, float scale,
                                                         __nv_bfloat16 *__restrict__ mag, float2 *__restrict__ need) {
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= R) return;
    const bool of_w = row < R_w;
    const int64_t at = of_w ? row : row - R_w;
    const __nv_bfloat16 *q = (of_w ? qw : qv) + at * ldk;
    const int64_t stride = (of_w ? R_w : R - R_w) * ldk;
    int E = kExpZero;
    for (int64_t l = lane; l < nd; l += 32) E = max(E, ed[l]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
    float sum = 0.f;
    for (int64_t k = 8 * lane; k < K; k += 256) {   // (ldk is a multiple of 8; what lies beyond K is not used)
        union Eight {
            uint4 v;
            __nv_bfloat16 x[8];
        } a, b, m;
        a.v = *(const uint4 *)(q + k);
        b.v = *(const uint4 *)(q + stride + k);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float h = fabsf(fmaf(256.f, __bfloat162float(a.x[j]), __bfloat162float(b.x[j])));
            m.x[j] = __float2bfloat16_rz(fmaxf(h - 1.f, 0.f));
            if (nd && !of_w && k + j < K) sum = fmaf(h + 1.f, exp2f((float)max(ed[k + j] - E, -200)), sum);
        }
        *(uint4 *)(mag + row * ldk + k) = m.v;
    }
    sum = warp_sum(sum);
    if (lane) return;
    float2 n = make_float2(of_w ? scale : 1.f, 0.f);
    const int er = of_w ? ew[at] : ev[at], er_u = of_w && nd ? eu[at] : kExpZero;
    if (er == kExpZero) n.x = er_u != kExpZero ? __int_as_float(0x7f800000) : 0.f;
    else if (nd) n.y = !of_w ? ldexpf(sum, -15) : er_u == kExpZero ? 0.f : scale * exp2f((float)max(er_u + E - er, -126));
    need[row] = n;
}

// The rounding of the digits, and the pairs left out (s + t >= NS), take at
// most (NS + 1.1) 2^(-8 NS) of the row x column scales per term.
template <int NS> constexpr double kTermLoss = NS == 8 ? 9.1 / 18446744073709551616.0 : 5.1 / 4294967296.0;

// A_hat = W V^T through the emulation, W = U D as well if U is given, but only
// if no entry loses anything against FMAs.  Those guarantee 2 r u S(i, j) (and
// the result's rounding), S = |W| |V|^T; the digits, with a = eta r, eta =
// kTermLoss, e the row exponents and e_U, e_D those of U's rows and D's
// columns,
//   a 2^(e_W(i) + e_V(j))  +  a 2^e_U(i) sum over l of 2^e_D(l) |V(j, l)|,
// the second for W's own error.  So S(i, j) has to be eta / 2u times the sum of
// the two powers: 1/450 of it in FP64, 1/100 in FP32.  S is bounded from below by a
// product of the magnitudes' first eight bits on the tensor cores, compared in
// its epilogue (both kernels: 28 of 415 us in FP64 at 2048 x 2048 x 600, 100 of
// 884 in FP32 at 8192 x 8192 x 455); where any entry falls short, flags[1] is
// set and the large product is not run.
// Dense factors pass (the least entry of 3000 x 3000 by a factor of 5 with D's
// diagonal falling as 1/l, of 66 with the FP64 form's test factors); rows of V
// with zeros against W's large entries do not, nor all of a diagonal that falls
// as fast as 1/l^2.
template <typename T>
cudaError_t decode(const T *U, const T *D, T *W, const T *V, int64_t m, int64_t n, int64_t r, T *A_hat, int64_t ld,
                   int *flags, cudaStream_t s) {
    constexpr bool f64 = std::is_same<T, double>::value;
    constexpr int NS = f64 ? kOzSlicesFine : kOzSlicesF32;
    Slices su, sd, sw, sv;
    __nv_bfloat16 *mag = nullptr;
    float2 *need = nullptr;
    GemmExtra x;
    cudaError_t e = cudaSuccess;
    if (U) {
        if constexpr (f64) {
            e = make_slices<NS>(U, m, r, 1, m, su, s, 0, flags + 1);
            if (e == cudaSuccess) e = make_slices<NS>(D, r, r, r, 1, sd, s, 2, flags + 1);
            if (e == cudaSuccess) {
                const OzOperand ou{su.q, su.e, 0, su.ldk, m * su.ldk}, od{sd.q, sd.e, 0, sd.ldk, r * sd.ldk};
                x.b_upper = true;
                e = run_ops<NS>(ou, od, m, r, r, 1.0, 0.0, W, m, x, flags, s, nullptr);
                x.b_upper = false;
            }
        } else {
            e = cudaErrorInvalidValue;
        }
    }
    if (e == cudaSuccess) e = make_slices<NS>(W, m, r, 1, m, sw, s, 0, flags + 1);
    if (e == cudaSuccess) e = make_slices<NS>(V, n, r, 1, n, sv, s, 0, flags + 1);
    if (e == cudaSuccess) e = room((void **)&mag, sizeof(__nv_bfloat16) * (size_t)((m + n) * sw.ldk), s);
    if (e == cudaSuccess) e = room((void **)&need, sizeof(float2) * (size_t)(m + n), s);
    if (e == cudaSuccess) {
        ProfScope prof(PROF_STREAM, 0.0, 6.0 * (m + n) * r, s);
        count_launch();
        const double u = f64 ? 1.0 / 9007199254740992.0 : 1.0 / 16777216.0;
        // S in units of 2^-30 of the scales; a fifth more for the FP32 sums
        const float scale = (float)(1.2 * 1073741824.0 * kTermLoss<NS> / (2.0 * u));
        cover_rows_kernel<<<(unsigned)((m + n + 7) / 8), 256, 0, s>>>(sw.q, sv.q, m, m + n, r, sw.ldk, sw.e, sv.e, su.e, sd.e,
                                                                      U ? r : 0, scale, mag, need);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        TcGemmDesc g;
        g.M = m;
        g.N = n;
        g.K = r;
        g.a[0] = {mag, r, m, sw.ldk};
        g.b[0] = {mag + m * sw.ldk, r, n, sv.ldk};
        g.epilogue = EPI_COVER;
        g.row_need = need;
        g.col_need = need + m;
        g.low = flags + 1;
        g.err_flag = flags;
        e = tc_gemm_run(g, nullptr, s);
    }
    if (e == cudaSuccess) {
        const OzOperand ow{sw.q, sw.e, 0, sw.ldk, m * sw.ldk}, ov{sv.q, sv.e, 0, sv.ldk, n * sv.ldk};
        x.skip = flags + 1;
        if constexpr (f64) e = run_ops<NS>(ow, ov, m, n, r, 1.0, 0.0, A_hat, ld, x, flags, s, nullptr);
        else e = run_ops<NS>(ow, ov, m, n, r, 1.0, 0.0, nullptr, ld, x, flags, s, A_hat);
    }
    free_slices(su, s);
    free_slices(sd, s);
    free_slices(sw, s);
    free_slices(sv, s);
    if (mag) cudaFreeAsync(mag, s);
    if (need) cudaFreeAsync(need, s);
    return e;
}
}  // namespace oz

template <typename T>
cudaError_t oz_decode(const T *U, const T *D, T *W, const T *V, int64_t m, int64_t n, int64_t r, T *A_hat, int64_t ld,
                      int *flags, cudaStream_t s) {
    return oz::decode<T>(U, D, W, V, m, n, r, A_hat, ld, flags, s);
}
template cudaError_t oz_decode<double>(const double *, const double *, double *, const double *, int64_t, int64_t, int64_t,
                                       double *, int64_t, int *, cudaStream_t);
template cudaError_t oz_decode<float>(const float *, const float *, float *, const float *, int64_t, int64_t, int64_t,
                                      float *, int64_t, int *, cudaStream_t);

int64_t oz_gemm_err_ctas(int64_t M, int64_t N) { return ((M + oz::BM - 1) / oz::BM) * ((N + oz::BN - 1) / oz::BN); }

}  // namespace eod
