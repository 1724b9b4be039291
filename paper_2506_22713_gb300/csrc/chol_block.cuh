// The leaf factorisation of chol_leaf.cuh (G + shift I = R^T R of a w x w
// Gram, w <= 128, with the rank test of Alg. 1 steps 6-11 and R^{-1}) in
// blocks of columns over a cluster of CTAs.
//
// What bounds it: FP64 issue.  A warp-wide DFMA occupies its sub-partition
// for 64 cycles, whatever the number of active lanes (71 for a dependent
// one, 76 with all four sub-partitions busy; probe), so the time is the
// number of FP64 instructions on the path from pivot to pivot times 64.
//   - One warp factors 8 columns in registers (diag8): its 28 off-diagonal
//     and 4 of its diagonal entries are one register, so a column costs
//     seven FP64 instructions (three of the reciprocal, the next pivot
//     straight from it as d' = s - u^2 r, one multiplier, one update).
//     It runs alone on its sub-partition.
//   - 32 columns are four of these; between them only the panel X and the
//     next 8 x 8 block are on the path, the rest of the update and the block's
//     inverse run on the other sub-partitions' warps meanwhile.  Every CTA of
//     the cluster does this on the same bits, so that the pivots, the
//     decisions and the block's inverse need no exchange.
//   - The remaining w^3 / 3 multiply-adds are products of 32 columns, spread
//     over the SMs: a CTA owns every C-th row of the trailing matrix and
//     every C-th column of L^{-1}; per block the panel X = S L_bb^{-T} and the
//     next diagonal block are pushed to every CTA through distributed shared
//     memory, one cluster barrier (about 480 cycles) each; what the next
//     block does not need at once runs beside its factorisation.
//   - Inside a block the entries are dealt to the lanes one by one, whatever
//     their row: with a row to a warp most lanes idled, and the FP64 issue
//     slots of the idle ones held up the 8-column chain (5400 cycles alone,
//     7800 beside them, and as long again waiting for them).  A leaf of 64, 96,
//     128 columns: 57, 86, 126 us before, 42, 68, 103 now.  Half of what is left
//     is the 8-column chain.
// Every CTA takes every decision on identical bits, so the barriers match.
#pragma once

#include "chol_leaf.cuh"

namespace eod {
namespace {

constexpr int kLB = 32;            // columns per block
constexpr int kLBS = kLB + 1;      // odd row stride of the 32-wide buffers
constexpr int kLeafCluster = 8;    // CTAs when the leaf is spread (portable cluster size)
// Widths up to this run on one CTA column by column (chol_leaf.cuh).  Launch
// and read back, one CTA against cluster, us: 8 26 / 27, 16 30 / 30, 20 33 / 32,
// 24 35 / 34, 32 40 / 38, 64 76 / 59, 96 148 / 85, 128 274 / 120 (of these 16 are
// the measurement's own).
constexpr int kLeafOneCta = 16;

__device__ __forceinline__ uint32_t leaf_smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// v into the same shared-memory place of the cluster's CTA `rank`
__device__ __forceinline__ void st_cluster(uint32_t local, uint32_t rank, double v) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// barrier over every thread of the cluster; what was stored before it, in
// any CTA's shared memory, is visible after it
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__host__ __device__ inline size_t block_leaf_smem_bytes(int w) {
    const size_t own = (size_t)(w + kLeafCluster - 1) / kLeafCluster, ld = (size_t)(w | 1);
    const size_t d = 2 * own * ld + 2 * (size_t)w * kLBS + 2 * own * kLBS + 2 * kLB * kLBS + 2 * kLB * 9 + 8 * kLBS +
                     4 * (size_t)w + 40;
    return sizeof(double) * d + sizeof(long long) * 3 * (size_t)w;
}

// 1/d for normal d > 0: PTX's approximate reciprocal of a double as the seed r0,
// then r0 (1 + e + e^2), e = 1 - d r0, the geometric series of 1/d = r0 / (1 - e)
// up to its second order (as in recip_pos): with a seed good to 18 bits or more
// the rest, e^3, is below the roundings of the last FMAs.  Within 2 ulp of
// CUDA's division (tested through the leaf over the exponent range).  A d whose
// reciprocal would be subnormal gives 0.  A subnormal d gives NaN (the seed is
// +inf) where recip_pos gives +inf; with either the columns behind such a pivot
// are not finite and the next pivot is refused.
__device__ __forceinline__ double recip_pivot(double d) {
    double r0;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(d));
    const double e = fma(-d, r0, 1.0);
    return fma(r0, fma(e, e, e), r0);
}

// The entry (i, c) of an 8 x 8 block that a lane of diag8 holds.
struct Diag8Lane {
    int i, c, bi, bc;   // bx = x (x - 1) / 2
    __device__ __forceinline__ explicit Diag8Lane(int lane) {
        if (lane >= 28) {
            i = c = lane - 24;
        } else {
            i = 1;
            while ((i + 1) * i / 2 <= lane) ++i;
            c = lane - i * (i - 1) / 2;
        }
        bi = i * (i - 1) / 2;
        bc = c * (c - 1) / 2;
    }
};

// One warp: L D L^T of the n x n block at S (n <= 8, lower triangle, ld kLBS)
// with the pivot decisions for columns j0.., and Z = L^{-1} into Zd (its upper
// triangle zero), by Gauss-Jordan in registers.  Lane i (i - 1) / 2 + c holds
// entry (i, c), c < i: S(i, c) while column c is ahead, Z(i, c) once it is
// done; lanes 28-31 hold the diagonal entries 4-7, lanes 0-3 the entries 0-3
// in a second register (needed for three columns only).  A column's path is
// the reciprocal (three FP64 instructions), the multiplier, the update and a
// shuffle.  Column j of S keeps u_j(i) = d_j L(i, j), i > j.  Returns the
// number of columns kept.
__device__ __forceinline__ int diag8(const Diag8Lane &ln, double *S, double *Zd, int n, int j0, const long long *klo,
                                     const long long *khi, const long long *krg, int decide, double *dv, double *di,
                                     int *code) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, i = ln.i, c = ln.c;
    double a = i < n ? S[i * kLBS + c] : 0.0;
    double b = lane < 4 && lane < n ? S[lane * kLBS + lane] : 0.0;
    double d = S[0];
    int p = n;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j < n && p == n) {
            const double r = recip_pivot(d);
            const int bj = j * (j - 1) / 2;
            // u(i), then row j of [Z | S] in this lane's column (S is symmetric)
            const double u = __shfl_sync(FULL, a, ln.bi + j);
            const double row = __shfl_sync(FULL, a, c < j ? bj + c : ln.bc + j);
            double ub2 = 0.0;
            if (j < 3) {
                const double ub = __shfl_sync(FULL, a, lane < 4 ? lane * (lane - 1) / 2 + j : 0);
                ub2 = lane < 4 && lane > j ? ub * ub : 0.0;
            }
            const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
            const bool finite = ((bits >> 52) & 0x7ff) != 0x7ff;
            const long long kd = dkey(d);
            bool keep;
            int c0 = CHOL_ALL;
            if (!finite) {
                keep = false;
                c0 = decide ? CHOL_UNCERTAIN : CHOL_FAIL;
            } else if (decide) {
                keep = kd >= klo[j0 + j] && kd > khi[j0 + j] && kd > krg[j0 + j];
                if (!keep) c0 = kd < klo[j0 + j] ? CHOL_BELOW : CHOL_UNCERTAIN;
            } else {
                keep = kd > 0;
                if (!keep) c0 = CHOL_FAIL;
            }
            if (!keep) {
                p = j;
                *code = c0;
            } else {
                if (c == j && i > j && i < n) S[i * kLBS + j] = a;
                if (lane == 0) {
                    dv[j0 + j] = d;
                    di[j0 + j] = r;
                }
                if (j < 3) {
                    b = fma(-ub2, r, b);
                    d = __shfl_sync(FULL, b, j + 1);
                }
                const double M = i > j ? -(u * r) : 0.0;
                const double x = fma(M, row, a);
                a = (c == j && i > j) ? M : x;
                if (j >= 3 && j < 7) d = __shfl_sync(FULL, a, 25 + j);
            }
        }
    }
    if (i < n && c < i) {
        Zd[i * kLBS + c] = a;
        Zd[c * kLBS + i] = 0.0;
    }
    if (lane < n) Zd[lane * kLBS + lane] = 1.0;
    return p;
}

// sum over k < 8 of x[k] y[k sy], two chains
__device__ __forceinline__ double dot8(const double *x, const double *y, int sy) {
    double s0 = x[0] * y[0], s1 = x[1] * y[sy];
#pragma unroll
    for (int k = 2; k < 8; k += 2) {
        s0 = fma(x[k], y[k * sy], s0);
        s1 = fma(x[k + 1], y[(k + 1) * sy], s1);
    }
    return s0 + s1;
}
// sum over k < 32 of x[k] y[k], four chains
__device__ __forceinline__ double dot32(const double *x, const double *y) {
    double s[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) s[h] = x[h] * y[h];
#pragma unroll
    for (int k = 4; k < 32; k += 4)
#pragma unroll
        for (int h = 0; h < 4; ++h) s[h] = fma(x[k + h], y[k + h], s[h]);
    return (s[0] + s[1]) + (s[2] + s[3]);
}

__global__ void __launch_bounds__(kLeafThreads) chol_block_kernel(const LeafArgs A) {
    extern __shared__ double sh[];
    constexpr int NT = kLeafThreads, NWARP = NT / 32, C = kLeafCluster;
    const int w = A.w, q = blockIdx.x;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cap = (w + C - 1) / C, nown = q < w ? (w - q + C - 1) / C : 0;
    const int ld = w | 1;
    double *So = sh;                        // own rows r = q + C rho: S(r, c), c <= r; done columns hold X(r, c)
    double *Wo = So + cap * ld;             // own columns c = q + C gam of L^{-1}: W(r, c) at Wo[gam ld + r]
    double *Xg = Wo + cap * ld;             // the panels of even and odd blocks, every row: X(r, k) at [r kLBS + k]
    double *Lo = Xg + 2 * w * kLBS;         // own rows of X D^{-1}
    double *Zr = Lo + cap * kLBS;           // D^{-1} (the block's rows of W), own columns
    double *Sd = Zr + cap * kLBS;           // the diagonal block
    double *Zd = Sd + kLB * kLBS;           // its unit lower factor's inverse
    double *Xi = Zd + kLB * kLBS, *Li = Xi + kLB * 9, *Zt = Li + kLB * 9;   // 8 columns inside the block
    double *dv = Zt + 8 * kLBS, *di = dv + w, *sq = di + w, *rs = sq + w;
    double *nid = rs + w;                   // [kLeafCluster] partial sums, then the block_sum scratch
    double *red = nid + 8;                  // 32
    long long *klo = (long long *)(red + 32), *khi = klo + w, *krg = khi + w;
    __shared__ int pl_sh, code_sh;

    if (A.ni_tau2 > 0.0) {
        // near-identity Gram: the first-order factor (see chol_leaf.cuh)
        double acc = 0.0;
        for (int c = q + C * warp; c < w; c += C * NWARP)
            for (int i = lane; i <= c; i += 32) {
                const double v = A.G[i + (int64_t)c * A.ldg] - (i == c ? 1.0 : 0.0);
                acc = fma(i == c ? v : 2.0 * v, v, acc);
            }
        const double part = block_sum(acc, red);
        cluster_sync();            // every CTA of the cluster runs before its memory is written
        if (tid < C) st_cluster(leaf_smem_addr(nid + q), tid, part);
        cluster_sync();
        double tot = 0.0;
        for (int z = 0; z < C; ++z) tot += nid[z];
        if (tot <= A.ni_tau2) {
            for (int c = q + C * warp; c < w; c += C * NWARP)
                for (int i = lane; i < w; i += 32) {
                    const double g = (i <= c) ? A.G[i + (int64_t)c * A.ldg] : 0.0;
                    const double x = (i < c) ? g : (i == c ? 0.5 * (g - 1.0) : 0.0);
                    const double one = i == c ? 1.0 : 0.0;
                    A.R[i + (int64_t)c * A.ldr] = one + x;
                    if (A.Rinv) A.Rinv[i + (int64_t)c * A.ldinv] = one - x;
                    if (A.RinvF) A.RinvF[i + (int64_t)c * A.ldf] = (float)(one - x);
                    if (A.tdiag && i == c) A.tdiag[c] = fabs(A.tR1[c + (int64_t)c * A.ldr] * (one + x));
                }
            if (q == 0 && tid == 0) {
                A.info[0] = w;
                A.info[1] = CHOL_ALL;
            }
            return;
        }
    }

    // own rows (row r of S is column r of G's upper triangle), the first
    // diagonal block (every CTA reads it), the decision thresholds
    for (int o = warp; o < nown; o += NWARP) {
        const int r = q + C * o;
        for (int c = lane; c <= r; c += 32) So[o * ld + c] = A.G[c + (int64_t)r * A.ldg] + (c == r ? A.shift : 0.0);
    }
    for (int e = tid; e < kLB * kLB; e += NT) {
        const int i = e >> 5, k = e & 31;
        if (k <= i && i < w) Sd[i * kLBS + k] = A.G[k + (int64_t)i * A.ldg] + (k == i ? A.shift : 0.0);
    }
    if (A.decide)
        for (int j = tid; j < w; j += NT) {
            const double g0 = A.G[j + (int64_t)j * A.ldg], delta = A.delta_coef * g0;
            klo[j] = dkey(A.eps2 - delta);
            khi[j] = dkey(A.eps2 + delta);
            krg[j] = dkey(A.rho * g0);
        }
    for (int e = tid; e < cap * ld; e += NT) Wo[e] = 0.0;
    // zero above the diagonal and in the rows a narrow last block does not
    // have: the products below run over whole blocks
    for (int e = tid; e < kLB * kLBS; e += NT) Zd[e] = 0.0;
    if (tid == 0) code_sh = CHOL_ALL;
    // every CTA of the cluster has started before any writes into another
    cluster_sync();

    const bool worker = (warp & 3) != 0;               // not on the chain's sub-partition
    const int wid = warp - (warp >> 2) - 1;            // 0 .. 11 among the workers
    constexpr int NWK = NWARP - NWARP / 4;
    const Diag8Lane l8(lane);

    int p = 0;
    for (int B0 = 0; B0 < w; B0 += kLB) {
        const int nv = w - B0 < kLB ? w - B0 : kLB, B1 = B0 + kLB;
        const double *Xp = Xg + ((B0 / kLB + 1) & 1) * w * kLBS;   // the previous block's panel
        double *Xc = Xg + ((B0 / kLB) & 1) * w * kLBS;             // this block's
        const int of0 = (B0 - q + C - 1) / C;              // first own row >= B0, and own columns < B0
        // ---- what the previous block left: its update of the rows below this
        // block and of the own columns of L^{-1} (part of `parts`; a warp takes
        // 32 columns of a row, or 32 rows of a column) ----
        auto left = [&](int part0, int part1, int parts, int me, int nme) {
            if (B0 == 0) return;
            const int nch = (w - B0 + 31) / 32, orow = (B1 - q + C - 1) / C;   // own rows >= B1
            const int nrow = nown > orow ? nown - orow : 0, T = (nrow + of0) * nch;
            // one task per warp at least in the first part, where the warps have nothing else
            const int least = T < NWK ? T : NWK;
            const int t0 = part0 == 0 ? 0 : max(T * part0 / parts, least), t1 = max(T * part1 / parts, least);
            for (int t = t0 + me; t < t1; t += nme) {
                const int ch = t / (nrow + of0), oo = t - ch * (nrow + of0);
                if (oo < nrow) {
                    const int o = nown - 1 - oo, r = q + C * o, c = B0 + 32 * ch + lane;
                    if (c <= r) So[o * ld + c] -= dot32(Lo + o * kLBS, Xp + c * kLBS);
                } else {
                    const int g = oo - nrow, r = B0 + 32 * ch + lane;
                    if (r < w) Wo[g * ld + r] -= dot32(Zr + g * kLBS, Xp + r * kLBS);
                }
            }
        };
        // ---- the diagonal block, 8 columns at a time ----
        int got = 0, c0 = 0;
        for (int s = 0;; ++s, c0 += 8) {
            const int n = nv - c0 < 8 ? nv - c0 : 8;
            if (warp == 0) {
                const int pl = diag8(l8, Sd + c0 * kLBS + c0, Zd + c0 * kLBS + c0, n, B0 + c0, klo, khi, krg, A.decide, dv, di,
                                     &code_sh);
                if (lane == 0) pl_sh = pl;
            } else if (worker) {
                if (s > 0) {
                    // the rest of step s - 1 (columns e0 .. e0 + 7): entries dealt
                    // to the lanes one by one (a row to a warp left most idle, and
                    // an FP64 instruction costs the same for any number of lanes)
                    const int e0 = c0 - 8, nr = nv - c0, me = wid * 32 + lane;
                    const int inv_nr = (65535 + nr) / nr, inv_c0 = (65535 + c0) / c0;   // t / x = t inv_x >> 16 for t < 2^10
                    for (int t = me; t < (nr - 8) * nr; t += NWK * 32) {
                        const int k = (t * inv_nr) >> 16, r = c0 + 8 + k, c = c0 + t - k * nr;
                        if (c <= r) Sd[r * kLBS + c] -= dot8(Li + r * 9, Xi + c * 9, 1);
                    }
                    if (me < 8 * e0) {              // e0 = 8 or 16
                        const int k = me >> (e0 == 16 ? 4 : 3), c = me & (e0 - 1);
                        Zt[k * kLBS + c] = dot8(Zd + (e0 + k) * kLBS + e0, Zd + e0 * kLBS + c, kLBS);
                    }
                    asm volatile("bar.sync 1, 384;" ::: "memory");
                    for (int t = me; t < nr * c0; t += NWK * 32) {
                        const int k = (t * inv_c0) >> 16, r = c0 + k, c = t - k * c0;
                        const double v = dot8(Li + r * 9, c < e0 ? Zt + c : Zd + e0 * kLBS + c, kLBS);
                        Zd[r * kLBS + c] = (c < e0 ? Zd[r * kLBS + c] : 0.0) - v;
                    }
                    if (me < 8 * e0) {
                        const int k = me >> (e0 == 16 ? 4 : 3), c = me & (e0 - 1);
                        Zd[(e0 + k) * kLBS + c] = Zt[k * kLBS + c];
                    }
                }
                left(s ? s + 1 : 0, s + 2, 5, wid, NWK);
            }
            __syncthreads();
            const int pl = pl_sh;
            got = c0 + pl;
            if (pl < n || c0 + 8 >= nv) {
                // the columns left of this step's rows of the inverse
                if (c0 > 0 && warp < n) {
                    if (lane < c0) Zt[warp * kLBS + lane] = dot8(Zd + (c0 + warp) * kLBS + c0, Zd + c0 * kLBS + lane, kLBS);
                }
                left(s + 2, 5, 5, warp, NWARP);
                __syncthreads();
                if (c0 > 0 && warp < n && lane < c0) Zd[(c0 + warp) * kLBS + lane] = Zt[warp * kLBS + lane];
                __syncthreads();
                break;
            }
            // the 8 columns of the rows below in this block (Zd is zero above its
            // diagonal)
            {
                const int k = tid & 7, r = c0 + 8 + (tid >> 3);
                if (r < nv) {
                    const double x = dot8(Sd + r * kLBS + c0, Zd + (c0 + k) * kLBS + c0, 1);
                    Xi[r * 9 + k] = x;
                    Li[r * 9 + k] = x * di[B0 + c0 + k];
                }
            }
            __syncthreads();
            // the next 8 x 8 block (two lanes per entry); the others keep u
            if (tid < 128) {
                const int e = tid >> 1, i = e >> 3, c = e & 7, h = (tid & 1) * 4, r = c0 + 8 + i;
                double s4 = 0.0;
                if (c <= i && r < nv) {
                    const double *x = Li + r * 9 + h, *y = Xi + (c0 + 8 + c) * 9 + h;
                    s4 = fma(x[0], y[0], x[1] * y[1]) + fma(x[2], y[2], x[3] * y[3]);
                }
                s4 += __shfl_xor_sync(0xffffffffu, s4, 1);
                if (h == 0 && c <= i && r < nv) Sd[r * kLBS + c0 + 8 + c] -= s4;
            } else {
                for (int e = tid - 128; e < (nv - c0 - 8) * 8; e += NT - 128) {
                    const int r = c0 + 8 + (e >> 3), k = e & 7;
                    Sd[r * kLBS + c0 + k] = Xi[r * 9 + k];
                }
            }
            __syncthreads();
        }
        p = B0 + got;
        const bool last = got < nv || B1 >= w;
        // ---- own rows of the block, own columns of its rows of L^{-1} ----
        for (int o = warp; o < nown; o += NWARP) {
            const int r = q + C * o;
            if (r >= p) break;
            if (r >= B0 && lane < r - B0) So[o * ld + B0 + lane] = Sd[(r - B0) * kLBS + lane];
            // as a column: c = r
            double z = 0.0;
            if (lane < got) {
                if (r >= B0) z = lane >= r - B0 ? Zd[lane * kLBS + (r - B0)] : 0.0;
                else if (nv == kLB) z = dot32(Zd + lane * kLBS, Wo + o * ld + B0);
                else
                    for (int l = 0; l <= lane; ++l) z = fma(Zd[lane * kLBS + l], Wo[o * ld + B0 + l], z);
            }
            __syncwarp();
            if (lane < got) {
                Wo[o * ld + B0 + lane] = z;
                Zr[o * kLBS + lane] = z * di[B0 + lane];
            }
        }
        if (last) break;
        // ---- the panel: X = S L_bb^{-T} for the own rows below, pushed to every CTA ----
        const int ofirst = (B1 - q + C - 1) / C;   // first own row >= B1
        for (int o = ofirst + warp; o < nown; o += NWARP) {
            const int k = lane, r = q + C * o;
            const double x = dot32(So + o * ld + B0, Zd + k * kLBS);
            Lo[o * kLBS + k] = x * di[B0 + k];
            const uint32_t at = leaf_smem_addr(Xc + r * kLBS + k);
#pragma unroll
            for (int z = 0; z < C; ++z) st_cluster(at, z, x);
        }
        cluster_sync();
        // ---- the next diagonal block from its own rows, pushed to every CTA;
        // the own rows keep X ----
        for (int o = ofirst + warp; o < nown; o += NWARP) {
            const int r = q + C * o;
            if (r < B1 + kLB) {
                const int c = B1 + lane;
                if (c <= r) {
                    const double v = So[o * ld + c] - dot32(Lo + o * kLBS, Xc + c * kLBS);
                    const uint32_t at = leaf_smem_addr(Sd + (r - B1) * kLBS + c - B1);
#pragma unroll
                    for (int z = 0; z < C; ++z) st_cluster(at, z, v);
                }
            }
            So[o * ld + B0 + lane] = Xc[r * kLBS + lane];
        }
        cluster_sync();
    }
    for (int j = tid; j < p; j += NT) {
        const double s = sqrt(dv[j]);
        sq[j] = s;
        rs[j] = 1.0 / s;
    }
    __syncthreads();
    // R(i, c) = u_i(c) / sqrt(d_i) for i < c (own rows c of S), sqrt(d_c) on
    // the diagonal; R^{-1}(i, c) = Z(c, i) / sqrt(d_c) for i < c (own columns i)
    for (int o = warp; o < nown; o += NWARP) {
        const int c = q + C * o;
        if (c >= p) break;
        for (int i = lane; i < p; i += 32)
            A.R[i + (int64_t)c * A.ldr] = i < c ? So[o * ld + i] * rs[i] : (i == c ? sq[c] : 0.0);
        if (A.tdiag && lane == 0) A.tdiag[c] = fabs(A.tR1[c + (int64_t)c * A.ldr] * sq[c]);
    }
    if (A.Rinv || A.RinvF)
        for (int e = tid; e < nown * p; e += NT) {
            const int c = e / nown, o = e - c * nown, i = q + C * o;
            if (i >= p) continue;
            const double z = c > i ? Wo[o * ld + c] * rs[c] : (c == i ? rs[c] : 0.0);
            if (A.Rinv) A.Rinv[i + (int64_t)c * A.ldinv] = z;
            if (A.RinvF) A.RinvF[i + (int64_t)c * A.ldf] = (float)z;
        }
    if (q == 0 && tid == 0) {
        A.info[0] = p;
        A.info[1] = code_sh;
    }
}

}  // namespace
}  // namespace eod
