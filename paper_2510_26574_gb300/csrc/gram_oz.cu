// Weighted Gram matrices of an FP64 factor on the tensor cores at FP64
// accuracy: A = F^T diag(wa) F and C = F^T diag(wc) F (Section 2.2), by an
// error-free slicing of the operands in the manner of Ozaki, Ogita, Oishi and
// Rump (2012), with BF16 slice products summed exactly in TMEM.
//
// Operands.  A = (sa F)^T (sa F) with sa = 1 / d~ and C = (sc F)^T (sc F) with
// sc = 1 / sqrt(q~): each Gram has one scaled operand for both sides, so one set of
// planes, and the scaling evens out the rows (with the whole weight on one side a
// row of small degree is tiny in the one operand and huge in the other, and its
// product is lost below their columns' largest entries).
//
// Slicing.  Every operand column c (over all rows) has an exponent E_c with
// max_i |x_ic| < 2^E_c.  T = round(x 2^(46 - E_c)) is an integer below 2^46,
// written in six balanced base-256 digits d_0 .. d_5 (d_s in [-128, 127]), so
// x = 2^(E_c - 6) sum_s d_s 2^(-8 s) up to 2^(E_c - 47).  Digit plane s holds
// p_s = d_s 2^(-8 s), an exact BF16 value.  U is the I block of columns, V the J block.
//
// Products.  The Gram entry is 2^(E_u + E_v - 12) sum_(s,t) sum_i p_s p_t; the
// pairs with s + t <= 5 and (3, 3) are kept (22 MMAs per 16 rows), the rest lie below
// 2^-48 of the largest product.  Level g = s + t has g + 1 pairs whose
// products are integer multiples of 2^(-8 g) below 2^14 in magnitude, so over
// 256 rows the level-g sum is an integer multiple of 2^(-8 g) below 2^24 for
// g <= 3: exact in an FP32 TMEM accumulator, whatever its rounding.  Levels 0-3
// have one accumulator each, level 4 two (pairs s <= 2 and s >= 3, each below
// 2^24 units of 2^-32: exact too) and level 5 a seventh.  One accumulator for
// levels 4 and 5 would not do: the tensor core truncates each addend to the
// accumulator's ulp, a bias that reaches ~2^-48 of the total over a chunk.
//
// Accumulation.  After every 256-row chunk the drain adds levels 0-4 (exact integers)
// to an INT64 running sum in units of 2^-32 and level 5 to an FP32 one.  The column
// scales 2^(E_u + E_v - 12) and the conversion to FP64 are applied once per CTA, and
// the partials of row splits and slabs are added in FP64.
//
// Seven digits (T below 2^54, 28 pairs with s + t <= 6, levels 5 and 6 in the seventh
// accumulator) serve the layouts of F that are not 16-byte aligned (oz_gram_digits).
//
// Layout.  The rows are taken in slabs sized so that the digit planes of one
// slab stay within a fixed budget.  k_oz_planes cuts a slab once: for each of
// sa F (and sc F) D planes of rank_pad columns x S rows of BF16, a
// column's rows contiguous, so that a TMA box of 32 rows x 128 (or 64) columns
// x D planes with the 64-byte swizzle lands as D K-major MMA operands of two
// 16-row quarters (64-byte rows: half as many L2 requests per byte as 32-byte
// rows).  Every tile of the Gram reads those planes instead of cutting
// FP64 data itself (the cutting, not the MMAs, bounded the rate when each CTA
// sliced its own tiles).
//
// Per CTA of k_gram_oz: one tile of M = 128 columns of the I block by N = 64
// columns of the J block, for one Gram and one range of rows of the slab:
//   * lane 0 of warp 0 keeps a ring of 32-row stages filled (two TMA loads per stage:
//     48 KB of U planes, 24 KB of V planes, three stages; 56 + 28 KB, two, with
//     seven digits);
//   * a lane of warp 1 issues the UMMAs (oz_mma.cuh: planes of U kept in the collector
//     buffer, the accumulators ending one after the other) and frees a stage by a commit;
//   * warps 2-17 drain (TMEM lane quarter w % 4, tile columns [16 h, 16 h + 16)
//     with h = (w - 2) / 4) and finally add the tile's FP64 partial.
// Bound: the issue of the MMAs (oz_mma.cuh).  Measured at N = 262,144, rank 1,101: both
// Grams 11.8 ms (17.9 ms with one reading of U's plane per MMA, level order and one
// barrier for all accumulators).  At N = 60,001, rank 401 (odd: seven digits) 0.70 ms,
// against 25.9 ms on the FP64 pipe.
// Every wait is bounded (about one second); on a timeout the CTA sets bit 2 of
// flags, waits (bounded) for its own copies and MMAs, frees TMEM and exits.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>

#include "common.cuh"
#include "gram_tc.cuh"
#include "oz_mma.cuh"
#include "tc_ptx.cuh"

namespace kevd {

constexpr int kOzQ = 16;          // rows per quarter (one MMA K step)
constexpr int kOzSQ = 2;          // quarters per stage (one 64-byte swizzled row of K)
constexpr int kOzDrainWarps = 16;
constexpr int kOzThreads = (2 + kOzDrainWarps) * 32;
constexpr int kOzM = 128, kOzN = 64;
constexpr uint32_t kOzPlaneU = kOzM * 64;               // one digit plane of a stage: 128 columns x 64 bytes
constexpr uint32_t kOzPlaneV = kOzN * 64;               // 4 KB
constexpr uint32_t kOzCols = 512;                       // TMEM: 7 accumulators x 64 columns (allocation: 512)
constexpr size_t kOzPlaneBudget = (size_t)6 << 30;      // bytes of digit planes per slab

// Per digit count D: one stage (72 KB at six digits, 84 KB at seven) and the ring depth.
template <int D>
struct OzGramCfg {
    static constexpr uint32_t kStageU = D * kOzPlaneU;
    static constexpr uint32_t kStage = kStageU + D * kOzPlaneV;
    static constexpr int kStages = D == 6 ? 3 : 2;
    static constexpr size_t kSmem = (size_t)kStages * kStage + 1024;
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

// Tile t -> (I, J) over I-blocks of 128 columns and J-blocks of 64 columns
// with J >= 2 I (the tiles holding some entry a <= c).
__device__ __forceinline__ void oz_tile_decode(int t, int nbi, int nbj, int& I, int& J) {
    I = 0;
    int len = nbj;
    while (t >= len && I + 1 < nbi) {
        t -= len;
        ++I;
        len = nbj - 2 * I;
    }
    J = 2 * I + t;
}

int oz_ntiles(int rank) {
    const int nbi = (rank + kOzM - 1) / kOzM, nbj = (rank + kOzN - 1) / kOzN;
    int n = 0;
    for (int I = 0; I < nbi; ++I) n += nbj - 2 * I;
    return n;
}

// D-digit planes of the slab of rows [row0, row0 + rows) (rows a multiple of 16;
// zero past N and past rank): set 0 from sa F, set 1 from sc F (when sc is given).
// Plane (set, s) is rank_pad x S BF16 pairs, word ((set D + s) rank_pad + c) S / 2 +
// i / 2 holding rows i, i + 1 of column c.  Block: 8 warps = 8 columns; a warp takes
// 64 rows per step (a lane two, as one 16-byte vector when the column is 16-byte
// aligned, else as two 8-byte loads: any F and ldf are cut).
template <int D>
__global__ void __launch_bounds__(256) k_oz_planes(const double* __restrict__ F, int64_t ldf, int64_t N, int rank,
                                                   int rank_pad, int64_t row0, int rows, int S,
                                                   const double* __restrict__ sa, const double* __restrict__ sc,
                                                   const int* __restrict__ Ecol, uint32_t* __restrict__ P) {
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= rank_pad) return;
    const bool on = c < rank;
    const size_t plane = (size_t)rank_pad * (S / 2);
    const int sets = sc ? 2 : 1;
    int E[2];
#pragma unroll
    for (int z = 0; z < 2; ++z) E[z] = (on && z < sets) ? Ecol[z * rank + c] : -900;
    const double* col = F + (int64_t)c * ldf;
    const bool vec = (reinterpret_cast<uintptr_t>(col) & 15) == 0;   // row0 is even
    for (int it = 0; it < 8; ++it) {
        const int il = blockIdx.y * 512 + it * 64 + 2 * lane;
        if (il >= rows) break;
        const int64_t i = row0 + il;
        double x0 = 0.0, x1 = 0.0;
        if (on && vec && i + 1 < N) {
            const double2 v = *reinterpret_cast<const double2*>(col + i);
            x0 = v.x;
            x1 = v.y;
        } else if (on && i < N) {
            x0 = col[i];
            if (i + 1 < N) x1 = col[i + 1];
        }
        const size_t at = (size_t)c * (S / 2) + (il >> 1);
#pragma unroll
        for (int z = 0; z < 2; ++z) {
            if (z >= sets) break;
            const double* w = z == 0 ? sa : sc;
            const double y0 = i < N ? __dmul_rn(w[i], x0) : 0.0;
            const double y1 = i + 1 < N ? __dmul_rn(w[i + 1], x1) : 0.0;
            uint32_t wd[D];
            oz_planes2<D>(oz_T_f64<D>(y0, E[z]), oz_T_f64<D>(y1, E[z]), wd);
#pragma unroll
            for (int s = 0; s < D; ++s) P[(size_t)(z * D + s) * plane + at] = wd[s];
        }
    }
}

// One tile (I, J) of Gram blockIdx.z over rows [blockIdx.y per, + per) of the
// slab's planes (rows of the slab: `rows`); the FP64 result is stored into
// (accumulate = 0) or added to (accumulate = 1) its partial in gpart.
template <int D>
__global__ void __launch_bounds__(kOzThreads, 1)
    k_gram_oz(const __grid_constant__ CUtensorMap tmUA, const __grid_constant__ CUtensorMap tmVA,
              const __grid_constant__ CUtensorMap tmUC, const __grid_constant__ CUtensorMap tmVC,
              const int* __restrict__ Ecol, int rank, int rows, int nbi,
              int nbj, int per, double* __restrict__ gpart, int ntiles, int accumulate, int* __restrict__ flags) {
    using Cfg = OzGramCfg<D>;
    constexpr int S = Cfg::kStages;
    constexpr int NA = kOzAccs<D>;
    constexpr uint32_t kIdesc = idesc_bf16(kOzM, kOzN);
    extern __shared__ uint8_t smem_raw[];
    // full[S], empty[S], acc_full[NA], acc_empty[NA]
    __shared__ __align__(8) uint64_t bars[2 * S + 2 * NA];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_fail;

    int I, J;
    oz_tile_decode(blockIdx.x, nbi, nbj, I, J);
    const int gram = blockIdx.z;                                   // 0: A (sa), 1: C (sc)
    const int r0 = blockIdx.y * per, r1 = min(r0 + per, rows);
    const int nq = r0 < r1 ? (r1 - r0 + kOzQ - 1) / kOzQ : 0;
    const int nst = (nq + kOzSQ - 1) / kOzSQ;                     // stages (the last may hold one quarter)
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto full = [&](int q) { return bar0 + 8u * (q % S); };
    auto empty = [&](int q) { return bar0 + 8u * (S + q % S); };
    auto acc_full = [&](int a) { return bar0 + 8u * (2 * S + a); };
    auto acc_empty = [&](int a) { return bar0 + 8u * (2 * S + NA + a); };

    if (tid == 0) {
        for (int q = 0; q < S; ++q) {
            mbar_init(full(q), 1);
            mbar_init(empty(q), 1);
        }
        for (int a = 0; a < NA; ++a) {
            mbar_init(acc_full(a), 1);
            mbar_init(acc_empty(a), kOzDrainWarps);
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (wid == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kOzCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    const CUtensorMap* tmU = gram ? &tmUC : &tmUA;
    const CUtensorMap* tmV = gram ? &tmVC : &tmVA;

    if (wid == 0) {
        // ---- TMA producer ----
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmU)) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmV)) : "memory");
            int q = 0;                                             // stage index
            for (; q < nst; ++q) {
                if (q >= S && !mbar_wait_or_fail(empty(q), (uint32_t)(q / S - 1) & 1, &s_fail)) break;
                const uint32_t dst = base + (uint32_t)(q % S) * Cfg::kStage;
                mbar_expect_tx(full(q), Cfg::kStage);
                tma_load_3d(dst, tmU, r0 + q * kOzSQ * kOzQ, I * kOzM, 0, full(q));
                tma_load_3d(dst + Cfg::kStageU, tmV, r0 + q * kOzSQ * kOzQ, J * kOzN, 0, full(q));
            }
            if (q < nst) {
                s_fail = 1;
                atomicOr(flags, 4);
            }
            // before the CTA ends: the copies of the last stages have landed
            for (int j = std::max(0, q - S); j < q; ++j) mbar_wait(full(j), (uint32_t)(j / S) & 1);
        }
    } else if (wid == 1) {
        // ---- MMA issuer: one elected lane ----
        if (elect_one()) {
            OzIssuer<D, kOzN, false> is{tmem, kIdesc, kOzPlaneU >> 4, kOzPlaneV >> 4, acc_full(0), acc_empty(0), &s_fail};
            int g = 0;
            bool ok = true;
            for (; g < nst && ok; ++g) {                           // stage g: quarters 2 g, 2 g + 1
                ok = mbar_wait_quick(full(g), (uint32_t)(g / S) & 1, &s_fail);
                if (!ok) break;
                tc_fence_after();
                const uint64_t du = sw64_desc(base + (uint32_t)(g % S) * Cfg::kStage);
                const uint64_t dv = sw64_desc(base + (uint32_t)(g % S) * Cfg::kStage + Cfg::kStageU);
                // (the second K step of the 64-byte rows is 32 bytes further: + 2 in the descriptors)
                for (int sub = 0; sub < kOzSQ && ok; ++sub)
                    if (2 * g + sub < nq) ok = is.quarter(du + 2 * sub, dv + 2 * sub, 2 * g + sub, nq);
                umma_commit(empty(g));
            }
            if (!ok) {
                s_fail = 1;
                atomicOr(flags, 4);
            }
            if (g > 0) mbar_wait(empty(g - 1), (uint32_t)((g - 1) / S) & 1);   // own MMAs complete
        }
        __syncwarp();
    } else {
        // ---- drain: TMEM lane quarter wid % 4, tile columns [16 h, 16 h + 16) ----
        const int wq = wid & 3, h = (wid - 2) >> 2;
        const int m = 32 * wq + lane;
        long long Tacc[16];
        float Macc[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            Tacc[e] = 0;
            Macc[e] = 0.f;
        }
        OzDrain<D, kOzN, false> dr{tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)(16 * h), acc_full(0), acc_empty(0),
                                   &s_fail};
        const bool ok = dr.tile(nq, Tacc, Macc);                   // rows per CTA are within kOzNarrowK
        if (!ok) {
            if (lane == 0) {
                s_fail = 1;
                atomicOr(flags, 4);
            }
        } else if (nq > 0) {
            // entry (m, 16 h + e) = 2^(E_u + E_v - 12) (T 2^-32 + M), into this split's FP64 partial
            const int ri = I * kOzM + m;
            const int Eoff = gram * rank;
            const int eu = ri < rank ? Ecol[Eoff + ri] : -900;
            double* o = gpart + (((size_t)gram * gridDim.y + blockIdx.y) * ntiles + blockIdx.x) * (kOzM * kOzN) +
                        (size_t)m * kOzN + 16 * h;
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                double v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int rj = J * kOzN + 16 * h + e + u;
                    const int ev = rj < rank ? Ecol[Eoff + rj] : -900;
                    v[u] = 0.0;
                    if (eu > -900 && ev > -900) v[u] = oz_value(Tacc[e + u], Macc[e + u], eu + ev - 12);
                }
                double2* dst = reinterpret_cast<double2*>(o + e);
                if (accumulate) {
                    const double2 old = *dst;
                    v[0] += old.x;
                    v[1] += old.y;
                }
                *dst = make_double2(v[0], v[1]);
            }
        } else if (!accumulate) {
            double* o = gpart + (((size_t)gram * gridDim.y + blockIdx.y) * ntiles + blockIdx.x) * (kOzM * kOzN) +
                        (size_t)m * kOzN + 16 * h;
            for (int e = 0; e < 16; ++e) o[e] = 0.0;
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (wid == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kOzCols) : "memory");
}

// Exponent mark of a column whose scaled entries are not finite: its digits are zero
// and its Gram entries come out as NaN (k_gram_oz_final).
constexpr int kOzNonFinite = 4000;

// High words (sign cleared) of sa_i and sc_i, once per row (sc may be NULL).
__global__ void k_weights_hi(const double* __restrict__ sa, const double* __restrict__ sc, int64_t N,
                             uint32_t* __restrict__ sa_hi, uint32_t* __restrict__ sc_hi) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    sa_hi[i] = (uint32_t)__double2hiint(sa[i]) & 0x7FFFFFFFu;
    if (sc) sc_hi[i] = (uint32_t)__double2hiint(sc[i]) & 0x7FFFFFFFu;
}

// log2 |x w| in units of 2^-20 (its fraction linear between powers of two), from
// the high words xh and wh: exponents added, the 20-bit significands multiplied in
// FP32.  Monotone up to the truncations, which take at most 4 units off, over the
// whole FP64 range (an FP32 product would overflow for weights above 2^128).
// Infinite and NaN factors give the largest key.
__device__ __forceinline__ int oz_log_key(uint32_t xh, uint32_t wh) {
    const float mx = __uint_as_float(0x3F800000u | ((xh & 0xFFFFFu) << 3));
    const float mw = __uint_as_float(0x3F800000u | ((wh & 0xFFFFFu) << 3));
    const int e = (int)(xh >> 20) + (int)(wh >> 20) - 2046;
    const int key = (int)((__float_as_uint(__fmul_rz(mx, mw)) - 0x3F800000u) >> 3) + (e << 20);
    return max(xh, wh) >= 0x7FF00000u ? INT_MAX : key;
}

// Column bounds of sa F and sc F for an FP64 factor: the keys (oz_log_key, biased by
// 2^31) of their largest entries, atomically maxed into cmax[0..2 rank) (zeroed
// before); only the exponents are needed.  All on the integer and FP32 pipes (FP64 is
// the slow pipe).  Each warp reads its column in 256-row steps: four 16-byte vectors
// per lane when the column is 16-byte aligned, else eight 8-byte loads (several loads
// in flight per lane either way), then the ragged end row by row.
__global__ void __launch_bounds__(256) k_colmax_f64(const double* __restrict__ F, int64_t ldf, int64_t N, int rank,
                                                    int64_t per, const uint32_t* __restrict__ sa_hi,
                                                    const uint32_t* __restrict__ sc_hi, uint32_t* __restrict__ cmax) {
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= rank) return;
    const int64_t i0 = (int64_t)blockIdx.y * per, i1 = min(i0 + per, N);
    const double* col = F + (int64_t)c * ldf;
    int ma = INT_MIN, mc = INT_MIN;
    auto take = [&](double x, uint32_t a, uint32_t w) {
        const uint32_t xh = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
        ma = max(ma, oz_log_key(xh, a));
        mc = max(mc, oz_log_key(xh, w));
    };
    int64_t i = i0;
    if ((reinterpret_cast<uintptr_t>(col + i0) & 15) == 0) {
        for (; i + 256 <= i1; i += 256) {
            double2 x[4];
            uint2 a[4], w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t e = i + 64 * u + 2 * lane;
                x[u] = *reinterpret_cast<const double2*>(col + e);
                a[u] = *reinterpret_cast<const uint2*>(sa_hi + e);
                w[u] = sc_hi ? *reinterpret_cast<const uint2*>(sc_hi + e) : make_uint2(0, 0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                take(x[u].x, a[u].x, w[u].x);
                take(x[u].y, a[u].y, w[u].y);
            }
        }
    } else {
        for (; i + 256 <= i1; i += 256) {
            double x[8];
            uint32_t a[8], w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int64_t e = i + 32 * u + lane;
                x[u] = col[e];
                a[u] = sa_hi[e];
                w[u] = sc_hi ? sc_hi[e] : 0;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) take(x[u], a[u], w[u]);
        }
    }
    for (i += lane; i < i1; i += 32) take(col[i], sa_hi[i], sc_hi ? sc_hi[i] : 0);
    ma = __reduce_max_sync(0xffffffffu, ma);
    mc = __reduce_max_sync(0xffffffffu, mc);
    if (lane == 0) {
        atomicMax(cmax + c, (uint32_t)ma + 0x80000000u);
        atomicMax(cmax + rank + c, (uint32_t)mc + 0x80000000u);
    }
}

// E = the smallest integer with max < 2^E (frexp's, or one higher when the maximum
// lies within 2^-18 of a power of two).  Negligible (< 2^-900) columns get E = -900,
// which makes all their digits zero; columns with infinities or NaN kOzNonFinite.
__global__ void k_colexp_f64(const uint32_t* __restrict__ cmax, int n, int* __restrict__ E) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    const int key = (int)(cmax[c] - 0x80000000u);
    const int e = ((min(key, INT_MAX - 4) + 4) >> 20) + 1;
    E[c] = key == INT_MAX || e > 1024 ? kOzNonFinite : e < -899 ? -900 : e;
}

// Sum of the split partials in a fixed order; entry (a, c) of tile (I, J) is
// Gram entry (128 I + a, 64 J + c), written with its mirror when it lies in the
// upper triangle (each unordered pair has exactly one such owner); acc adds to A and C.
__global__ void k_gram_oz_final(const double* __restrict__ gpart, int nsplit, int ntiles, int nbi, int nbj, int rank,
                                int ngram, const int* __restrict__ Ecol, int acc, double* __restrict__ A,
                                double* __restrict__ C) {
    int I, J;
    oz_tile_decode(blockIdx.x, nbi, nbj, I, J);
    const int gram = blockIdx.y;
    if (gram >= ngram) return;
    double* G = gram ? C : A;
    for (int e = threadIdx.x; e < kOzM * kOzN; e += blockDim.x) {
        const int a = e / kOzN, c = e % kOzN;
        const int ra = I * kOzM + a, rc = J * kOzN + c;
        if (ra >= rank || rc >= rank || ra > rc) continue;
        double sum = 0.0;
        for (int q = 0; q < nsplit; ++q)
            sum += gpart[(((size_t)gram * nsplit + q) * ntiles + blockIdx.x) * (kOzM * kOzN) + e];
        if (Ecol[gram * rank + ra] == kOzNonFinite || Ecol[gram * rank + rc] == kOzNonFinite)
            sum = __longlong_as_double(0x7FF8000000000000ll);
        if (acc) sum += G[(int64_t)rc * rank + ra];                // (each unordered pair has one thread)
        G[(int64_t)rc * rank + ra] = sum;
        G[(int64_t)ra * rank + rc] = sum;
    }
}

bool gram_oz_eligible(int64_t N, int rank) {
    if (const char* e = getenv("KEVD_GRAM")) {
        if (e[0] == 'f') return false;                          // KEVD_GRAM=fp64 / ffma: the FP64-pipe kernel
    }
    return rank >= 1 && N >= 1 && N < ((int64_t)1 << 31);
}

static int oz_rank_pad(int rank) { return (rank + kOzM - 1) / kOzM * kOzM; }

// Digits of F's planes: six when F's columns are 16-byte aligned, seven for the
// layouts that are not (an odd leading dimension), which the FP64-pipe kernel served
// before: its error against 64 bits (7e-16 of the Grams' 2-norm at N = 60,001, rank 401)
// is below six digits' (2e-14), seven digits keep it.
static int oz_gram_digits(const double* F, int64_t ldf) {
    return (reinterpret_cast<uintptr_t>(F) & 15) == 0 && ldf % 2 == 0 ? 6 : 7;
}

// Rows per slab: a multiple of 256 with the planes of all sets within kOzPlaneBudget, the
// rows spread evenly over the slabs (a short last slab would leave most SMs idle).
static int64_t oz_slab_rows(int64_t N, int rank, int ngram, int D) {
    const size_t per_row = (size_t)ngram * D * oz_rank_pad(rank) * 2;
    const int64_t most = std::max<int64_t>(256, (int64_t)(kOzPlaneBudget / per_row) / 256 * 256);
    const int64_t nslab = (N + most - 1) / most;
    return ((N + nslab - 1) / nslab + 255) / 256 * 256;
}

// Row splits per slab (the same in every slab): ntiles x ngram x nsplit CTAs
// filling whole waves of one CTA per SM, at least 4,096 rows per split and at most
// kOzNarrowK.
static int oz_nsplit(int64_t S, int64_t nctas, int nsm, int64_t least = 4096) {
    const int lo = (int)((S + kOzNarrowK - 1) / kOzNarrowK);
    int best = lo;
    double best_eff = -1.0;
    for (int sp = lo; sp <= lo + 8; ++sp) {
        if (sp > lo && S / sp < least) break;
        const int64_t blocks = nctas * sp;
        const double eff = (double)blocks / (double)(((blocks + nsm - 1) / nsm) * nsm);
        if (eff > best_eff + 0.01) {
            best_eff = eff;
            best = sp;
        }
    }
    return best;
}

size_t gram_oz_partial_doubles(int64_t N, int rank, int ngram, int nsm) {
    const int nt = oz_ntiles(rank);
    int ns = 1;
    for (int D = 6; D <= 7; ++D)
        ns = std::max(ns, oz_nsplit(oz_slab_rows(N, rank, ngram, D), (int64_t)nt * ngram, nsm));
    return (size_t)ngram * ns * nt * kOzM * kOzN;
}

size_t gram_oz_plane_bytes(int64_t N, int rank, int ngram) {
    size_t b = 0;
    for (int D = 6; D <= 7; ++D)
        b = std::max(b, (size_t)ngram * D * oz_rank_pad(rank) * (size_t)oz_slab_rows(N, rank, ngram, D) * 2);
    return b;
}

typedef CUresult (*EncodeTiledFnOz)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 3-D map over one set of planes (rows S, columns rank_pad, D digits), box
// 32 rows x `cols` columns x D digits with the 64-byte swizzle.
static bool oz_plane_map(EncodeTiledFnOz enc, CUtensorMap* map, uint16_t* base, int64_t S, int rank_pad, int cols,
                         int D) {
    const cuuint64_t dims[3] = {(cuuint64_t)S, (cuuint64_t)rank_pad, (cuuint64_t)D};
    const cuuint64_t strides[2] = {(cuuint64_t)S * 2, (cuuint64_t)S * 2 * rank_pad};
    const cuuint32_t box[3] = {(cuuint32_t)(kOzSQ * kOzQ), (cuuint32_t)cols, (cuuint32_t)D};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
static cudaError_t gram_oz_slabs(EncodeTiledFnOz enc, int64_t S, int ns, int acc, const double* F, int64_t ldf,
                                 int64_t N, int rank, const double* sa, const double* sc, const int* Ecol, double* gpart,
                                 uint16_t* planes, int* flags, double* A, double* C, cudaStream_t s) {
    cudaError_t e;
    const int ngram = sc ? 2 : 1;
    const int rank_pad = oz_rank_pad(rank);
    const size_t set = (size_t)D * rank_pad * S;                  // BF16 elements per set
    CUtensorMap mua, mva, muc, mvc;
    uint16_t* pc = planes + (ngram == 2 ? set : 0);
    if (!oz_plane_map(enc, &mua, planes, S, rank_pad, kOzM, D) || !oz_plane_map(enc, &muc, pc, S, rank_pad, kOzM, D) ||
        !oz_plane_map(enc, &mva, planes, S, rank_pad, kOzN, D) || !oz_plane_map(enc, &mvc, pc, S, rank_pad, kOzN, D))
        return cudaErrorInvalidValue;
    const int nbi = (rank + kOzM - 1) / kOzM, nbj = (rank + kOzN - 1) / kOzN;
    const int nt = oz_ntiles(rank);
    if ((e = cudaFuncSetAttribute(k_gram_oz<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)OzGramCfg<D>::kSmem)) != cudaSuccess)
        return e;
    for (int64_t row0 = 0; row0 < N; row0 += S) {
        const int rows = (int)((std::min<int64_t>(S, N - row0) + kOzQ - 1) / kOzQ * kOzQ);
        k_oz_planes<D><<<dim3((unsigned)(rank_pad / 8), (unsigned)((rows + 511) / 512)), 256, 0, s>>>(
            F, ldf, N, rank, rank_pad, row0, rows, (int)S, sa, sc, Ecol, reinterpret_cast<uint32_t*>(planes));
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        const int per = ((rows + ns - 1) / ns + kOzQ - 1) / kOzQ * kOzQ;
        k_gram_oz<D><<<dim3((unsigned)nt, (unsigned)ns, (unsigned)ngram), kOzThreads, OzGramCfg<D>::kSmem, s>>>(
            mua, mva, muc, mvc, Ecol, rank, rows, nbi, nbj, per, gpart, nt, row0 > 0 ? 1 : 0, flags);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    k_gram_oz_final<<<dim3((unsigned)nt, (unsigned)ngram), 256, 0, s>>>(gpart, ns, nt, nbi, nbj, rank, ngram, Ecol, acc,
                                                                        A, C);
    return cudaGetLastError();
}

// Column exponents of the scaled F, then the tensor-map encoder.
static cudaError_t gram_oz_begin(const double* F, int64_t ldf, int64_t N, int rank, const double* sa, const double* sc,
                                 uint32_t* sa_hi, uint32_t* sc_hi, uint32_t* cmax, int* Ecol, EncodeTiledFnOz* out,
                                 cudaStream_t s) {
    cudaError_t e;
    if ((e = cudaMemsetAsync(cmax, 0, 2 * (size_t)rank * sizeof(uint32_t), s)) != cudaSuccess) return e;
    const int ncs = (int)std::max<int64_t>(1, std::min<int64_t>(64, N / 8192));
    const int64_t pr = ((N + ncs - 1) / ncs + 255) / 256 * 256;
    k_weights_hi<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(sa, sc, N, sa_hi, sc ? sc_hi : nullptr);
    k_colmax_f64<<<dim3((rank + 7) / 8, (unsigned)((N + pr - 1) / pr)), 256, 0, s>>>(F, ldf, N, rank, pr, sa_hi,
                                                                                    sc ? sc_hi : nullptr, cmax);
    k_colexp_f64<<<(2 * rank + 255) / 256, 256, 0, s>>>(cmax, 2 * rank, Ecol);
    static EncodeTiledFnOz enc = nullptr;
    if (!enc) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &qr) !=
                cudaSuccess ||
            qr != cudaDriverEntryPointSuccess)
            return cudaErrorNotSupported;
        enc = reinterpret_cast<EncodeTiledFnOz>(p);
    }
    *out = enc;
    return cudaSuccess;
}

cudaError_t launch_gram_oz(const double* F, int64_t ldf, int64_t N, int rank, const double* sa, const double* sc,
                           uint32_t* sa_hi, uint32_t* sc_hi, uint32_t* cmax, int* Ecol, double* gpart,
                           uint16_t* planes, int* flags, double* A, double* C, int nsm, cudaStream_t s) {
    EncodeTiledFnOz enc;
    const cudaError_t e = gram_oz_begin(F, ldf, N, rank, sa, sc, sa_hi, sc_hi, cmax, Ecol, &enc, s);
    if (e != cudaSuccess) return e;
    const int D = oz_gram_digits(F, ldf), ngram = sc ? 2 : 1;
    const int64_t S = oz_slab_rows(N, rank, ngram, D);
    const int ns = oz_nsplit(S, (int64_t)oz_ntiles(rank) * ngram, nsm);
    return D == 6 ? gram_oz_slabs<6>(enc, S, ns, 0, F, ldf, N, rank, sa, sc, Ecol, gpart, planes, flags, A, C, s)
                  : gram_oz_slabs<7>(enc, S, ns, 0, F, ldf, N, rank, sa, sc, Ecol, gpart, planes, flags, A, C, s);
}

// Panels of the low-memory form: the planes stay within 64 MiB (its panel takes 128), and a
// split may be as short as 1,024 rows, since one panel has few tiles.  Seven digits, as the
// FP64-pipe Grams that it replaces have the error of.  Measured on N = 60,000, rank 512
// (factor and normalisation without stored F): 61.2 ms, 80.4 with the FP64-pipe Grams.
constexpr size_t kOzPanelBudget = (size_t)64 << 20;
static int64_t oz_panel_rows(int64_t P, int rank) {
    const int64_t most = (int64_t)(kOzPanelBudget / ((size_t)2 * kDigits * oz_rank_pad(rank) * 2)) / 256 * 256;
    const int64_t nslab = (P + std::max<int64_t>(most, 256) - 1) / std::max<int64_t>(most, 256);
    return ((P + nslab - 1) / nslab + 255) / 256 * 256;
}
static int oz_panel_splits(int64_t P, int rank, int nsm) {
    return oz_nsplit(oz_panel_rows(P, rank), (int64_t)oz_ntiles(rank) * 2, nsm, 1024);
}
size_t gram_oz_panel_partial_doubles(int64_t P, int rank, int nsm) {
    return (size_t)2 * oz_panel_splits(P, rank, nsm) * oz_ntiles(rank) * kOzM * kOzN;
}
size_t gram_oz_panel_plane_bytes(int64_t P, int rank) {
    return (size_t)2 * kDigits * oz_rank_pad(rank) * oz_panel_rows(P, rank) * 2;
}
cudaError_t launch_gram_oz_panel(const double* F, int64_t ldf, int64_t P, int64_t N, int rank, const double* sa,
                                 const double* sc, uint32_t* sa_hi, uint32_t* sc_hi, uint32_t* cmax, int* Ecol,
                                 double* gpart, uint16_t* planes, int* flags, double* A, double* C, int acc, int nsm,
                                 cudaStream_t s) {
    EncodeTiledFnOz enc;
    const cudaError_t e = gram_oz_begin(F, ldf, N, rank, sa, sc, sa_hi, sc_hi, cmax, Ecol, &enc, s);
    if (e != cudaSuccess) return e;
    return gram_oz_slabs<kDigits>(enc, oz_panel_rows(P, rank), oz_panel_splits(P, rank, nsm), acc, F, ldf, N, rank, sa,
                                  sc, Ecol, gpart, planes, flags, A, C, s);
}

}  // namespace kevd
