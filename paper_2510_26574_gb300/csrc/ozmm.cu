// FP64-accurate products C = A B^T on the tensor cores from precomputed digit
// planes, for the kernel-column engine of the FP64 path (Algorithm 2):
// X X(S,:)^T, F(:, :k) F(S, :k)^T and the solve G = R L^-T of each round.
//
// Operands.  A matrix enters as the seven-digit slicing of oz_digits.cuh with
// one exponent per row (max |row| < 2^E, so x = 2^(E - 6) sum_s d_s 2^(-8 s)
// up to 2^(E - 55)): plane s holds p_s = d_s 2^(-8 s) as BF16, in the tiles of
// oz_tile_at.  The producers (factor.cu, eig.cu) cut each operand once: X at the start
// of the factorisation, F's new columns in the epilogue of the solve (rows of
// F have norm <= 1 for the Gaussian kernel, so one exponent, E = 1, serves
// every row and the planes of old columns never change), R and L^-1 once per
// round, the pivot panels as gathers of rows of the X and F planes.  Columns
// past K up to the next multiple of 16 are zero in both operands; rows past the
// operand's end up to a multiple of 128 may hold anything.
//
// Products.  The 28 digit pairs with s + t <= 6 (issue order, accumulators and their
// drain: oz_mma.cuh), in 256-column chunks; after each chunk the exact levels go into an
// INT64 running sum T and the rest into an FP32 one M.  C(i, j) = 2^(E_i + E_j - 12)
// (T 2^-32 + M).
//
// Tiles: M = 128 rows of A by N = 64 rows of B (128 for three digits, whose
// three accumulators leave TMEM room for the wider shape), the contraction in
// 16-column quarters through a ring of bulk copies (A's tile, 4 D KB; B's as one copy
// per plane when a tile is half a row block).  Persistent CTAs, one per SM, walk the tiles: lane 0 of warp 0
// loads, warp 1 issues the 28 UMMAs of each quarter (A's planes in the collector
// buffer) and hands each finished accumulator to warps 2-17, which drain TMEM (lane
// quarter w % 4, columns [16 h + 64 g, 16 h + 64 g + 16), h = (w - 2) / 4, g < N / 64)
// into registers, release it, and write C (and, for the solve, the digit planes of C's
// new columns of F) while the next tile's products run.  Every wait is bounded (about
// one second); on a timeout the CTA sets bit 2 of flags, waits (bounded) for its own
// copies and MMAs, frees TMEM and exits.
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "factor.cuh"
#include "oz_digits.cuh"
#include "oz_mma.cuh"
#include "ozgemm.cuh"
#include "tc_ptx.cuh"

namespace kevd {

namespace {

constexpr int kQ = 16;
constexpr int kDrainWarps = 16;
constexpr int kThreads = (2 + kDrainWarps) * 32;
constexpr int kM = 128;
constexpr uint32_t kPlaneA = kM * 32;                    // one plane of a quarter: 128 rows x 32 bytes
constexpr uint32_t kCols = 512;                          // TMEM: 7 accumulators x 64 or 3 x 128 columns

// B rows per tile for a digit count: 64 for seven digits (seven accumulators), 128
// for three (three accumulators of 128 columns).
__host__ __device__ constexpr int oz_tile_n(int D) { return D == 3 ? 128 : 64; }

// Per digit count D (7: FP64 operands, 3: FP32 operands): the tile's B rows, the
// stage of one quarter (D planes of A and of B) and the ring depth.
template <int D>
struct OzCfg {
    static constexpr int kN = oz_tile_n(D);
    static constexpr uint32_t kPlaneB = kN * 32;
    static constexpr int kStages = D >= 6 ? 5 : 8;
    static constexpr uint32_t kStageA = D * kPlaneA;
    static constexpr uint32_t kStage = kStageA + D * kPlaneB;
    static constexpr size_t kSmem = (size_t)kStages * kStage + 1024;
    static_assert(kSmem <= 227 * 1024, "shared memory");
    static_assert(D * kN <= (int)kCols, "TMEM");
};

// D digits (levels 0 .. D - 1 of the pairs s + t <= D - 1; D = 3 or 7; WIDE: level 7 too).  rowdiv:
// C(i, :) is divided by rowdiv[i] (one reciprocal per row), when not NULL.
template <int D, bool STRICT, bool WIDE>
__global__ void __launch_bounds__(kThreads, 1)
    k_ozmm(const OzOperand A, const OzOperand B, int64_t M, int n, int K, const FactorState* __restrict__ st,
           double* __restrict__ Cout, int64_t ldc, int64_t c_koff, uint16_t* __restrict__ pout, int pout_nq,
           const double* __restrict__ rowdiv, int* __restrict__ flags) {
    const int* __restrict__ ea = A.e;
    const int* __restrict__ eb = B.e;
    constexpr int kN = OzCfg<D>::kN;
    constexpr int kNH = kN / 64;                               // 16-column groups per drain warp
    constexpr uint32_t kPlaneB = OzCfg<D>::kPlaneB;
    constexpr uint32_t kIdesc = idesc_bf16(kM, kN);
    constexpr int kStages = OzCfg<D>::kStages;
    constexpr uint32_t kStageA = OzCfg<D>::kStageA;
    constexpr uint32_t kStage = OzCfg<D>::kStage;
    extern __shared__ uint8_t smem_raw[];
    constexpr int NA = kOzAccs<D>;
    __shared__ __align__(8) uint64_t bars[2 * kStages + 2 * NA];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_fail;

    int ncols = n, pk = 0;
    if (st) {   // engine products: skipped rounds write nothing
        if (st->done || st->m == 0) return;
        if (K == -1) K = st->k;                                  // contraction over the current rank
        if (K == -2) K = st->m;                                  // ... over this round's pivots
        if (K == -3) K = st->kp;                                 // ... over F's padded planes
        if (c_koff) {                                            // output at columns k .. k + m - 1
            Cout += (int64_t)st->k * c_koff;
            pk = st->kp;
            ncols = min(n, st->m);
        }
    }
    // tiles: 128-row block rb, kN-column block jt, t = rb nj + jt (the j tiles of a row
    // block are neighbours, so they read A's planes at about the same time); CTA b
    // takes t = b, b + gridDim.x, ... and keeps the TMA ring and the MMAs running
    // across its tiles: a tile's epilogue overlaps the next tile's products
    const int nj = (n + kN - 1) / kN;
    const int64_t ntile = (M + kM - 1) / kM * nj;
    const int nq = (K + kQ - 1) / kQ;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t bar0 = smem_u32(&bars[0]);
    auto full = [&](int st) { return bar0 + 8u * (uint32_t)st; };
    auto empty = [&](int st) { return bar0 + 8u * (uint32_t)(kStages + st); };
    auto acc_full = [&](int a) { return bar0 + 8u * (uint32_t)(2 * kStages + a); };
    auto acc_empty = [&](int a) { return bar0 + 8u * (uint32_t)(2 * kStages + NA + a); };

    if (tid == 0) {
        for (int q = 0; q < kStages; ++q) {   // (stage indexes and phases run by increments: no divisions in the loops)
            mbar_init(full(q), 1);
            mbar_init(empty(q), 1);
        }
        for (int a = 0; a < NA; ++a) {
            mbar_init(acc_full(a), 1);
            mbar_init(acc_empty(a), kDrainWarps);
        }
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (wid == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);

    if (wid == 0) {
        // ---- copies of the quarters into the ring ----
        if (lane == 0) {
            int st_ = 0;
            uint32_t ph = 1;                                       // the first pass finds the stages empty
            bool ok = true;
            for (int64_t t = blockIdx.x; t < ntile && ok; t += gridDim.x) {
                const uint16_t* pa = A.p + oz_tile_at((t / nj) * kM, 0, 0, A.nq, D);
                const uint16_t* pb = B.p + oz_tile_at((t % nj) * kN, 0, 0, B.nq, D);
                for (int q = 0; q < nq; ++q) {
                    ok = mbar_wait_quick(empty(st_), ph, &s_fail);
                    if (!ok) break;
                    const uint32_t dst = base + (uint32_t)st_ * kStage;
                    mbar_expect_tx(full(st_), kStage);
                    bulk_g2s(dst, pa, kStageA, full(st_));
                    if (kN == 128) {
                        bulk_g2s(dst + kStageA, pb, D * kPlaneB, full(st_));
                    } else {
#pragma unroll
                        for (int s = 0; s < D; ++s)
                            bulk_g2s(dst + kStageA + s * kPlaneB, pb + s * 2048, kPlaneB, full(st_));
                    }
                    pa += D * 2048;
                    pb += D * 2048;
                    if (++st_ == kStages) {
                        st_ = 0;
                        ph ^= 1;
                    }
                }
            }
            if (!ok) {
                s_fail = 1;
                atomicOr(flags, 4);
            }
            // this CTA's copies have landed before it exits: every stage's last phase (a stage
            // never used waits on the phase before its first, which is complete)
            for (int j = 0; j < kStages; ++j) mbar_wait(full(j), j < st_ ? ph ^ 1 : ph);
        }
    } else if (wid == 1) {
        // ---- MMA issuer: one elected lane ----
        if (elect_one()) {
            OzIssuer<D, kN, STRICT, WIDE> is{tmem, kIdesc, kPlaneA >> 4, kPlaneB >> 4, acc_full(0), acc_empty(0), &s_fail};
            int st_ = 0, prev = -1;
            uint32_t ph = 0, prev_ph = 0;
            bool ok = true;
            for (int64_t t = blockIdx.x; t < ntile && ok; t += gridDim.x) {
                for (int q = 0; q < nq && ok; ++q) {
                    ok = mbar_wait_quick(full(st_), ph, &s_fail);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t sa = base + (uint32_t)st_ * kStage;
                    ok = is.quarter(sw32_desc(sa), sw32_desc(sa + kStageA), q, nq);
                    umma_commit(empty(st_));
                    prev = st_;
                    prev_ph = ph;
                    if (++st_ == kStages) {
                        st_ = 0;
                        ph ^= 1;
                    }
                }
            }
            if (!ok) {
                s_fail = 1;
                atomicOr(flags, 4);
            }
            if (prev >= 0) mbar_wait(empty(prev), prev_ph);        // the last commit covers the earlier ones
        }
        __syncwarp();
    } else {
        // ---- drain and epilogue: TMEM lane quarter wid % 4, columns [16 h + 64 g, + 16) ----
        const int wq = wid & 3, h = (wid - 2) >> 2;
        const int m = 32 * wq + lane;
        const int pcols = (ncols + kQ - 1) / kQ * kQ;   // new columns' planes: zeros past ncols up to 16
        OzDrain<D, kN, STRICT> dr{tmem + ((uint32_t)(32 * wq) << 16) + (uint32_t)(16 * h), acc_full(0), acc_empty(0),
                                  &s_fail};
        bool ok = true;
        for (int64_t t = blockIdx.x; t < ntile; t += gridDim.x) {
            const int64_t i0 = (t / nj) * kM;
            const int j0 = (int)(t % nj) * kN;
            // row and column exponents of the tile, loaded while its products run (lane 16 g + e
            // holds column j0 + 64 g + 16 h + e's)
            const int64_t gi = i0 + m;
            const int cj = j0 + 64 * (lane >> 4) + 16 * h + (lane & 15);
            const int ei = gi < M ? (ea ? ea[gi] : A.e_const) : -900;
            const int ejl = cj < ncols ? (eb ? eb[cj] : B.e_const) : -900;
            const double dinv = rowdiv && gi < M ? 1.0 / rowdiv[gi] : 1.0;
            long long Tacc[16 * kNH];
            float Macc[16 * kNH];
#pragma unroll
            for (int e = 0; e < 16 * kNH; ++e) {
                Tacc[e] = 0;
                Macc[e] = 0.f;
            }
            ok = dr.tile(nq, Tacc, Macc);
            if (!ok) break;
            // values four at a time (rolled, the sums moving down: see oz_mma.cuh on code size)
            double* cp = Cout + gi + (int64_t)(j0 + 16 * h) * ldc;
#pragma unroll 1
            for (int u = 0; u < 4 * kNH; ++u) {
                const int c0 = 4 * u + 48 * (u >> 2);           // 16 columns, then 16 more 64 further
                long long Tq[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int ej = __shfl_sync(0xffffffffu, ejl, 4 * u + e);
                    double v = 0.0;
                    if (ei > -900 && ej > -900)
                        v = STRICT ? oz_value_strict(Tacc[e], Macc[e], ei + ej - 12)
                                   : oz_value(Tacc[e], Macc[e], ei + ej - 12);
                    if (gi < M && j0 + 16 * h + c0 + e < ncols) cp[(int64_t)(c0 + e) * ldc] = rowdiv ? v * dinv : v;
                    Tq[e] = D == kDigits ? oz_T_f64<kDigits>(v, 1) : 0;
                }
#pragma unroll
                for (int e = 0; e < 16 * kNH - 4; ++e) {
                    Tacc[e] = Tacc[e + 4];
                    Macc[e] = Macc[e + 4];
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) Tacc[16 * kNH - 4 + e] = Tq[e];
            }
            if constexpr (D == kDigits) {                       // the solve: the digits of F's new columns are now in Tacc
                if (pout && gi < M && j0 + 16 * h < pcols)
                    oz_store_quarter<kDigits>(pout, gi, (pk + j0) / 16 + h, pout_nq, Tacc);
            }
        }
        if (!ok && lane == 0) {
            s_fail = 1;
            atomicOr(flags, 4);
        }
    }

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (wid == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

}  // namespace

template <int D, bool STRICT, bool WIDE = false>
static cudaError_t launch_ozmm_d(const OzOperand& A, const OzOperand& B, int64_t M, int n, int K,
                                 const FactorState* st, double* C, int64_t ldc, int64_t c_koff, uint16_t* pout,
                                 int pout_nq, const double* rowdiv, int* flags, int sms, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_ozmm<D, STRICT, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)OzCfg<D>::kSmem);
    if (e != cudaSuccess) return e;
    const int64_t ntile = (M + kM - 1) / kM * ((n + OzCfg<D>::kN - 1) / OzCfg<D>::kN);
    const dim3 grid((unsigned)std::min<int64_t>(ntile, sms));   // persistent: one CTA per SM
    k_ozmm<D, STRICT, WIDE><<<grid, kThreads, OzCfg<D>::kSmem, s>>>(A, B, M, n, K, st, C, ldc, c_koff, pout, pout_nq,
                                                                    rowdiv, flags);
    return cudaGetLastError();
}

cudaError_t launch_ozmm(const OzOperand& A, const OzOperand& B, int64_t M, int n, int K, const FactorState* st,
                        double* C, int64_t ldc, int64_t c_koff, uint16_t* pout, int pout_nq, int* flags,
                        cudaStream_t s, int digits, const double* rowdiv, bool strict, bool wide) {
    if (M < 1 || n < 1 || M >= ((int64_t)1 << 31) || (digits != 3 && digits != kDigits)) return cudaErrorInvalidValue;
    if (!A.p || !B.p || (reinterpret_cast<uintptr_t>(A.p) % 16) || (reinterpret_cast<uintptr_t>(B.p) % 16) ||
        (pout && (digits != kDigits || (reinterpret_cast<uintptr_t>(pout) % 32))))
        return cudaErrorInvalidValue;
    static int nsm[64] = {};
    int dev = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    int sms = dev >= 0 && dev < 64 ? nsm[dev] : 0;
    if (sms == 0) {
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) nsm[dev] = sms;
    }
    strict = strict || 16 * (int64_t)std::min(A.nq, B.nq) > kOzNarrowK;   // K <= 16 nq of both
    if (digits == 3)
        return strict ? launch_ozmm_d<3, true>(A, B, M, n, K, st, C, ldc, c_koff, pout, pout_nq, rowdiv, flags, sms, s)
                      : launch_ozmm_d<3, false>(A, B, M, n, K, st, C, ldc, c_koff, pout, pout_nq, rowdiv, flags, sms, s);
    if (strict) return launch_ozmm_d<kDigits, true>(A, B, M, n, K, st, C, ldc, c_koff, pout, pout_nq, rowdiv, flags, sms, s);
    return wide
               ? launch_ozmm_d<kDigits, false, true>(A, B, M, n, K, st, C, ldc, c_koff, pout, pout_nq, rowdiv, flags, sms, s)
               : launch_ozmm_d<kDigits, false>(A, B, M, n, K, st, C, ldc, c_koff, pout, pout_nq, rowdiv, flags, sms, s);
}

}  // namespace kevd
