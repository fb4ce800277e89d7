// Issue and drain of the exact digit products (gram_oz.cu, ozmm.cu): the MMAs of one
// 16-deep quarter of D digit planes, and the sums of a finished chunk from TMEM.
//
// Levels lv = s + t < D of the digit pairs (s, t).  Levels 0-3 and the two halves of
// level 4 ({s <= 2}, {s >= 3}) each have a TMEM accumulator in which sums over 256
// rows are exact; levels 5 and 6 share a seventh (see oz_digits.cuh).  D = 3 uses
// three.
//
// Issue.  At N = 64 an MMA is bound by shared memory, not by the tensor pipe: 4 KB of
// A and 2 KB of B at 128 bytes per cycle are 48 cycles against 32 of arithmetic.
// Ordering the pairs by s and keeping plane s of A in the collector buffer
// (collector::a::fill, ::use) reads A once per plane instead of once per MMA: 35.1 cycles
// per MMA in isolation, ~43 in the kernels, where the issuing lane shares its scheduler
// with the drain.  One elected lane runs the whole loop, without divisions.
//
// A sum is exact for 16 quarters (a chunk).  The first and last quarter of a chunk are
// issued accumulator by accumulator, each with its own barriers, so that the drain of one
// accumulator overlaps the MMAs of the others.  (Ending the accumulators one after the
// other inside a chunk, in a spare slot of TMEM, was measured no faster: runtime slots cost
// the issuing lane what the overlap gains.)
//
// Drain.  Level g < 5 holds integers I_g = L_g 2^(8 g) below 2^24: one conversion and
// one widening multiply-add each into an INT64 sum in units of 2^-32 (exact below 2^62
// for contractions up to 2^15 = kOzNarrowK).  The rest of the kernels' arithmetic is on the
// integer pipe too: an FP64 operation of any kind costs 17 cycles per warp and SM here.
//
// WIDE (seven digits): the six pairs of level 7 that seven digits have join the seventh
// accumulator.  Without them a product is off by 2^-54 of its operands' largest entries per term,
// several times what the operands lose in being cut; with them by a third of that.  The low-memory
// form takes it (lowmem.cu): its products stand where FP64 arithmetic stood.
//
// STRICT: levels 5 and 6 in level order, sums in units of 2^-24 with the rest of level 4
// in the FP32 sum, and one rounding at the end.  It serves contractions beyond
// kOzNarrowK, and the r x r stage: the subspace iteration stops at a residual of 1e-6,
// so another rounding of its products would move its vectors by as much.
#pragma once


#include "oz_digits.cuh"
#include "tc_ptx.cuh"

namespace kevd {

constexpr int kOzNarrowK = 32768;

// True in one lane of a converged warp.
static __device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}" : "=r"(p));
    return p != 0;
}

// umma_bf16 that fills (FILL) or uses A's collector buffer.
template <bool FILL>
static __device__ __forceinline__ void umma_bf16_col(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                     uint32_t accumulate) {
    if constexpr (FILL) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    }
}

template <int D>
constexpr int kOzAccs = D == 3 ? 3 : 7;

// The pairs formed: s + t < D, and (3, 3) beside them for six digits, whose one use is
// Grams of one operand with itself: of the level 6 terms left out there only d_3 d_3 has
// a sign on the diagonal (it biased the diagonal of a KS factor's Gram by -1.6e-12); WIDE: level 7.
template <int D, bool WIDE>
__host__ __device__ constexpr bool oz_pair(int s, int t) {
    return s + t < D || (D == 6 && s == 3 && t == 3) || (WIDE && D == 7 && s + t == 7 && s > 0 && t > 0);
}

// TMEM accumulator of the pair (s, lv - s), and whether it is the accumulator's
// first pair of a quarter (in both issue orders).
template <int D>
__host__ __device__ constexpr int oz_acc_of(int lv, int s) {
    return D == 3 || lv < 4 ? lv : lv == 4 ? (s <= 2 ? 4 : 5) : 6;
}
__host__ __device__ constexpr bool oz_lead(int lv, int s) { return (s == 0 && lv <= 5) || (lv == 4 && s == 3); }

// True when the accumulators end with quarter q of nq.
static __device__ __forceinline__ bool oz_chunk_end(int q, int nq) { return q == nq - 1 || (q & 15) == 15; }

// mbarrier wait whose common case (already complete) costs one poll.
static __device__ __forceinline__ bool mbar_wait_quick(uint32_t bar, uint32_t parity, const volatile int* fail) {
    return mbar_try_wait(bar, parity) || mbar_wait_or_fail(bar, parity, fail);
}

// Issue state of one CTA (held by the elected lane).  da, db: descriptors of plane 0 of the
// quarter; pa, pb: plane strides in 16-byte units.
template <int D, int N, bool STRICT, bool WIDE = false>
struct OzIssuer {
    static constexpr int NA = kOzAccs<D>;
    uint32_t tmem, idesc, pa, pb;
    uint32_t acc_full, acc_empty;    // barrier addresses of accumulator 0 (8 bytes apart)
    const volatile int* fail;
    uint32_t chunks = 0;             // chunks ended so far

    // Quarter q of nq of the current tile; false when a wait gave up.
    __device__ __forceinline__ bool quarter(uint64_t da, uint64_t db, int q, int nq) {
        const bool end = oz_chunk_end(q, nq), start = (q & 15) == 0;
        if (end || start) {
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                // the drain has read accumulator a's previous sum
                if (start && chunks > 0 && !mbar_wait_quick(acc_empty + 8u * a, (chunks - 1) & 1, fail)) return false;
#pragma unroll
                for (int lv = 0; lv <= D; ++lv)
#pragma unroll
                    for (int s = 0; s <= lv; ++s)
                        if (oz_pair<D, WIDE>(s, lv - s) && oz_acc_of<D>(lv, s) == a)
                            umma_bf16(tmem + (uint32_t)(N * a), da + (uint64_t)(s * pa), db + (uint64_t)((lv - s) * pb),
                                      idesc, (start && oz_lead(lv, s)) ? 0u : 1u);
                if (end) umma_commit(acc_full + 8u * a);
            }
            chunks += end;
            return true;
        }
        // plane s of A in the collector; STRICT: levels 5 and 6 afterwards, in level order
#pragma unroll
        for (int s = 0; s < D; ++s) {
#pragma unroll
            for (int t = 0; t < D; ++t) {
                if (!oz_pair<D, WIDE>(s, t) || (STRICT && s + t > 4)) continue;
                const uint32_t d = tmem + (uint32_t)(N * oz_acc_of<D>(s + t, s));
                const uint64_t pda = da + (uint64_t)(s * pa), pdb = db + (uint64_t)(t * pb);
                if (t == 0) umma_bf16_col<true>(d, pda, pdb, idesc, 1u);
                else umma_bf16_col<false>(d, pda, pdb, idesc, 1u);
            }
        }
        if constexpr (STRICT && D > 5) {
#pragma unroll
            for (int lv = 5; lv < D; ++lv)
#pragma unroll
                for (int s = 0; s <= lv; ++s)
                    umma_bf16(tmem + (uint32_t)(N * 6), da + (uint64_t)(s * pa), db + (uint64_t)((lv - s) * pb), idesc, 1u);
        }
        return true;
    }
};

static __device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// Adds the 16 values r of level g < 5 (a half of level 4) of this thread to its sums T and
// M; FIRST: g = 0.
template <bool FIRST, bool STRICT>
static __device__ __forceinline__ void oz_add_level(int g, const uint32_t (&r)[16], long long* T, float* M) {
    const float up = FIRST ? 1.f : __int_as_float((127 + 8 * g) << 23);
    const int mul = STRICT ? 1 << max(24 - 8 * g, 0) : 1 << (32 - 8 * max(g, 1));
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int i = __float2int_rn(__uint_as_float(r[e]) * up);
        if constexpr (STRICT) {
            if (FIRST || g < 4) {
                T[e] = mad_wide(i, mul, T[e]);
            } else {
                T[e] += (long long)(i >> 8);
                M[e] += (float)(i & 255) * 0x1p-32f;
            }
        } else if constexpr (FIRST) {
            T[e] = (long long)((unsigned long long)T[e] + ((unsigned long long)(uint32_t)i << 32));
        } else {
            T[e] = mad_wide(i, mul, T[e]);
        }
    }
}

// Drain state of one warp: TMEM address of its 32 lanes and 16 columns of accumulator 0.
template <int D, int N, bool STRICT>
struct OzDrain {
    static constexpr int NA = kOzAccs<D>;
    static constexpr int NH = N / 64;   // 16-column groups, 64 columns apart
    uint32_t taddr, acc_full, acc_empty;
    const volatile int* fail;
    uint32_t ends = 0;               // parity of accumulator a's number of ends: bit a

    // Accumulator a's sums of this warp into T and M; false when the wait gave up.
    __device__ __forceinline__ bool take(int a, long long* T, float* M) {
        const bool w = mbar_wait_quick(acc_full + 8u * a, (ends >> a) & 1, fail);
        if (!__all_sync(0xffffffffu, w)) return false;
        ends ^= 1u << a;
        tc_fence_after();
#pragma unroll
        for (int half = 0; half < NH; ++half) {
            uint32_t r[16];
            tmem_ld16_async(taddr + (uint32_t)(N * a + 64 * half), r);
            tmem_wait_ld16(r);
            if (half == NH - 1) {                               // the accumulator may be overwritten
                tc_fence_before();
                __syncwarp();
                if ((threadIdx.x & 31) == 0) mbar_arrive(acc_empty + 8u * a);
            }
            if (a == 0) {
                oz_add_level<true, STRICT>(0, r, T + 16 * half, M + 16 * half);
            } else if (D == 3 || a < 6) {
                oz_add_level<false, STRICT>(a < 4 ? a : 4, r, T + 16 * half, M + 16 * half);
            } else {
#pragma unroll
                for (int e = 0; e < 16; ++e) M[16 * half + e] += __uint_as_float(r[e]);
            }
        }
        return true;
    }

    // The sums of a whole tile of nq quarters.  (Three digits: rolled, for the registers.)
    __device__ __forceinline__ bool tile(int nq, long long* T, float* M) {
        for (int q = max(0, min(15, nq - 1)); q < nq; ++q) {   // (a walk over the quarters: fewer spills than by chunks)
            if (!oz_chunk_end(q, nq)) continue;
            if constexpr (D == 3) {
#pragma unroll 1
                for (int a = 0; a < NA; ++a)
                    if (!take(a, T, M)) return false;
            } else {
#pragma unroll
                for (int a = 0; a < NA; ++a)
                    if (!take(a, T, M)) return false;
            }
        }
        return true;
    }
};

// (T 2^-32 + M) 2^sc as a double, in integer arithmetic: an FP64 operation of any kind
// costs 17 cycles per warp and SM on this GPU, so that four additions per value took
// 19,000 cycles of a 128 x 64 tile's epilogue (measured; its MMAs at K = 128: 8,000).  T is
// normalised to 62 bits (|T| < 2^62), M added at its scale, the sum rounded once (|M| < 2^-5 for
// contractions up to kOzNarrowK).
static __device__ __forceinline__ double oz_value(long long T, float M, int sc) {
    const unsigned long long a = (unsigned long long)(T < 0 ? -T : T);
    const int sh = __clzll((long long)(a | (1ull << 27))) - 2;
    const uint32_t mb = __float_as_uint(M);
    const int k = (int)((mb >> 23) & 0xFF) - 118 + sh;          // M = m 2^(e - 150), wanted in units of 2^(-32 - sh)
    const unsigned long long m = (mb & 0x7FFFFFu) | 0x800000u;
    long long mv = (long long)(k >= 0 ? m << min(k, 38) : m >> min(-k, 63));
    if (mb >> 31) mv = -mv;
    const long long V = (long long)((unsigned long long)T << sh) + mv;
    if (V == 0) return 0.0;
    const unsigned long long v = (unsigned long long)(V < 0 ? -V : V);
    const int lz = __clzll((long long)v);
    const unsigned long long n = v << lz;
    const unsigned long long r = (n >> 11) + ((n >> 10) & 1);   // 53 bits, possibly 2^53
    const int be = 63 - lz + sc - 32 - sh + 1023;               // biased exponent
    const unsigned long long sign = (unsigned long long)V & 0x8000000000000000ull;
    if (be >= 1 && be <= 2045) return __longlong_as_double((long long)((((unsigned long long)(be - 1)) << 52) + r + sign));
    const double t = ldexp((double)(long long)r, be - 1023 - 52);
    return V < 0 ? -t : t;
}

// (T 2^-24 + M) 2^sc, the form of the STRICT sums: T and M become doubles by bit assembly
// (exact: |T| < 2^53 for contractions below 2^17 columns, M normal or negligible), one FMA,
// and the scale by an exponent add when it stays normal.
static __device__ __forceinline__ double oz_value_strict(long long T, float M, int sc) {
    double td = 0.0;
    if (T != 0) {
        const unsigned long long u = T < 0 ? (unsigned long long)(-T) : (unsigned long long)T;
        const int msb = 63 - __clzll(u);
        if (msb <= 52) {
            td = __longlong_as_double((long long)(((unsigned long long)(T < 0) << 63) |
                                                  ((unsigned long long)(msb + 1023) << 52) |
                                                  ((u << (52 - msb)) & 0xFFFFFFFFFFFFFull)));
        } else {
            td = (double)T;
        }
    }
    double md = 0.0;
    const uint32_t mb = __float_as_uint(M), me = (mb >> 23) & 0xFF;
    if (me != 0 && me != 0xFF)
        md = __longlong_as_double((long long)(((unsigned long long)(mb >> 31) << 63) |
                                              ((unsigned long long)(me - 127 + 1023) << 52) |
                                              ((unsigned long long)(mb & 0x7FFFFF) << 29)));
    const double t = fma(md, 0x1p24, td);
    const long long b = __double_as_longlong(t);
    const int be = (int)((b >> 52) & 0x7FF);
    sc -= 24;
    if ((b & 0x7FFFFFFFFFFFFFFFll) == 0) return t;              // zero (integer test: no FP64 compare)
    if (be + sc >= 1 && be + sc <= 2046) return __longlong_as_double(b + ((long long)sc << 52));
    return ldexp(t, sc);
}

}  // namespace kevd
