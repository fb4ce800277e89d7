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
// (collector::a::fill, ::use) reads A once per plane instead of once per MMA, and
// issuing from a warp-uniform loop under elect.sync (not one divergent lane) keeps the
// descriptors in uniform registers: measured 35.1 cycles per MMA (level order, one
// lane: 48.0; collector without elect: 44.9).  The last stage of a chunk is issued
// accumulator by accumulator instead, each committed to its own barrier, so that the
// drain of the first accumulators overlaps the MMAs of the last.
//
// Drain.  Level g < 5 holds integers I_g = L_g 2^(8 g) below 2^24: one conversion and
// one widening multiply-add each into an INT64 sum in units of 2^-32 (exact below 2^63
// for contractions up to 2^16 = kOzNarrowK).
//
// STRICT: levels 5 and 6 in level order, sums in units of 2^-24 with the rest of level 4
// in the FP32 sum, and one rounding at the end.  It serves contractions beyond
// kOzNarrowK, and the r x r stage: the subspace iteration stops at a residual of 1e-6,
// so another rounding of its products would move its vectors by as much.
#pragma once
#include "oz_digits.cuh"
#include "tc_ptx.cuh"

namespace kevd {

constexpr int kOzNarrowK = 65536;

// True in one lane of a converged warp.
static __device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}" : "=r"(p));
    return p != 0;
}

// umma_bf16 with a use of A's collector buffer: 0 none, 1 fill, 2 use, 3 last use.
template <int COL>
static __device__ __forceinline__ void umma_bf16_col(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                     uint32_t accumulate) {
    if constexpr (COL == 0) {
        umma_bf16(dtmem, adesc, bdesc, idesc, accumulate);
    } else if constexpr (COL == 1) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else if constexpr (COL == 2) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
            "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
            : "memory");
    }
}

template <int D>
constexpr int kOzAccs = D == 3 ? 3 : 7;

// The pairs formed: s + t < D, and (3, 3) beside them for six digits, whose one use is
// Grams of one operand with itself: of the level 6 terms left out there only d_3 d_3 has
// a sign on the diagonal (it biased the diagonal of a KS factor's Gram by -1.6e-12).
template <int D>
__host__ __device__ constexpr bool oz_pair(int s, int t) {
    return s + t < D || (D == 6 && s == 3 && t == 3);
}

// TMEM accumulator of the pair (s, lv - s), and whether it is the accumulator's
// first pair of a quarter (in both issue orders).
template <int D>
__host__ __device__ constexpr int oz_acc_of(int lv, int s) {
    return D == 3 || lv < 4 ? lv : lv == 4 ? (s <= 2 ? 4 : 5) : 6;
}
__host__ __device__ constexpr bool oz_lead(int lv, int s) { return (s == 0 && lv <= 5) || (lv == 4 && s == 3); }

// The pairs of accumulator a only.
template <int D, int N>
static __device__ __forceinline__ void oz_issue_acc(int a, uint32_t tmem, uint64_t da, uint64_t db, uint32_t pa,
                                                    uint32_t pb, uint32_t idesc, bool first) {
#pragma unroll
    for (int lv = 0; lv <= D; ++lv) {
#pragma unroll
        for (int s = 0; s <= lv; ++s) {
            if (!oz_pair<D>(s, lv - s) || oz_acc_of<D>(lv, s) != a) continue;
            umma_bf16(tmem + (uint32_t)(N * a), da + (uint64_t)(s * pa), db + (uint64_t)((lv - s) * pb), idesc,
                      (first && oz_lead(lv, s)) ? 0u : 1u);
        }
    }
}

// All pairs of one quarter, plane s of A held in the collector (one elected lane).
// da, db: descriptors of plane 0; pa, pb: plane strides in 16-byte units.
template <int D, int N, bool STRICT = false>
static __device__ __forceinline__ void oz_issue_planes(uint32_t tmem, uint64_t da, uint64_t db, uint32_t pa,
                                                       uint32_t pb, uint32_t idesc, bool first) {
#pragma unroll
    for (int s = 0; s < D; ++s) {
#pragma unroll
        for (int t = 0; t < D; ++t) {
            if (!oz_pair<D>(s, t) || (STRICT && s + t > 4)) continue;
            const uint32_t d = tmem + (uint32_t)(N * oz_acc_of<D>(s + t, s));
            const uint64_t a = da + (uint64_t)(s * pa), b = db + (uint64_t)(t * pb);
            const uint32_t acc = (first && oz_lead(s + t, s)) ? 0u : 1u;
            if (s == D - 1) umma_bf16_col<0>(d, a, b, idesc, acc);
            else if (t == 0) umma_bf16_col<1>(d, a, b, idesc, acc);
            else if (!oz_pair<D>(s, t + 1) || (STRICT && s + t == 4)) umma_bf16_col<3>(d, a, b, idesc, acc);
            else umma_bf16_col<2>(d, a, b, idesc, acc);
        }
    }
    if constexpr (STRICT && D > 5) oz_issue_acc<D, N>(6, tmem, da, db, pa, pb, idesc, first);
}

static __device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// Adds accumulator a's 16 values r of this thread to its sums T and M.
template <int D, bool STRICT = false>
static __device__ __forceinline__ void oz_add_level(int a, const uint32_t (&r)[16], long long* T, float* M) {
    if (D == 3 || a < 6) {
        const int g = a < 4 ? a : 4;
        const float up = __int_as_float((127 + 8 * g) << 23);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int i = __float2int_rn(__uint_as_float(r[e]) * up);
            if constexpr (STRICT) {
                if (g < 4) {
                    T[e] = mad_wide(i, 1 << (24 - 8 * g), T[e]);
                } else {
                    T[e] += (long long)(i >> 8);
                    M[e] += (float)(i & 255) * 0x1p-32f;
                }
            } else if (g == 0) {
                T[e] = (long long)((unsigned long long)T[e] + ((unsigned long long)(uint32_t)i << 32));
            } else {
                T[e] = mad_wide(i, 1 << (32 - 8 * (g ? g : 1)), T[e]);
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < 16; ++e) M[e] += __uint_as_float(r[e]);
    }
}

// M 2^up as a double by bit assembly (exact; 0 for subnormal, infinite or NaN M).
static __device__ __forceinline__ double oz_float_up(float M, int up) {
    const uint32_t mb = __float_as_uint(M), me = (mb >> 23) & 0xFF;
    return me != 0 && me != 0xFF
               ? __hiloint2double((int)((mb & 0x80000000u) | ((me + 896 + up) << 20) | ((mb >> 3) & 0xFFFFFu)),
                                  (int)(mb << 29))
               : 0.0;
}

// T 2^-32 + M (T 2^-24 + M when STRICT) times 2^sc as a double: T by its 32-bit halves
// over magic constants (exact), then additions only (an FP64 addition costs a quarter of
// a multiply-add on this GPU), STRICT in one rounding; the scale is an exponent add while
// the result stays normal.
template <bool STRICT = false>
static __device__ __forceinline__ double oz_value(long long T, float M, int sc) {
    const double hi = __hiloint2double(0x45300000, (int)((uint32_t)(T >> 32) ^ 0x80000000u));   // 2^84 + 2^63 + Th 2^32
    const double lo = __hiloint2double(0x43300000, (int)(uint32_t)T);                           // 2^52 + Tl
    double t;
    if constexpr (STRICT) {
        t = fma(oz_float_up(M, 0), 0x1p24, __dadd_rn(__dadd_rn(hi, -0x1.00000801p84), lo));   // T, then its one rounding
        sc -= 24;
    } else {
        t = __dadd_rn(__dadd_rn(hi, -0x1.000008p84), __dadd_rn(__dadd_rn(lo, -0x1p52), oz_float_up(M, 32)));
        sc -= 32;
    }
    const long long b = __double_as_longlong(t);
    const int be = (int)((b >> 52) & 0x7FF);
    if ((b & 0x7FFFFFFFFFFFFFFFll) == 0) return t;
    if (be + sc >= 1 && be + sc <= 2046) return __longlong_as_double(b + ((long long)sc << 52));
    return ldexp(t, sc);
}

}  // namespace kevd
