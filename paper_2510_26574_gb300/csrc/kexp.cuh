// exp(-d2 s) for the Gaussian kernel values of the FP64 engine on the tensor cores, as a
// double, in integer arithmetic throughout (FP64 is the slow pipe of this GPU, 17 cycles per
// warp and SM for an operation of any kind; the integer pipe is not).  Tang's table-driven method (P. T. P. Tang, ACM TOMS 15(2), 1989) with 2^10
// table points and fixed point:
//   t = d2 s from the two significands' product, to units of 2^-54 (an FP64 product of
//   t >= 1 rounds more coarsely), n = rint(t 2^10 / ln 2) from t's upper word,
//   r = t - n ln 2 / 2^10 in units of 2^-62 (ln 2 / 2^10 to 2^-94; r is small, so 64 bits
//   hold it whatever overflows on the way),
//   exp(-t) = 2^-q 2^(j / 2^10) (1 + x + x^2/2 + x^3/6 + x^4/24), x = -r, -n = j - 2^10 q.
// |x| < 2^50.5 units: half a step, ln 2 / 2^11 = 2^50.47, and 2^-22 of t left out in choosing
// n.  The terms left out are below 2^-64 and those of third and fourth order, below 2^-36, are
// 32-bit products; every product is truncated to units of 2^-62 (errors of a few), and the
// product with the table entry is rounded once, to its 53 bits.  So the error is relative,
// below 0.76 ulp (1.5 from t = 256 on, where t has hi's own resolution): a kernel value keeps
// its digits however small it is, which the rows of F that lie far from every pivot need (the
// normalisation divides them by their own size).  For t >= 708 the result is 0 (exp(-708) <
// 2^-1021, far below every use).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace kevd {

// The table round(2^(j / 1024) 2^62), j < 1024, on the current device (filled
// once per process and device from host long double arithmetic): its device
// address in *tbl.
cudaError_t kexp_table(cudaStream_t s, const unsigned long long** tbl);

// A positive scale s = m 2^(e - 64), m >= 2^63 (1 / eps; any double, subnormal and
// infinite included).
struct KexpScale {
    unsigned long long m;
    int e;
};
inline KexpScale kexp_scale(double s) {
    if (!(s <= 1.7976931348623157e308)) return {1ull << 63, 4096};
    int e = 0;
    const double f = frexp(s, &e);                                   // in [1/2, 1)
    return {(unsigned long long)ldexp(f, 53) << 11, e};
}

__device__ __forceinline__ long long kexp_mulq62(long long a, long long b) {   // (a b) >> 62, signed
    const unsigned long long hi = (unsigned long long)__mul64hi(a, b);
    const unsigned long long lo = (unsigned long long)a * (unsigned long long)b;
    return (long long)((hi << 2) | (lo >> 62));
}

// The bits of exp(-d2 s).  d2 < 0 (a rounding residue of the squared distance) counts as 0.
// tbl: the 1024-entry table (shared or global memory).
__device__ __forceinline__ unsigned long long kexp_bits(double d2, KexpScale s, const unsigned long long* tbl) {
    const unsigned long long b1 = (unsigned long long)__double_as_longlong(d2);
    const int e1 = (int)(b1 >> 52);                                  // >= 2048: negative
    const unsigned long long hi = __umul64hi((b1 << 11) | (e1 ? 1ull << 63 : 0ull), s.m);
    const int sh = 1032 - (e1 ? e1 : 1) - s.e;                       // t 2^54 = hi 2^-sh
    unsigned long long t = ((hi >> ((sh - 1) & 63)) + 1) >> 1;
    if (sh > 64) t = 0;
    if (sh < 1) t = sh == 0 ? hi : sh == -1 && !(hi >> 63) ? hi << 1 : ~0ull;   // t >= 256
    if (e1 >= 2048) t = 0;
    if (t >= 708ull << 54) return 0;
    const int n = (int)(((t >> 32) * 3098164009ull + (1ull << 42)) >> 43);   // 2^31 / ln 2
    const unsigned long long c = (unsigned long long)n * 0xB17217F7D1CF7ull + ((unsigned long long)n * 0x9ABC9E3Bull >> 32);
    const long long x = (long long)(c - (t << 8));                   // ln 2 2^52 in two words
    const int x32 = (int)(x >> 20);                                  // units of 2^-42
    const int c3 = 357913941 + (int)(((long long)x32 * 89478485) >> 42);     // 1/6 + x/24 in units of 2^-31
    const long long c2 = (1ll << 61) + (((long long)x32 * c3) >> 11);        // 1/2 + x c3
    const long long c1 = (1ll << 62) + kexp_mulq62(x, c2);
    const unsigned long long p = (unsigned long long)((1ll << 62) + kexp_mulq62(x, c1));
    const unsigned long long T = tbl[-n & 1023];
    unsigned long long M = (__umul64hi(T, p) << 2) | ((T * p) >> 62);        // in [2^62 (1 - 2^-11.4), 2^63)
    int be = 1022 - ((n + 1023) >> 10);                              // biased exponent less the leading bit
    if (M < 1ull << 62) {
        M <<= 1;
        --be;
    }
    return ((unsigned long long)be << 52) + ((M + (1ull << 9)) >> 10);
}

}  // namespace kevd
