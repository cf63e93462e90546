// Arithmetic of the float64 digit products (gemm_digits.cu) that is not the tensor cores': the order in
// which a unit's accumulators are issued, restarted and drained, the scale and digits of an entry, and
// the rounding of the exact sums. Host-compilable, so that a host test runs the same functions.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define FO_DG __host__ __device__
#else
#define FO_DG
#endif

namespace fo {

constexpr int kPoison = 1 << 20;   // exponent of a matrix holding an infinity or a NaN

FO_DG inline int dg_clz(unsigned long long a) {   // a != 0
#if defined(__CUDA_ARCH__)
    return __clzll((long long)a);
#else
    return __builtin_clzll(a);
#endif
}

// The accumulator restarts: accumulator a's groups of k16 blocks (8 for the low orders, whose
// largest has 8 pairs: 64 MMAs; 16 for the high orders, at most 4 pairs) are shifted by a quarter
// group each. gs = log2 of a quarter group. begins / ends: whether block l of cnt starts / ends a
// group of accumulator a.
FO_DG constexpr bool acc_begins(int a, int l, int gs) {
    return l == 0 || ((l + (a << gs)) & ((4 << gs) - 1)) == 0;
}
FO_DG constexpr bool acc_ends(int a, int l, int cnt, int gs) {
    return l == cnt - 1 || ((l + 1 + (a << gs)) & ((4 << gs) - 1)) == 0;
}
// The accumulator issued q-th in block l: one that ends there first, one that begins there last.
FO_DG constexpr int acc_order(int q, int l, int gs) {
    const int qm = (1 << gs) - 1;
    if (((l + 1) & qm) == 0) return ((4 - (((l + 1) >> gs) & 3)) + q) & 3;
    if ((l & qm) == 0 && l > 0) return ((4 - ((l >> gs) & 3)) + 1 + q) & 3;
    return q;
}
// The block whose order and starts stand for phase `ph` (block l mod 4 << gs) at the issuer, which
// knows only the phase: block 4 << gs for phase 0, as inside a range; block 0 itself starts every
// accumulator, in that block's order.
FO_DG constexpr int acc_place(int ph, int gs) { return ph == 0 ? (4 << gs) : ph; }

// An e with b < 0.99 2^e (kPoison when b is not finite); any e serves a zero matrix.
FO_DG inline int scale_exp(double b) {
    if (!(b <= 1.7e308)) return kPoison;
    if (b < 1e-290) return -960;
    return ilogb(b * (1.0 / 0.989)) + 1;
}

// The digits of x at scale 2^e (|x| < 0.99 2^e) as the bytes d_i + 128, d_0 in the top byte: x
// 2^(63-e) rounded to an integer below 0.99 2^63, plus 128 at every byte.
FO_DG inline unsigned long long digits_of(double x, int e) {
    unsigned long long b;
    memcpy(&b, &x, 8);
    const int ex = (int)((b >> 52) & 0x7ff);
    const unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
    const int sh = (ex ? ex : 1) - 1012 - e;
    unsigned long long v;
    if (sh >= 0) v = m << (sh < 10 ? sh : 10);
    else if (sh > -55) v = (m + (1ull << (-sh - 1))) >> -sh;
    else v = 0;
    if ((long long)b < 0) v = 0ull - v;
    return v + 0x8080808080808080ull;
}

// (hi 2^32 + lo) 2^(e - 70) rounded to float64, to nearest even.
FO_DG inline double fixed_to_double(long long hi, long long lo, int e) {
    unsigned long long l = ((unsigned long long)hi << 32) + (unsigned long long)lo;
    unsigned long long h = (unsigned long long)((hi >> 32) + (lo >> 63)) + (l < (unsigned long long)lo ? 1ull : 0ull);
    const unsigned long long sign = h & 0x8000000000000000ull;
    if (sign) {
        l = 0ull - l;
        h = ~h + (l == 0ull ? 1ull : 0ull);
    }
    if ((h | l) == 0ull) return 0.0;
    const int lz = h ? dg_clz(h) : 64 + dg_clz(l);
    unsigned long long m, rest;   // the leading 64 bits, and what is left below them
    if (lz == 0) {
        m = h;
        rest = l;
    } else if (lz < 64) {
        m = (h << lz) | (l >> (64 - lz));
        rest = l << lz;
    } else {
        m = l << (lz - 64);
        rest = 0;
    }
    unsigned long long r = m >> 11;
    const unsigned long long low = m & 0x7ffull;
    r += (low > 0x400ull || (low == 0x400ull && (rest != 0ull || (r & 1ull)))) ? 1ull : 0ull;
    const int E = 127 - lz + e - 70 + 1023;   // biased exponent of the leading bit
    if (E > 0 && E < 2046) {
        const unsigned long long b = (((unsigned long long)E << 52) + (r - (1ull << 52))) | sign;
        double d;
        memcpy(&d, &b, 8);
        return d;
    }
    const double v = scalbn((double)r, E - 1023 - 52);
    return sign ? -v : v;
}

}  // namespace fo
