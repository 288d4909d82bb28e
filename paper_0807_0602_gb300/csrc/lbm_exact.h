// FP64 arithmetic of the equilibrium on integers, with the same bits.
//
// sm_103a's FP64 pipe issues one warp instruction in some 76 cycles per
// scheduler, its integer pipe one in two.  The factors 3, 4.5 and 1.5 of Eqs.
// 3-5 and the sums ((1 +- 3 c) + 4.5 c^2) - 1.5 u^2 have operands of known
// size (|u| < 0.2), so each rounding to nearest even is done here on 64-bit
// fixed-point integers in units of 2^-61, at some 18 integer instructions an
// operation.  Plain C++ with no floating-point instruction, so that it can be
// compared with the compiler's FP64 on any machine.
#pragma once

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace sc {
namespace exact {

typedef unsigned long long u64;

LBM_HD int clz64(u64 v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

// A non-negative number m 2^(e - 1075): m = 0, or of 53 bits (2^53 itself
// after a rounding).
struct Num {
    u64 m;
    int e;
};

// |x| from the bits of x.  Subnormals count as zero: the sums below do not
// change by numbers that small.
LBM_HD Num num(u64 bits) {
    Num r;
    r.e = (int)((bits >> 52) & 0x7ff);
    r.m = r.e ? (bits & 0xfffffffffffffull) | 0x10000000000000ull : 0;
    return r;
}

// q / 2^k rounded to nearest even (k >= 1)
LBM_HD u64 rne(u64 q, int k) { return (q + ((1ull << (k - 1)) - 1) + ((q >> k) & 1)) >> k; }

// 3 x / 2^h and 9 x / 2^h, rounded to 53 bits
LBM_HD Num times3(Num x, int h) {
    const u64 q = 3 * x.m;
    const int k = 1 + (int)(q >> 54);
    return Num{rne(q, k), x.e + k - h};
}
LBM_HD Num times9(Num x, int h) {
    const u64 q = 9 * x.m;
    const int k = 3 + (int)(q >> 56);
    return Num{rne(q, k), x.e + k - h};
}

// Fixed point in units of 2^-61: the floor and whether bits were lost.
struct Fix {
    u64 v;
    u64 lost;
};
LBM_HD Fix fix(Num x) {   // x < 1
    const u64 w = x.m << 8;
    int q = 1022 - x.e;
    q = q > 63 ? 63 : q;
    Fix f;
    f.v = w >> q;
    f.lost = (f.v << q) != w;
    return f;
}

// a + x and a - x rounded to 53 bits (a a multiple of 2^-61 without lost
// bits, results between 2^-5 and 4)
LBM_HD u64 round53(u64 v, u64 lost) {
    const int k = 11 - clz64(v);   // bits below the 53rd
    v |= lost;                     // k >= 2: below half a unit either way
    v += ((1ull << (k - 1)) - 1) + ((v >> k) & 1);
    return v >> k << k;
}
LBM_HD u64 plus(u64 a, Fix x) { return round53(a + x.v, x.lost); }
LBM_HD u64 minus(u64 a, Fix x) { return round53(a - x.v - x.lost, x.lost); }

constexpr u64 kOne = 1ull << 61;

// Bits of the FP64 number v 2^-61 (v of at most 53 significant bits).
LBM_HD u64 bits(u64 v) {
    const int lz = clz64(v);
    return ((u64)(1024 - lz) << 52) + ((v << lz) >> 11);
}

// High word of u.u below which the functions below apply: u.u < 0.0390625, so
// that 3 |c| < 0.84, 4.5 c c < 0.36 and 1.5 u.u < 0.06 for all directions.
constexpr int kMaxUsqHigh = 0x3fa40000;

// b = 1.5 u.u, and 1 - b (the rest direction's bracket)
LBM_HD Fix b_of(u64 usq_bits) { return fix(times3(num(usq_bits), 1)); }
LBM_HD u64 rest(Fix b) { return bits(minus(kOne, b)); }

// Brackets ((1 +- 3 c) + 4.5 cc) - b of a pair of opposite directions, c for
// the first of them; cc = c c.
LBM_HD void pair(u64 c_bits, u64 cc_bits, Fix b, u64& first, u64& second) {
    const Fix t = fix(times3(num(c_bits), 0)), s = fix(times9(num(cc_bits), 1));
    const u64 p = bits(minus(plus(plus(kOne, t), s), b)), m = bits(minus(plus(minus(kOne, t), s), b));
    const bool neg = (c_bits >> 63) != 0;
    first = neg ? m : p;
    second = neg ? p : m;
}

}  // namespace exact
}  // namespace sc
