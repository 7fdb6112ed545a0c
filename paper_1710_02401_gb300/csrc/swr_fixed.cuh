// swr_fixed.cuh -- fixed-point arithmetic on the integer pipes for the
// matrix-vector products of the time windows.
//
// This part's FP64 unit does 1.6 multiply-adds per clock and SM (66 clocks
// latency); a 32 x 32 + 64-bit multiply-add is five integer instructions, 13 per
// clock and SM, measured with independent chains.
// A vector is therefore held as 56-bit integers relative to a power of two
// above its largest component (exponent shared by the vector), each cut into
// two 32-bit limbs, F = 2^28 hi + lo with |hi| <= 2^28, |lo| <= 2^27; a matrix
// likewise with one exponent.  A product takes three multiply-adds:
// hi hi into one accumulator (units 2^-56 of the scales), hi lo + lo hi into a
// second (2^-84); lo lo, below 2^-58 of the scales, is dropped.  Sums are exact
// and so independent of their order.  Against plain FP64: the representation
// error is 2^-57 of the largest component instead of 2^-53 of each, the sums
// carry no rounding at all.  (A double-single multiply-add on the FP32 pipes
// takes 13 instructions and keeps about 2^-46.)
//
// Bounds: at most 64 terms of at most 2^56 go into the first accumulator of a
// thread, at most 128 of at most 2^55 into the second; it is folded into the
// first (rounded) before more are added.  Sums over whole rows stay below 2^62
// by Cauchy-Schwarz: row norms of the matrices are at most 1 (2^28 scaled), the
// vector's 2-norm at most sqrt(2 K) times its scale.
#pragma once

#include "swr_internal.cuh"

namespace swr {

#define FX_BITS 28
#define FX_BAD 0x7ff  // exponent field of infinities and NaN

// Biased exponent field of x (0 for zero and subnormals).
__device__ inline int fx_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Limbs of x relative to 2^(emax - 1022), emax >= fx_exp(x).
__device__ inline int2 fx_limbs(double x, int emax) {
    const long long u = __double_as_longlong(x);
    const int e = (int)((u >> 52) & 0x7ff), sh = e - emax + 3;
    const unsigned long long m = ((unsigned long long)u & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
    long long f;
    if (sh >= 0) f = (long long)(m << sh);
    else f = sh > -54 ? (long long)((m + (1ULL << (-sh - 1))) >> -sh) : 0;
    if (e == 0) f = 0;
    if (u < 0) f = -f;
    const int hi = (int)((f + (1LL << (FX_BITS - 1))) >> FX_BITS);
    return make_int2(hi, (int)(f - ((long long)hi << FX_BITS)));
}
// Weight of a unit of the first accumulator for a vector with exponent emax
// and a matrix scaled by 2^eg: 2^(emax - 1022 + eg - 56).
__device__ inline double fx_unit(int emax, int eg) {
    const int e = emax - 55 + eg;  // biased
    return e > 0 && e < 0x7ff ? __hiloint2double(e << 20, 0) : 0.0;
}
// s 2^e, rounded to nearest, without the FP64 pipe (0 below the normal range,
// NaN for exponents of non-finite operands).
__device__ inline double fx_double(long long s, int e) {
    if (s == 0) return 0.0;
    unsigned long long m = s < 0 ? 0ULL - (unsigned long long)s : (unsigned long long)s;
    const int z = __clzll((long long)m);
    m <<= z;                                   // leading bit 63
    m = (m >> 11) + ((m >> 10) & 1ULL);        // 53 bits, the next one rounds
    const int be = 1023 + 63 - z + e;          // biased exponent of bit 52 of m
    if (be <= 0) return 0.0;
    if (be >= 0x7fe) return __longlong_as_double(0x7ff8000000000000LL);
    const unsigned long long u = ((unsigned long long)(be - 1) << 52) + m;  // (a carry out of the rounding raises be)
    return __longlong_as_double((long long)(u | (s < 0 ? 0x8000000000000000ULL : 0ULL)));
}
__device__ inline long long fx_fold(long long s1, long long s2) { return s1 + ((s2 + (1LL << (FX_BITS - 1))) >> FX_BITS); }
__device__ inline void fx_mac(long long& s, int a, int b) { s += (long long)a * b; }
// (s1, s2) += a b for limb pairs.
__device__ inline void fx_mac2(long long& s1, long long& s2, int ah, int al, int bh, int bl) {
    fx_mac(s1, ah, bh);
    fx_mac(s2, ah, bl);
    fx_mac(s2, al, bh);
}
__device__ inline long long fx_shfl_xor(long long v, int o) {
    const int lo = __shfl_xor_sync(0xffffffffu, (int)(v & 0xffffffffLL), o);
    const int hi = __shfl_xor_sync(0xffffffffu, (int)(v >> 32), o);
    return ((long long)hi << 32) | (unsigned)lo;
}

}  // namespace swr
