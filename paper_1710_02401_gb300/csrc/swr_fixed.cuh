// swr_fixed.cuh -- fixed-point arithmetic on the integer pipes for the
// matrix-vector products of the time windows.
//
// This part's FP64 unit does 1.6 multiply-adds per clock and SM (66 clocks
// latency); a 32 x 32 + 64-bit multiply-add is five integer instructions, 13 per
// clock and SM, measured with independent chains.
// A vector is therefore held as 56-bit integers relative to a power of two
// above its largest component (exponent shared by the vector), each cut into
// two 32-bit limbs, F = 2^28 hi + lo with |hi| <= 2^28, |lo| <= 2^27; a matrix
// likewise with one exponent a row (real time: one a matrix, which is used by
// rows and by columns), the power of two next to its 2-norm.  A product takes three
// multiply-adds: hi hi into one accumulator (units 2^-56 of the scales), hi lo +
// lo hi into a second (2^-84); lo lo is dropped, below 2^-58 of the scales (2^-57
// where limbs of two numbers have been added, in Karatsuba's products).  The
// accumulators are exact; every thread rounds its second one to a unit of the first
// when it folds it in, so another cut of a row into lanes, tiles or CTAs changes the
// sum by a few of these units.  (A double-single multiply-add on the FP32 pipes
// takes 13 instructions and keeps about 2^-46.)
//
// Against plain FP64 the representation error is 2^-57 of the row or the vector
// instead of 2^-53 of every product and partial sum: smaller in norm (a step matrix
// of 40 Gaussians times a vector, restated in exact arithmetic: 0.4e-16 against 0.8
// to 1.4e-16), larger in components far below the largest, which hold fewer than 53
// bits from 1/8 of it down (the same product: 3e-15 against 6e-16 relative in the
// worst component of a random vector; a smooth one's smallest, 1e-6 of the largest,
// 1e-11).  Nothing here reads single components against their own size: energies,
// norms, traces and residuals are sums over them.
//
// Bounds: a thread's first accumulator takes up to 96 terms of 2^56 before it is
// folded (real time, one electron, Q' of 96 Gaussians: 2^62.6), its second 192 of
// 2^55 there, 128 elsewhere.  A wrap of a partial sum would not matter, it is
// arithmetic modulo 2^64 and the total is what has to fit; sums over whole rows stay
// below 2^62 by Cauchy-Schwarz (fx_row_exp; vectors at most sqrt(2 K) times
// their scale).
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
// Exponent of a matrix row whose largest entry has exponent e and whose 2-norm
// squared is q in units of 2^(2 (e - 1022)): the smallest power of two of which the
// norm does not exceed sqrt(2) times.  Entries may then pass the scale by that
// factor, |hi| < 1.42 2^28; the product with a vector of K <= 1024 entries stays
// below 2^28.5 x 32 x 2^28 = 2^61.5 (complex: 2^62).
__device__ inline int fx_row_exp(int e, float q) {
    int x = -1;
    while (x < 6 && 1.99f * ldexpf(1.f, 2 * x) <= q) ++x;  // (q <= 2 K)
    return e >= FX_BAD ? FX_BAD : max(e + x, 0);
}
// 2^(1022 - e), the factor that takes entries of exponent e to units of that q.
__device__ inline double fx_row_scale(int e) { return e > 0 && e < 2045 ? __hiloint2double((2045 - e) << 20, 0) : 0.0; }
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
