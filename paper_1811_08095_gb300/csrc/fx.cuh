// Block fixed point for the FP64-accuracy hops.
//
// GB300 issues about 2 FP64 operations per clock and SM but about 28 integer
// multiply-adds 32 x 32 + 64 -> 64 bits, so the SU(3) products of the hopping term, which are nearly all of its
// arithmetic, run in integers: a spinor of one 5D site is 24 signed integers with one exponent,
//     value = q 2^e,  |q| < 2^59,
// a link 18 integers with one exponent (|u| < 2^60 2^eu), both split into 31-bit limbs
//     q = q1 2^31 + q0,  -2^30 <= q0 < 2^30,
// and an output component sums q1 u1 and q1 u0 + q0 u1 in two 64-bit accumulators (q0 u0 is below
// the last unit kept).  The result resolves 2^-57 of the largest component of the neighbour, four
// bits beyond FP64's own rounding of it.  Components more than 2^kFxSpread below the largest of
// their 5D site, non-finite values and denormals keep their FP64 bits instead (exponent kFxRaw);
// warps that read such a neighbour take the FP64 arithmetic (fx_hop_f64), so nothing is lost on
// fields of extreme range and NaN and Inf propagate as in FP64.  (Components below 2^-1042 beside
// one above 2^-958 count as zero.)
//
// A link array holds nine (re1, re0, im1, im0) records per link, rows first, in the order of the FP64
// links ((p * 4 + mu) * Vh + h), and one exponent each behind them (kFxRaw: a non-finite link).
//
// Storage of a field: the 16-byte chunks of the FP64 layout (SpF64), each a complex number as
// (re1, re0, im1, im0), and one int32 exponent per 5D site at ex[h * Ns + s].  Limbs of a sum of two
// spins fit 32 bits without a carry.
#pragma once

#include "kernels.cuh"

namespace odwf {

constexpr int kFxRaw = 1 << 28;      // exponent marking FP64 bits
constexpr int kFxZero = -(1 << 24);  // exponent of an all-zero site (never the largest)
constexpr int kFxSpread = 32;        // largest exponent range of a site's nonzero components
constexpr int kFxMinField = 64;      // smallest biased exponent of a site's largest component

// (m << UP) >> (emax - exponent of d) of the 53-bit significand m of d, with d's sign.  A zero has
// exponent field 0 and is shifted out (shr.u64 clamps), emax being at least kFxMinField.
template <int UP>
__device__ __forceinline__ long long fx_from_double(double d, int emax) {
    const int hi = __double2hiint(d);
    unsigned long long m =
        ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(d);
    const int down = emax - ((hi & 0x7fffffff) >> 20);
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m << UP), "r"(down));
    const long long s = (long long)(hi >> 31);
    return ((long long)m ^ s) - s;
}

// One real as limbs
struct FxLimbs {
    int hi, lo;
};
__device__ __forceinline__ FxLimbs fx_split(long long q) {
    FxLimbs l;
    l.lo = (int)((unsigned)q << 1) >> 1;
    l.hi = (int)((q + (1ll << 30)) >> 31);
    return l;
}

__device__ __forceinline__ long long fx_join(int hi, int lo) { return ((long long)hi << 31) + lo; }

// q 2^e, the exponent added to the converted double's; |q| < 2^63 and kFxMinExp <= e <= kFxMaxExp for
// a hop's sums, |q| < 2^59 and any exponent of a stored site: no result leaves the normal range
constexpr int kFxMinExp = -1000, kFxMaxExp = 950;
__device__ __forceinline__ double fx_to_double(long long q, int e) {
    const double d = __ll2double_rn(q);
    const int hi = __double2hiint(d);
    return __hiloint2double(hi == 0 ? 0 : hi + (e << 20), __double2loint(d));
}

// 64-bit accumulation of a 32 x 32-bit product (one instruction)
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

// -a, opaque to the compiler: it would turn c + (-a) b into a product and a 64-bit subtraction
__device__ __forceinline__ int fx_neg(int a) {
    int r;
    asm("neg.s32 %0, %1;" : "=r"(r) : "r"(a));
    return r;
}

}  // namespace odwf
