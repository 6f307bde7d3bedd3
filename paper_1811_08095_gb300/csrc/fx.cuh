// Block fixed point for the FP64-accuracy hops.
//
// GB300 issues about 2 FP64 operations per clock and SM but about 28 integer
// multiply-adds 32 x 32 + 64 -> 64 bits, so the SU(3) products of the hopping term, which are nearly all of its
// arithmetic, run in integers: a spinor of one 5D site is 24 signed integers with one exponent,
//     value = q 2^e,  |q| < 2^59,
// a link 18 integers with one exponent (|u| < 2^60 2^eu), both split into 31-bit limbs
//     q = q1 2^31 + q0,  -2^30 <= q0 < 2^30,
// and an output component sums q1 u1 and q1 u0 + q0 u1 in two 64-bit accumulators (q0 u0 is below
// the last unit kept).
//
// What this resolves is relative to the largest component: half of 2^-58 of the 5D site's when it is stored, and
// about 2^-56 of the largest neighbour's in the sum over the eight directions.  FP64 keeps every complex
// component to 2^-53 of the terms it is made of, so two tests send what would be worse than that to FP64
// arithmetic:
//   * a term of the stencil adds an upper and a lower spin of one colour.  A 5D site where the larger
//     of such a pair is more than 2^kFxSpread below the largest component of the site, for any of the twelve pairs
//     (two upper spins, two lower spins, three colours), keeps its FP64 bits (exponent + kFxRaw).  A pair that
//     is stored in fixed point resolves 2^-52 of itself or better.  One chirality alone may be smaller, as it is on
//     the domain walls.  Warps that read FP64 bits convert them (fx_hop_conv): nothing is lost for the next test.
//     Share of such 5D sites at kFxSpread = 6 / 7 / 8, 16^3x32x16, m_q = 0.002: solution for a Gaussian source
//     5e-6 / 0 / 0, for a point source 5e-3 / 5e-4 / 5e-5.  On diagonal links a colour 2^-7 below the others errs by
//     1.1e-16 of itself at 7, as in FP64, and by 1.4e-16 at 8.
//   * the stencil adds up |w| of its terms for each complex component.  A sum of leading words below kFxWeak,
//     3/32 to 3/16 of the largest neighbour component, or twice that beside links with an entry of
//     modulus 1, means that the component is made of small terms only (links that do not mix colours, a large
//     neighbour in other spins), and the warp repeats the stencil in FP64 (fx_hop_f64).  Above it the stencil errs
//     by 2^-51.6 (rms) of the component's terms or less, as FP64 does.  In a Gaussian field the sum is 10 to 20 times
//     that line; S^dag S takes 1.5% longer for the sums.
// Measured against extended precision, the error of a component is that of the FP64 hops or below for links from
// 1 to exp(0.7 i H), for fields that fall by e^-0.7 per s and per chirality or by e^-1.2 per site, and for a colour
// 1 to 2^-30 of the others on diagonal links (1.1e-16 rms at every ratio, FP64 1.1e-16; without the tests 8e-16 at
// 2^-7 and 4e-10 at 2^-30).
// Non-finite values, sites below 2^-958 (both with exponent kFxHard) and sums near the ends of the exponent range take
// the FP64 stencil at once, so NaN and Inf propagate as in FP64.  (Components below 2^-1042 beside one above 2^-958 count as zero.)
//
// A link array holds nine (re1, re0, im1, im0) records per link, rows first, in the order of the FP64
// links ((p * 4 + mu) * Vh + h), and one exponent each behind them (kFxHard: a non-finite link).
//
// Storage of a field: the 16-byte chunks of the FP64 layout (SpF64), each a complex number as
// (re1, re0, im1, im0), and one int32 exponent per 5D site at ex[h * Ns + s].  Limbs of a sum of two
// spins fit 32 bits without a carry.
#pragma once

#include "kernels.cuh"

namespace odwf {

constexpr int kFxRaw = 1 << 28;      // added to the exponent of a site that keeps its FP64 bits
constexpr int kFxHard = 1 << 29;     // exponent of one that only FP64 arithmetic can take
constexpr int kFxBias = 1081;        // 1023 + 52 + 6: exponent of a site from its largest component's exponent field
constexpr int kFxZero = -(1 << 24);  // exponent of an all-zero site (never the largest)
constexpr int kFxSpread = 7;         // largest exponent range of a site's nonzero pairs of spins
constexpr unsigned kFxWeak = 3u << 20;  // smallest sum of |w|, high words of the stencil's 64-bit terms
constexpr int kFxMinField = 64;      // smallest biased exponent of a site's largest component

// (m << UP) >> (emax - exponent of d) of the 53-bit significand m of d.  A zero has
// exponent field 0 and is shifted out (shr.u64 clamps), emax being at least kFxMinField.
template <int UP>
__device__ __forceinline__ long long fx_magnitude(double d, int emax) {
    const int hi = __double2hiint(d);
    unsigned long long m =
        ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(d);
    const int down = emax - ((hi & 0x7fffffff) >> 20);
    asm("shr.u64 %0, %1, %2;" : "=l"(m) : "l"(m << UP), "r"(down));
    return (long long)m;
}
// and with d's sign
template <int UP>
__device__ __forceinline__ long long fx_from_double(double d, int emax) {
    const long long s = (long long)(__double2hiint(d) >> 31);
    return (fx_magnitude<UP>(d, emax) ^ s) - s;
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

// d in limbs, in units of 2^-58 of 2^(emax - 1023), rounded to nearest: twice the value in ones' complement
// rounds at no cost
__device__ __forceinline__ FxLimbs fx_round(double d, int emax) {
    const long long p = (fx_magnitude<7>(d, emax) ^ (long long)(__double2hiint(d) >> 31)) + 1;
    FxLimbs l;
    l.lo = (int)(unsigned)p >> 1;
    l.hi = (int)((p + (1ll << 31)) >> 32);
    return l;
}

// a complex number in FP64 bits into limbs
__device__ __forceinline__ int4 fx_convert(int4 q, int emax) {
    const FxLimbs re = fx_round(__hiloint2double(q.x, q.y), emax), im = fx_round(__hiloint2double(q.z, q.w), emax);
    return make_int4(re.hi, re.lo, im.hi, im.lo);
}
__device__ __forceinline__ bool fx_is_raw(int e) { return e >= kFxRaw / 2; }

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
