// Block fixed point for the FP64-accuracy hops.
//
// GB300 issues about 2 FP64 operations per clock and SM but 64 integer multiply-adds
// 32 x 32 + 64 -> 64 bits, so the SU(3) products of the hopping term, which are nearly all of its
// arithmetic, run in integers: a spinor of one 5D site is 24 signed integers with one exponent,
//     value = q 2^e,  |q| < 2^59,
// a link 18 integers with one exponent (|u| < 2^60 2^eu), both split into 31-bit limbs
//     q = q1 2^31 + q0,  -2^30 <= q0 < 2^30,
// and an output component sums q1 u1 and q1 u0 + q0 u1 in two 64-bit accumulators (q0 u0 is below
// the last unit kept).  The result resolves 2^-57 of the largest component of the neighbour, four
// bits beyond FP64's own rounding of it.  Components more than 2^kFxSpread below the largest of
// their 5D site, non-finite values and denormals keep their FP64 bits instead (exponent kFxRaw);
// sites that read such a neighbour take the FP64 arithmetic (fx_hop_slow), so nothing is lost on
// fields of extreme range and NaN and Inf propagate as in FP64.
//
// Storage of a field: the 16-byte chunks of the FP64 layout (SpF64) holding integers, and one
// int32 exponent per 5D site at ex[h * Ns + s].
#pragma once

#include "kernels.cuh"

namespace odwf {

constexpr int kFxRaw = 1 << 28;      // exponent marking FP64 bits
constexpr int kFxZero = -(1 << 24);  // exponent of an all-zero site (never the largest)
constexpr int kFxSpread = 32;        // largest exponent range of a site's nonzero components
constexpr int kFxMinField = 64;      // smallest biased exponent of a site's largest component

// (m << up) >> down of the 53-bit significand of d, down = emax - exponent of d, with d's sign
template <int UP>
__device__ __forceinline__ long long fx_from_double(double d, int emax) {
    const int hi = __double2hiint(d);
    const unsigned long long m =
        ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(d);
    const int down = min(emax - ((hi >> 20) & 0x7ff), 63);
    const long long q = (long long)((m << UP) >> down);
    const long long s = (long long)(hi >> 31);
    return (q ^ s) - s;
}

__device__ __forceinline__ void fx_store(void* base, int* ex, size_t h, int s, int ns, const double v[24]) {
    int mx = 0, mn = 0x7fffffff;
#pragma unroll
    for (int k = 0; k < 24; ++k) {
        const int hi = __double2hiint(v[k]) & 0x7fffffff;
        mx = max(mx, hi);
        mn = min(mn, (hi | __double2loint(v[k])) == 0 ? 0x7fffffff : hi);
    }
    const int emax = mx >> 20, emin = mn >> 20;
    longlong2* p = reinterpret_cast<longlong2*>(base);
    if (mn != 0x7fffffff && (emax == 0x7ff || emax < kFxMinField || emax - emin > kFxSpread)) {
        for (int k = 0; k < 12; ++k)
            p[chunk_off(h, k, 12, ns, s)] =
                make_longlong2(__double_as_longlong(v[2 * k]), __double_as_longlong(v[2 * k + 1]));
        ex[h * ns + s] = kFxRaw;
        return;
    }
    const int e = mn == 0x7fffffff ? 2046 : emax;  // an all-zero site: every significand shifted out
#pragma unroll
    for (int k = 0; k < 12; ++k)
        p[chunk_off(h, k, 12, ns, s)] = make_longlong2(fx_from_double<6>(v[2 * k], e), fx_from_double<6>(v[2 * k + 1], e));
    ex[h * ns + s] = mn == 0x7fffffff ? kFxZero : emax - 1081;  // 1023 + 52 + 6
}

// q 2^e for |q| < 2^63; the exponent is added to the converted double's where no result can leave
// the normal range
__device__ __forceinline__ double fx_to_double(long long q, int e) {
    const double d = __ll2double_rn(q);
    if (e < -1000 || e > 950) return q == 0 ? 0.0 : ldexp(d, max(e, -4000));
    return __hiloint2double(__double2hiint(d) + (q == 0 ? 0 : e << 20), __double2loint(d));
}

__device__ __forceinline__ void fx_load_double(const void* base, const int* ex, size_t h, int s, int ns, double v[24]) {
    const longlong2* p = reinterpret_cast<const longlong2*>(base);
    const int e = __ldg(ex + h * ns + s);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const longlong2 q = __ldg(p + chunk_off(h, k, 12, ns, s));
        v[2 * k] = e == kFxRaw ? __longlong_as_double(q.x) : fx_to_double(q.x, e);
        v[2 * k + 1] = e == kFxRaw ? __longlong_as_double(q.y) : fx_to_double(q.y, e);
    }
}

// One real of a half spinor as limbs
struct FxLimbs {
    int hi, lo;
};
__device__ __forceinline__ FxLimbs fx_split(long long q) {
    FxLimbs l;
    l.lo = (int)((unsigned)q << 1) >> 1;
    l.hi = (int)((q + (1ll << 30)) >> 31);
    return l;
}

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

}  // namespace odwf
