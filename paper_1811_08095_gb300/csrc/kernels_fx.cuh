// The FP64-accuracy hops in block fixed point (fx.cuh): the fused hop of kernels.cuh with its
// epilogues, two threads per 5D site (one spin of each chirality).  The input is a fixed-point field;
// a non-dagger hop reads (1 + L) psi, written by the kernel that produced it.
//
// What bounds it: three pipes at about half each, 5 blocks of 128 threads per SM overlapping phases.
// Per 5D site a hop takes 1728 integer multiply-adds at about 28 per clock and SM (62 clocks) and, at 2 per
// clock and SM, 120 to 190 FP64 operations (60 to 95 clocks): conversions of the 24 sums, 3 per real for
// a solve along s, 1 to 2 for a bidiagonal operator.  16^3x32x16, one system, the four hops of S^dag S:
// 0.42 / 0.53 / 0.44 / 0.54 ms at 52 to 72% FP64 pipe (FP64 stencil, 1334 to 1700 FP64 operations: 2.6 to
// 3.0 ms; one thread per 5D site at 168 registers: 0.57 / 0.69 / 0.61 / 0.49 ms; with the two threads in
// adjacent lanes a quarter warp touched four lines: 0.47 / 0.57 / 0.51 / 0.54 ms).  Four blocks per SM
// take 10% longer, six spill.  Warps that meet what fixed point cannot hold take other routes, fx_hop_conv and
// fx_hop_f64.
#pragma once

#include "fx.cuh"
#include "kernels.h"

namespace odwf {

constexpr int kFxThreads = 128;
constexpr int kFxMinBlocks = 5;
constexpr int kFxSite = 73;  // int4 words of a site's staged links (8 x 9, one more to spread the banks)

// Epilogue flags beyond kernels.cuh's: z and out formats are fixed by the epilogue
enum : int { FX_ZFX = 1 << 20, FX_OUTFX = 1 << 21, FX_OUTB = 1 << 22 };

// ---------------------------------------------------------------- fifth dimension
// Operators along s run as serial recurrences: the block's spinors are turned in shared memory so that
// a thread walks the Ns values of one real of one site.  M^-1 and 1 + L take the upper spins forward
// and the lower ones backward, M^-dag and L^dag the reverse, so every neighbour term is the value
// before in that order (the first takes the last one's, times -r).  The cyclic solve
//   w_i = inv_d t_i + al w_{i-1},  then  w_i += A_i fac w_last
// costs three FP64 operations per real against six of the log2 Ns shuffle scan (minv_apply), and the
// division of fac = -r / (1 + r A_last) is done once per block.
// B = omega (1 + L): the fixed-point input of a non-dagger hop is (1 + L) psi, and omega, which the
// hop does not mix along s, is folded into what follows the hop.
// The columns of the lower spins are stored backward, so that every column is walked the same way:
// forward for M^-1 and L, backward for the adjoints.
// Tables (Engine::init), Ns doubles each, for the upper spins and then, backward, for the lower: inv_d;
// al = -c_s / d_s and A, its running product in the order of the recurrence, for M^-1 and for M^-dag;
// omega inv_d; omega; d; e.
enum : int {
    C_ONEL = 1,       // t = v + L v
    C_BDAG = 2,       // t = omega v + L^dag (omega v)
    C_ZM = 4,         // t = M z + omega v
    C_ZMDAG = 8,      // t = M^dag z + sign B^dag v (with C_BDAG)
    C_MINV = 16,      // t = M^-1 t
    C_MINVDAG = 32,   // t = M^-dag t
    C_OMEGA = 64,     // C_MINV: of omega v
    C_OUTL = 128,     // then t = t + L t
    C_NEG = 256,      // C_ZMDAG: sign -1
};

__device__ __forceinline__ double fx_corner(const double* tab, double r, int ns) {
    return -r / fma(r, __ldg(tab + 3 * ns - 1), 1.0);  // A_last of M^-1 up: the same product for all four
}

template <int OPS>
__device__ __forceinline__ void fx_columns(double* buf, const double* zbuf, const double* tab, double r, double fac,
                                           int sites, int ns) {
    constexpr bool DAG = (OPS & (C_BDAG | C_MINVDAG | C_ZMDAG)) != 0;
    constexpr bool SOLVE = (OPS & (C_MINV | C_MINVDAG)) != 0;
    constexpr int step = DAG ? -1 : 1;
    const int first = DAG ? ns - 1 : 0, last = ns - 1 - first;
    const int ncol = sites * 24, nt = blockDim.x;
    // blocks start at different warps, so that the FP64 units of the four schedulers share what is not a
    // multiple of the block
    for (int c = (threadIdx.x + 32 * (blockIdx.x & 3)) & (nt - 1); c < ncol; c += nt) {
        const double* t9 = tab + ((c % 24) >= 12 ? 9 * ns : 0);
        const double *inv = t9 + ((OPS & C_OMEGA) ? 5 * ns : 0), *al = t9 + ((OPS & C_MINVDAG) ? 3 * ns : ns);
        const double *om = t9 + 6 * ns, *dd = t9 + 7 * ns, *ee = t9 + 8 * ns;
        double* p = buf + c * (ns + 1);
        const double* z = zbuf + c * (ns + 1);
        double w = 0.0, prev = 0.0, zprev = 0.0;
        if (OPS & C_ONEL) prev = -r * p[last];
        if (OPS & C_BDAG) prev = -r * (__ldg(om + last) * p[last]);
        if (OPS & C_ZM) zprev = -r * z[last];
        if (OPS & C_ZMDAG) zprev = -r * (__ldg(ee + last) * z[last]);
        int i = first;
#pragma unroll 4
        for (int n = 0; n < ns; ++n, i += step) {
            double t = p[i];
            if (OPS & (C_ONEL | C_BDAG)) {
                const double q = (OPS & C_BDAG) ? __ldg(om + i) * t : t;
                t = q + prev;
                prev = q;
            }
            if (OPS & C_ZM) {
                t = fma(__ldg(om + i), t, fma(__ldg(ee + i), zprev, __ldg(dd + i) * z[i]));
                zprev = z[i];
            }
            if (OPS & C_ZMDAG) {
                const double m = fma(__ldg(dd + i), z[i], zprev);
                t = (OPS & C_NEG) ? m - t : m + t;
                zprev = __ldg(ee + i) * z[i];
            }
            if (SOLVE) {
                w = fma(__ldg(al + i), w, __ldg(inv + i) * t);
                t = w;
            }
            p[i] = t;
        }
        if (SOLVE) {
            const double wc = fac * w;
            if (OPS & C_OUTL) prev = -r * fma(__ldg(al + ns + last), wc, w);
            i = first;
#pragma unroll 4
            for (int n = 0; n < ns; ++n, i += step) {
                const double t = fma(__ldg(al + ns + i), wc, p[i]);
                p[i] = (OPS & C_OUTL) ? t + prev : t;
                prev = t;
            }
        }
    }
}

// Thread of a block -> (s, a): a site's first Ns threads hold a = 0 in slot order and the next Ns a = 1, so
// that quarter warps read whole lines; the two halves of a 5D site exchange by a shuffle, so for Ns = 32
// (64 threads per site) they are adjacent lanes instead.
struct FxLane {
    int a, s, partner;  // partner: lane mask of the other half
    __device__ __forceinline__ FxLane(int t, int ns, int lg_ns) {
        const bool wide = ns == 32;
        const int slot = (wide ? t >> 1 : t) & (ns - 1), half = ns >> 1;
        a = (wide ? t : t >> lg_ns) & 1;
        partner = wide ? 1 : ns;
        s = slot < half ? 2 * slot : 2 * (slot - half) + 1;
    }
};

// A thread holds half a 5D site: spin a of the upper and of the lower pair, twelve reals in the order
// [up, down][colour][re, im].  Its columns of a site: 6 a + k (k < 6) and 12 + 6 a + (k - 6).
__device__ __forceinline__ int fx_col(int a, int k) { return k < 6 ? 6 * a + k : 6 + 6 * a + k; }
// its value of column k: mine[fx_at(a, s, k, ns)], the lower spins' columns backward
__device__ __forceinline__ int fx_at(int a, int s, int k, int ns) { return fx_col(a, k) * (ns + 1) + (k < 6 ? s : ns - 1 - s); }
__device__ __forceinline__ void fx_to_cols(const double v[12], double* mine, int a, int s, int ns) {
#pragma unroll
    for (int k = 0; k < 12; ++k) mine[fx_at(a, s, k, ns)] = v[k];
}
template <int OPS>
__device__ __forceinline__ void fx_turn(double v[12], double* buf, double* mine, const double* zbuf, const double* tab,
                                        double r, double fac, int a, int s, int sites, int ns) {
    fx_to_cols(v, mine, a, s, ns);
    __syncthreads();
    fx_columns<OPS>(buf, zbuf, tab, r, fac, sites, ns);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = mine[fx_at(a, s, k, ns)];
}

// chunk of colour c of the thread's upper (lo = 0) or lower (lo = 1) spin
__device__ __forceinline__ size_t fx_chunk(size_t h, int a, int lo, int c, int ns, int s) {
    return chunk_off(h, 6 * lo + 3 * a + c, 12, ns, s);
}
// FP64 fields in the internal chunk layout or, f.ext = 1 / 2, in the caller's: psi[s][site][spin][colour]
// over the even sites (site = h) or all sites (site of parity p).  The thread's six complex numbers are
// at q + lo (k / 3) + st (k % 3).
struct FxF64 {
    double2* q;
    int st, lo;
    __device__ __forceinline__ FxF64(const FieldRef& f, int sys, const Geom& g, int p, int h, int s, int a, int ns) {
        double2* base = reinterpret_cast<double2*>(f.d(sys));
        if (f.ext == 0) {
            q = base + fx_chunk((size_t)h, a, 0, 0, ns, s);
            st = ns;
            lo = 6 * ns;
        } else {
            size_t site = (size_t)h, n = (size_t)g.Vh;
            if (f.ext == 2) {  // lexicographic sites 2h and 2h + 1 have the two parities
                int c[4];
                site_coords(g, p, h, c);
                site = 2 * site + (c[0] & 1);
                n *= 2;
            }
            q = base + ((size_t)s * n + site) * 12 + 3 * a;
            st = 1;
            lo = 6;
        }
    }
    __device__ __forceinline__ void load(double v[12]) const {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 x = __ldg(q + (k / 3) * lo + (k % 3) * st);
            v[2 * k] = x.x;
            v[2 * k + 1] = x.y;
        }
    }
    __device__ __forceinline__ void store(const double v[12]) const {
#pragma unroll
        for (int k = 0; k < 6; ++k) q[(k / 3) * lo + (k % 3) * st] = make_double2(v[2 * k], v[2 * k + 1]);
    }
};
__device__ __forceinline__ void fx_load_fx(const void* base, const int* ex, size_t h, int s, int a, int ns, double v[12]) {
    const int4* p = reinterpret_cast<const int4*>(base);
    const int e = __ldg(ex + h * ns + s);
    int4 q[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) q[k] = __ldg(p + fx_chunk(h, a, k / 3, k % 3, ns, s));
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        v[2 * k] = fx_is_raw(e) ? __hiloint2double(q[k].x, q[k].y) : fx_to_double(fx_join(q[k].x, q[k].y), e);
        v[2 * k + 1] = fx_is_raw(e) ? __hiloint2double(q[k].z, q[k].w) : fx_to_double(fx_join(q[k].z, q[k].w), e);
    }
}
// Both threads of a 5D site call; `valid` is the same for both.
__device__ __forceinline__ void fx_store(void* base, int* ex, size_t h, const FxLane& t, int ns, bool valid,
                                         const double v[12]) {
    const int s = t.s, a = t.a;
    int mx = 0;
    unsigned mn = 0xffffffffu;  // smallest high word of a nonzero group (fx.cuh), less one
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int up = 0, dn = 0;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            up = max(up, __double2hiint(v[2 * c + k]) & 0x7fffffff);
            dn = max(dn, __double2hiint(v[6 + 2 * c + k]) & 0x7fffffff);
        }
        const int other = __shfl_xor_sync(0xffffffffu, dn, t.partner);
        mx = max(mx, max(up, dn));
        mn = min(mn, min((unsigned)(max(up, dn) - 1), (unsigned)(max(up, other) - 1)));
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, t.partner));
    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, t.partner));
    const int emax = mx >> 20, emin = (int)((mn + 1) >> 20);
    const bool wide = mn != 0xffffffffu && emax - emin > kFxSpread, odd = emax == 0x7ff || emax < kFxMinField;
    bool zero = false;
    if (__any_sync(0xffffffffu, odd)) {
        zero = odd;
        for (int k = 0; k < 12; ++k) zero = zero && v[k] == 0.0;
        zero = __shfl_xor_sync(0xffffffffu, (int)zero, t.partner) && zero;
    }
    if (!valid) return;
    int4* p = reinterpret_cast<int4*>(base);
    const bool hard = odd && !zero, raw = hard || (wide && !zero);
    const int e = zero ? 2046 : emax;  // an all-zero site: every significand shifted out
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        int4 q;
        if (raw) {
            q = make_int4(__double2hiint(v[2 * k]), __double2loint(v[2 * k]), __double2hiint(v[2 * k + 1]),
                          __double2loint(v[2 * k + 1]));
        } else {
            const FxLimbs re = fx_round(v[2 * k], e), im = fx_round(v[2 * k + 1], e);
            q = make_int4(re.hi, re.lo, im.hi, im.lo);
        }
        p[fx_chunk(h, a, k / 3, k % 3, ns, s)] = q;
    }
    if (a == 0) ex[h * ns + s] = hard ? kFxHard : zero ? kFxZero : emax - kFxBias + (raw ? kFxRaw : 0);
}

// ---------------------------------------------------------------- the stencil
// One direction for spin a of the half spinor h = v^up + sg G v^dn: h_a takes the lower spin 1 - a for
// mu = 0, 1 and a for mu = 2, 3, with the factors (chiral basis)
//   mu 0: -i (both),  mu 1: -1 (a = 0), +1 (a = 1),  mu 2: -i (a = 0), +i (a = 1),  mu 3: 1 (both),
// and w_a = U h_a returns to that lower spin with the conjugate factor.  Where the factor's sign differs
// between the two threads of a site, thread 1 takes the opposite direction (whose sg has the other
// sign), so both run the same code.  acc: upper spin a, lower spin 1 - a (mu 0, 1), lower spin a (mu 2, 3).
// size: |w| of each colour, leading words (see kFxWeak), the real part of one direction and the imaginary part of
// the other, so that neither real nor imaginary fields look small.
// CONV: a neighbour with en >= kFxRaw / 2 holds FP64 bits.
template <int MU, bool PLUS, bool CONV>
__device__ __forceinline__ void fx_dir(const int4* __restrict__ up, const int4* __restrict__ dn, int ns, const int4* U,
                                       int sh, long long acc[18], unsigned size[3], int en = 0) {
    FxLimbs h[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        int4 u = __ldg(up + c * ns), d = __ldg(dn + c * ns);
        if (CONV && fx_is_raw(en)) {
            u = fx_convert(u, en - kFxRaw + kFxBias);
            d = fx_convert(d, en - kFxRaw + kFxBias);
        }
        // G d as (re, im): -i d = (im, -re) for mu 0, 2; -d for mu 1; d for mu 3
        const FxLimbs gr = (MU == 0 || MU == 2) ? FxLimbs{d.z, d.w} : FxLimbs{d.x, d.y};
        const FxLimbs gi = (MU == 0 || MU == 2) ? FxLimbs{d.x, d.y} : FxLimbs{d.z, d.w};
        constexpr bool nr = (MU == 1) == PLUS;              // minus sign of the real part
        constexpr bool ni = (MU == 3) != PLUS;              // and of the imaginary part
        h[c][0].hi = nr ? u.x - gr.hi : u.x + gr.hi;
        h[c][0].lo = nr ? u.y - gr.lo : u.y + gr.lo;
        h[c][1].hi = ni ? u.z - gi.hi : u.z + gi.hi;
        h[c][1].lo = ni ? u.w - gi.lo : u.w + gi.lo;
    }
    long long* lower = acc + (MU < 2 ? 6 : 12);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        // leading sums, and the cross sums (the first rounded) in two shorter chains
        long long A[2] = {0, 0}, B[2] = {1ll << 30, 1ll << 30}, C[2] = {0, 0};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 u = U[3 * i + b];
            const int m1 = fx_neg(u.z), m0 = fx_neg(u.w);
            const FxLimbs x = h[b][0], y = h[b][1];
            A[0] = fx_mad(u.x, x.hi, fx_mad(m1, y.hi, A[0]));
            A[1] = fx_mad(u.x, y.hi, fx_mad(u.z, x.hi, A[1]));
            B[0] = fx_mad(u.x, x.lo, fx_mad(u.y, x.hi, B[0]));
            C[0] = fx_mad(m1, y.lo, fx_mad(m0, y.hi, C[0]));
            B[1] = fx_mad(u.x, y.lo, fx_mad(u.y, y.hi, B[1]));
            C[1] = fx_mad(u.z, x.lo, fx_mad(u.w, x.hi, C[1]));
        }
        const long long wr = (A[0] + ((B[0] + C[0]) >> 31)) >> sh, wi = (A[1] + ((B[1] + C[1]) >> 31)) >> sh;
        acc[2 * i] += wr;
        acc[2 * i + 1] += wi;
        size[i] += (unsigned)abs((int)((PLUS ? wr : wi) >> 32));
        // sg G^dag w: i w for mu 0, 2; -w for mu 1; w for mu 3
        if (MU == 0 || MU == 2) {
            lower[2 * i] = PLUS ? lower[2 * i] - wi : lower[2 * i] + wi;
            lower[2 * i + 1] = PLUS ? lower[2 * i + 1] + wr : lower[2 * i + 1] - wr;
        } else {
            constexpr bool n = (MU == 1) == PLUS;
            lower[2 * i] = n ? lower[2 * i] - wr : lower[2 * i] + wr;
            lower[2 * i + 1] = n ? lower[2 * i + 1] - wi : lower[2 * i + 1] + wi;
        }
    }
}

// d with its sign bit flipped where `mask` has bit 31
__device__ __forceinline__ double fx_flip(double d, unsigned mask) {
    return __hiloint2double((int)((unsigned)__double2hiint(d) ^ mask), __double2loint(d));
}

// fx_dir in FP64: the neighbour's stored exponent e, U the FP64 link, taken adjoint for a backward
// hop and negated where `minus`
template <int MU, bool PLUS>
__device__ __forceinline__ void fx_dir_f64(const int4* __restrict__ up, const int4* __restrict__ dn, int e, int ns,
                                           const double2* __restrict__ U, bool back, bool minus, double acc[18]) {
    double h[3][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int4 u = __ldg(up + c * ns), d = __ldg(dn + c * ns);
        double ur, ui, dr, di;
        if (fx_is_raw(e)) {
            ur = __hiloint2double(u.x, u.y);
            ui = __hiloint2double(u.z, u.w);
            dr = __hiloint2double(d.x, d.y);
            di = __hiloint2double(d.z, d.w);
        } else {
            ur = fx_to_double(fx_join(u.x, u.y), e);
            ui = fx_to_double(fx_join(u.z, u.w), e);
            dr = fx_to_double(fx_join(d.x, d.y), e);
            di = fx_to_double(fx_join(d.z, d.w), e);
        }
        constexpr bool nr = (MU == 1) == PLUS, ni = (MU == 3) != PLUS, turn = MU == 0 || MU == 2;  // as fx_dir
        h[c][0] = nr ? ur - (turn ? di : dr) : ur + (turn ? di : dr);
        h[c][1] = ni ? ui - (turn ? dr : di) : ui + (turn ? dr : di);
    }
    double* lower = acc + (MU < 2 ? 6 : 12);
    const unsigned fr = minus ? 0x80000000u : 0u, fi = fr ^ (back ? 0x80000000u : 0u);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double wr = 0.0, wi = 0.0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double2 u = __ldg(U + (back ? 3 * b + i : 3 * i + b));
            const double ur = fx_flip(u.x, fr), ui = fx_flip(u.y, fi);
            wr = fma(ur, h[b][0], wr);
            wr = fma(-ui, h[b][1], wr);
            wi = fma(ur, h[b][1], wi);
            wi = fma(ui, h[b][0], wi);
        }
        acc[2 * i] += wr;
        acc[2 * i + 1] += wi;
        if (MU == 0 || MU == 2) {
            lower[2 * i] = PLUS ? lower[2 * i] - wi : lower[2 * i] + wi;
            lower[2 * i + 1] = PLUS ? lower[2 * i + 1] + wr : lower[2 * i + 1] - wr;
        } else {
            constexpr bool n = (MU == 1) == PLUS;
            lower[2 * i] = n ? lower[2 * i] - wr : lower[2 * i] + wr;
            lower[2 * i + 1] = n ? lower[2 * i + 1] - wi : lower[2 * i + 1] + wi;
        }
    }
}

// index of the link of direction j at site h (parity p_out) with neighbour hn
__device__ __forceinline__ size_t fx_link_index(const HopParams<double>& P, int j, int h, int hn) {
    return (j & 1) ? (size_t)((1 - P.p_out) * 4 + (j >> 1)) * P.g.Vh + hn : (size_t)(P.p_out * 4 + (j >> 1)) * P.g.Vh + h;
}

// The fixed-point stencil for warps that meet neighbours with FP64 bits: those are converted where they are read.
// Such sites are rare in most fields, and a warp that went to the FP64 stencil for one finished 4 us after the
// others, which a small launch waits for: FP64 CG on 8^3x16x8 52.3 -> 49.8 ms, S^dag S on 16^3x32x16 of a field
// with one colour 1e-15 of the others on rough links 3.8 -> 2.5 ms.
template <bool DAG>
static __device__ __noinline__ void fx_hop_conv(const HopParams<double>& P, const int4* in, const int* ex, int h, int s, int a,
                                                const int4* my_links, int M, long long* acc_out, unsigned* size_out) {
    const int ns = P.ns, cross = (9 - 6 * a) * ns, same = 6 * ns;
    const int* nb = P.nbr + ((size_t)P.p_out * P.g.Vh + h) * 8;
    long long acc[18];
    unsigned size[2][3];
#pragma unroll
    for (int k = 0; k < 18; ++k) acc[k] = 0;
#pragma unroll
    for (int k = 0; k < 6; ++k) size[k / 3][k % 3] = 0;
#define ODWF_FX_DIRC(MU_, DIR_)                                                                                      \
    {                                                                                                                \
        const int j_ = (MU_ == 1 || MU_ == 2) ? ((2 * MU_ + DIR_) ^ a) : 2 * MU_ + DIR_;                             \
        const int n_ = checked_index(__ldg(nb + j_) & 0x7fffffff, P.g.Vh, P.bounds_flag, kBoundsNeighbour);          \
        const int en_ = __ldg(ex + (size_t)n_ * ns + s), eu_ = __ldg(P.link_ex + fx_link_index(P, j_, h, n_));       \
        const int4* p_ = in + (size_t)n_ * (12 * ns);                                                                \
        fx_dir<MU_, (DIR_ == 0) == DAG, true>(p_, p_ + (MU_ < 2 ? cross : same), ns, my_links + 9 * j_,               \
                                              min(M - (en_ - (fx_is_raw(en_) ? kFxRaw : 0) + eu_), 63), acc,         \
                                              size[MU_ / 2], en_);                                                   \
    }
    ODWF_FX_DIRC(0, 0) ODWF_FX_DIRC(0, 1)
    ODWF_FX_DIRC(1, 0) ODWF_FX_DIRC(1, 1)
    ODWF_FX_DIRC(2, 0) ODWF_FX_DIRC(2, 1)
    ODWF_FX_DIRC(3, 0) ODWF_FX_DIRC(3, 1)
#undef ODWF_FX_DIRC
#pragma unroll
    for (int k = 0; k < 18; ++k) acc_out[k] = acc[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) size_out[k] = size[k / 3][k % 3];
}

// The stencil in FP64, for warps that meet a neighbour or a link outside the fixed-point range or whose sums
// hold a small one: half a 5D site per thread as the fixed-point one, 530 FP64 operations each with the
// conversions.  S^dag S on 16^3x32x16: fields of which every warp runs both stencils 8.7 ms (a small colour) or 9.8
// (a zero colour on unit links), FP64 hops throughout 12.7, others 1.97.  All lanes of the warp call.
template <bool DAG>
static __device__ __noinline__ void fx_hop_f64(const HopParams<double>& P, const int4* in, const int* ex, int h, int s, int a,
                                               int partner, double* v) {
    const int ns = P.ns, cross = (9 - 6 * a) * ns, same = 6 * ns;
    const int* nb = P.nbr + ((size_t)P.p_out * P.g.Vh + h) * 8;
    double acc[18];
#pragma unroll
    for (int k = 0; k < 18; ++k) acc[k] = 0.0;
#define ODWF_FX_DIR64(MU_, DIR_)                                                                                     \
    {                                                                                                                \
        const int j_ = (MU_ == 1 || MU_ == 2) ? ((2 * MU_ + DIR_) ^ a) : 2 * MU_ + DIR_;                             \
        const int raw_ = __ldg(nb + j_), n_ = checked_index(raw_ & 0x7fffffff, P.g.Vh, P.bounds_flag, kBoundsNeighbour); \
        const int4* p_ = in + (size_t)n_ * (12 * ns);                                                                \
        fx_dir_f64<MU_, (DIR_ == 0) == DAG>(p_, p_ + (MU_ < 2 ? cross : same), __ldg(ex + (size_t)n_ * ns + s), ns,   \
                                            static_cast<const double2*>(P.links_d) + fx_link_index(P, j_, h, n_) * 9, \
                                            j_ & 1, raw_ >= 0, acc);                                                 \
    }
    ODWF_FX_DIR64(0, 0) ODWF_FX_DIR64(0, 1)
    ODWF_FX_DIR64(1, 0) ODWF_FX_DIR64(1, 1)
    ODWF_FX_DIR64(2, 0) ODWF_FX_DIR64(2, 1)
    ODWF_FX_DIR64(3, 0) ODWF_FX_DIR64(3, 1)
#undef ODWF_FX_DIR64
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        v[k] = 0.5 * acc[k];
        v[6 + k] = 0.5 * (acc[12 + k] + __shfl_xor_sync(0xffffffffu, acc[6 + k], partner));
    }
}

template <int F>
__global__ void __launch_bounds__(kFxThreads, kFxMinBlocks) hop_fx_kernel(const __grid_constant__ HopParams<double> P) {
    constexpr bool DAG = (F & F_DAG) != 0;
    constexpr int ZOP = (F & F_ZOP_MASK) >> F_ZOP_SHIFT;
    constexpr int HOPOP = (F & F_HOP_MASK) >> F_HOP_SHIFT;
    constexpr bool NEG = (F & F_NEG) != 0;
    constexpr int POST = (F & F_POST_MASK) >> F_POST_SHIFT;
    constexpr bool NORM = (F & F_NORM) != 0;
    constexpr bool CG = (F & F_CG) != 0;
    constexpr bool RESID = (F & F_RESID) != 0;
    constexpr int FIN = (F & F_FIN_MASK) >> F_FIN_SHIFT;
    constexpr bool REDUCE = NORM || CG || RESID;
    constexpr bool ZM = ZOP == ZOP_M || ZOP == ZOP_MDAG;  // z through M in the column pass
    extern __shared__ __align__(16) int4 s_links[];

    const int sys = blockIdx.y + P.sys_base;
    if (P.gate && P.st[sys].status != P.need_status) return;  // uniform over the block
    if (P.prof_count && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(P.prof_count, 1ull);

    const int ns = P.ns, g2 = P.lg_ns + 1;  // 2 Ns threads per site
    const FxLane t(threadIdx.x, ns, P.lg_ns);
    const int a = t.a, s = t.s;
    const size_t gi = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t hh = gi >> g2;
    const bool valid = hh < (size_t)P.g.Vh;
    const int h = valid ? (int)hh : 0;  // threads past the last site read site 0's neighbours and store nothing
    const int site = threadIdx.x >> g2, sites = blockDim.x >> g2;
    const double r = P.r_sys[sys];

    int nb[8];
    {
        const int4* tp = reinterpret_cast<const int4*>(P.nbr + ((size_t)P.p_out * P.g.Vh + h) * 8);
        const int4 n0 = __ldg(tp), n1 = __ldg(tp + 1);
        const int raw[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) nb[j] = checked_index(raw[j] & 0x7fffffff, P.g.Vh, P.bounds_flag, kBoundsNeighbour);
    }
    // the site's eight links into shared memory, 72 elements over its 2 Ns threads: the adjoint for a
    // backward hop, negated (the -1 of -1/2 W) except across the antiperiodic boundary
    int4* my_links = s_links + site * kFxSite;
    const int4* lk = reinterpret_cast<const int4*>(P.links);
    for (int i = threadIdx.x & (2 * ns - 1); i < 72; i += 2 * ns) {
        const int d = i / 9, k = i - 9 * d;
        const int raw = __ldg(P.nbr + ((size_t)P.p_out * P.g.Vh + h) * 8 + d);
        const bool back = d & 1;
        const size_t idx = fx_link_index(P, d, h, checked_index(raw & 0x7fffffff, P.g.Vh, P.bounds_flag, kBoundsNeighbour));
        int4 u = __ldg(lk + idx * 9 + k);
        if (raw >= 0) u = make_int4(-u.x, -u.y, -u.z, -u.w);
        if (back) {
            u.z = -u.z;
            u.w = -u.w;
        }
        my_links[9 * d + (back ? 3 * (k % 3) + k / 3 : k)] = u;
    }

    const int4* in = reinterpret_cast<const int4*>(P.in.d(sys)) + chunk_slot(s, ns) + 3 * a * ns;
    const int* ex = reinterpret_cast<const int*>(P.in.n(sys));
    int e[8], M = kFxZero;
    bool slow = false, conv = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int en = __ldg(ex + (size_t)nb[j] * ns + s), eu = __ldg(P.link_ex + fx_link_index(P, j, h, nb[j]));
        slow |= max(en, eu) >= kFxHard;
        conv |= fx_is_raw(en);
        e[j] = en - (fx_is_raw(en) ? kFxRaw : 0) + eu;
        M = max(M, e[j]);
    }
    __syncthreads();  // a site's threads may lie in two warps (Ns = 32)
    double v[12];
    bool redo = __any_sync(0xffffffffu, slow || ((M < kFxMinExp || M >= kFxMaxExp) && M > kFxZero / 2));
    if (!redo) {
        long long acc[18];
        unsigned size[2][3];  // mu = 0, 1 and mu = 2, 3
#pragma unroll
        for (int k = 0; k < 18; ++k) acc[k] = 0;
#pragma unroll
        for (int k = 0; k < 6; ++k) size[k / 3][k % 3] = 0;
        if (__any_sync(0xffffffffu, conv)) {
            long long t_acc[18];
            unsigned t_size[6];
            fx_hop_conv<DAG>(P, in, ex, h, s, a, my_links, M, t_acc, t_size);
#pragma unroll
            for (int k = 0; k < 18; ++k) acc[k] = t_acc[k];
#pragma unroll
            for (int k = 0; k < 6; ++k) size[k / 3][k % 3] = t_size[k];
        } else {
            const int cross = (9 - 6 * a) * ns, same = 6 * ns;  // from upper spin a to lower spin 1 - a, to lower spin a
#define ODWF_FX_DIR(MU_, DIR_)                                                                                      \
    {                                                                                                               \
        constexpr int j_ = 2 * MU_ + DIR_;                                                                          \
        constexpr bool swap_ = MU_ == 1 || MU_ == 2; /* thread 1 takes the opposite direction */                    \
        const int n_ = swap_ && a ? nb[j_ ^ 1] : nb[j_], e_ = swap_ && a ? e[j_ ^ 1] : e[j_];                       \
        const int4* p_ = in + (size_t)n_ * (12 * ns);                                                               \
        fx_dir<MU_, (DIR_ == 0) == DAG, false>(p_, p_ + (MU_ < 2 ? cross : same), ns,                               \
                                               my_links + 9 * (swap_ ? (j_ ^ a) : j_), min(M - e_, 63), acc,        \
                                               size[MU_ / 2]);                                                      \
    }
            ODWF_FX_DIR(0, 0) ODWF_FX_DIR(0, 1)
            ODWF_FX_DIR(1, 0) ODWF_FX_DIR(1, 1)
            ODWF_FX_DIR(2, 0) ODWF_FX_DIR(2, 1)
            ODWF_FX_DIR(3, 0) ODWF_FX_DIR(3, 1)
#undef ODWF_FX_DIR
        }
        // -1/2 W psi (or -1/2 W^dag psi) = acc 2^(M + 2) / 2, the lower spin with the other thread's part
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            v[k] = fx_to_double(acc[k], M + 1);
            v[6 + k] = fx_to_double(acc[12 + k] + __shfl_xor_sync(0xffffffffu, acc[6 + k], t.partner), M + 1);
        }
        unsigned least = 0xffffffffu;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const unsigned other = __shfl_xor_sync(0xffffffffu, size[0][c], t.partner);
            least = min(least, size[1][c] + min(size[0][c], other));
        }
        redo = __any_sync(0xffffffffu, least < kFxWeak && M > kFxZero / 2);
    }
    if (redo) {
        double y[12];
        fx_hop_f64<DAG>(P, in, ex, h, s, a, t.partner, y);
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = y[k];
    }

    // the links are read: their shared memory now holds the columns of fx_columns
    double* buf = reinterpret_cast<double*>(s_links);
    double* mine = buf + site * 24 * (ns + 1);
    __shared__ double s_fac;
    if ((HOPOP != OP_ID || POST != 0) && threadIdx.x == 0) s_fac = fx_corner(P.tab5, r, ns);
    __syncthreads();
    const double fac = s_fac;

    double z[12];
    if (ZOP != ZOP_NONE) {
        if (F & FX_ZFX) fx_load_fx(P.z.d(sys), reinterpret_cast<const int*>(P.z.n(sys)), (size_t)h, s, a, ns, z);
        else FxF64(P.z, sys, P.g, P.p_out, h, s, a, ns).load(z);
    }
    if (ZM) {
        double* zbuf = buf + sites * 24 * (ns + 1);
        fx_to_cols(z, zbuf + (mine - buf), a, s, ns);
        if (DAG) fx_turn<C_BDAG | C_ZMDAG | (NEG ? C_NEG : 0)>(v, buf, mine, zbuf, P.tab5, r, fac, a, s, sites, ns);
        else fx_turn<C_ZM>(v, buf, mine, zbuf, P.tab5, r, fac, a, s, sites, ns);
    } else if (DAG) {
        fx_turn<C_BDAG | (HOPOP == OP_MINVDAG ? C_MINVDAG : 0)>(v, buf, mine, buf, P.tab5, r, fac, a, s, sites, ns);
    } else if (HOPOP == OP_MINV) {
        fx_turn<C_MINV | C_OMEGA | ((F & FX_OUTB) ? C_OUTL : 0)>(v, buf, mine, buf, P.tab5, r, fac, a, s, sites, ns);
    } else {
        const double om = __ldg(P.tab5 + 6 * ns + s);
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] *= om;
    }
    if (ZOP == ZOP_ID) {
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = NEG ? z[k] - v[k] : z[k] + v[k];
    }
    double nrm = 0.0;
    if (NORM && valid) {
#pragma unroll
        for (int k = 0; k < 12; ++k) nrm = fma(v[k], v[k], nrm);
    }
    if (POST != 0) {
        __syncthreads();  // the first pass's columns have been read
        fx_turn<POST == OP_MINV ? C_MINV : C_MINVDAG>(v, buf, mine, buf, P.tab5, r, fac, a, s, sites, ns);
    }

    if (CG && valid) {
        // v = A p;  r <- r - alpha A p;  x <- x + alpha p;  nrm = |r|^2
        const double alpha = P.st[sys].alpha;
        double w[12];
        const FxF64 cr(P.cg_r, sys, P.g, 0, h, s, a, ns), cx(P.cg_x, sys, P.g, 0, h, s, a, ns);
        cr.load(w);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            w[k] = fma(-alpha, v[k], w[k]);
            nrm = fma(w[k], w[k], nrm);
        }
        cr.store(w);
        cx.load(w);
        FxF64(P.cg_p, sys, P.g, 0, h, s, a, ns).load(v);
#pragma unroll
        for (int k = 0; k < 12; ++k) w[k] = fma(alpha, v[k], w[k]);
        cx.store(w);
    }
    if (RESID) {
        double b[12];
        FxF64(P.b, sys, P.g, 0, h, s, a, ns).load(b);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            v[k] = b[k] - v[k];
            if (valid) nrm = fma(v[k], v[k], nrm);
        }
    }
    if (F & FX_OUTFX) fx_store(P.out.d(sys), reinterpret_cast<int*>(P.out.n(sys)), (size_t)h, t, ns, valid, v);
    else if (!CG && valid) FxF64(P.out, sys, P.g, P.p_out, h, s, a, ns).store(v);
    if (REDUCE) reduce_and_finalize(nrm, P.partials, P.counters, P.st, sys, FIN, P.part_stride);
}

// Threads per block: 128 (64 5D sites), or 64 while all blocks of 128 would be resident at once (5 on each
// of 152 SMs), when a smaller block is a shorter chain.  FP64 CG on 8^3x16x8 (32768 sites) 55.4 -> 51.0 ms,
// D on 6x10x4x14x16 (26880) 62.4 -> 65.6 us; at 1 M sites 64 threads take 5% longer.
inline int fx_threads(size_t n5) { return 2 * n5 < (size_t)kFxThreads * 760 ? 64 : kFxThreads; }
// dynamic shared memory of a block: its staged links or `bufs` column buffers, whichever is larger
inline size_t fx_smem(int bs, int ns, int bufs, bool links) {
    const size_t sites = (size_t)bs / (2 * ns), cols = bufs * sites * 24 * (ns + 1) * sizeof(double);
    const size_t lk = links ? sites * kFxSite * sizeof(int4) : 0;
    return cols > lk ? cols : lk;
}

template <int F>
cudaError_t hop_fx(const HopParams<double>& P, int nsys, cudaStream_t st) {
    constexpr int ZOP = (F & F_ZOP_MASK) >> F_ZOP_SHIFT;
    const size_t n = (size_t)P.g.Vh * P.ns;
    const int bs = fx_threads(n);
    note_launch();
    hop_fx_kernel<F><<<dim3(blocks_for(2 * n, bs), nsys), bs,
                       fx_smem(bs, P.ns, ZOP == ZOP_M || ZOP == ZOP_MDAG ? 2 : 1, true), st>>>(P);
    return cudaGetLastError();
}

}  // namespace odwf
