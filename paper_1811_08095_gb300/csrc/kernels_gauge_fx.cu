// Wilson gauge force and action (definitions in kernels_md.cu) in fixed point: FP64 accuracy on the
// integer pipe.
//
// Thirteen SU(3) products per link are 1400 FP64 operations on a pipe of 2 per clock and SM; as 31-bit
// limbs (fx.cuh) they are 4212 integer multiply-adds at about 28 per clock and SM.  Entries of SU(3) matrices
// are at most 1, so every link has 60 fraction bits and no exponent; products are kept to 2^-58, staples
// and U Sigma to 2^-56, against 2^-53 of each FP64 operation.  Fields whose rows or columns are not of
// unit length to 2^-16 (the entry points take any matrices) raise a flag in the pass that splits the
// links, and the FP64 kernel of kernels_md.cu runs instead; both are launched and one of them returns at
// once.
//
// Where the links have one large entry per row (near the unit field, or an abelian one) the force comes from
// the small entries, whose products FP64 keeps to 2^-53 of themselves and limbs to 2^-58 of 1.  With links
// exp(i eps H) both err by 1.4e-16 of the force (rms, FP64 at every eps) at eps = 0.035, where the off-diagonal
// entries are about 2^-6; the limbs by 1.0e-16 at 0.25, 2.1e-16 at 0.02 and 3.7e-15 at 0.001.  The pass that
// splits the links marks those whose other six entries are below 2^-6; the FP64 kernel takes the marked ones
// and this one the others, each adding to its block's sum.  From one marked link in 64 the whole field goes to
// the FP64 kernel, since a warp that holds one takes as long there as a full one.  16^3x32: 0.50 ms at eps =
// 0.25, 0.58 at 0.1, 1.29 at 0.05, 2.07 from 0.03 down.
//
// Splitting the links where they are used instead of in a pass before gives the same bits and needs no
// workspace for the limbs, but takes twice as long (16^3x32 1.03 ms; 8^4, where the chip is not full, 88 us
// against 57): for calls that would have to allocate it first, see Engine::gauge_force.
//
// 16^3x32, action and force: 2.04 ms in FP64, 0.50 ms here (split 27 us, force 0.44 ms); bound by
// the latency of the integer chains with the 8 warps per SM that 252 registers leave (three blocks per
// SM spill 300 bytes: 0.50 ms, four 0.56 ms).
//
// Bounds: entries of a product of unit-row matrices are at most 1, of a staple sqrt(3), of six 10.4
// (limbs allow 16 at 58 fraction bits); by Cauchy and row sums of |re| + |im| of at most sqrt 6 times
// the row's length, the cross sums stay below 2^62.6.
#include "fx.cuh"
#include "kernels.h"

namespace odwf {

namespace {

constexpr int kBSG = 128;
constexpr int kWeakEntry = 0x3f900000;  // high word of 2^-6

// Element k of a link as (re1, re0, im1, im0).  Limbs: split by a pass before, element k of link (mu, s) at
// p[(k * 4 + mu) * V + s].  Direct: the caller's FP64 links, split where they are used.
struct FxM {
    int4 e[9];
};

__device__ __forceinline__ int4 fx_split_entry(double2 u) {  // |u| < 2 to 60 fraction bits
    const FxLimbs r = fx_split(fx_from_double<8>(u.x, 1023)), q = fx_split(fx_from_double<8>(u.y, 1023));
    return make_int4(r.hi, r.lo, q.hi, q.lo);
}

// loads are issued where they stand: rows are read again from L1 rather than held in registers
struct Limbs {
    const int4* p;
    size_t st;  // between the elements of a link
    __device__ __forceinline__ Limbs(const void* links, size_t V, int mu, size_t s)
        : p((const int4*)links + (size_t)mu * V + s), st(4 * V) {}
    __device__ __forceinline__ int4 at(int k) const {
        int4 v;
        asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p + k * st));
        return v;
    }
};
struct Direct {
    const double2* p;
    __device__ __forceinline__ Direct(const void* links, size_t V, int mu, size_t s)
        : p((const double2*)links + ((size_t)mu * V + s) * 9) {}
    __device__ __forceinline__ int4 at(int k) const {
        double2 v;
        asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p + k));
        return fx_split_entry(v);
    }
};

// (A, B) += x y of the limb pairs: A the product of the leading limbs, B the cross terms
__device__ __forceinline__ void fx_macc(int x1, int x0, int y1, int y0, long long& A, long long& B) {
    A = fx_mad(x1, y1, A);
    B = fx_mad(x1, y0, fx_mad(x0, y1, B));
}
// limbs with a nonnegative lower one (two instructions; the product of two lower limbs, which is left
// out, is then up to a unit of the sum kept instead of a quarter)
__device__ __forceinline__ void fx_limbs(long long q, int& hi, int& lo) {
    hi = (int)(q >> 31);
    // opaque: known to be nonnegative, its products with signed limbs would become 64 x 64-bit ones
    asm("and.b32 %0, %1, 0x7fffffff;" : "=r"(lo) : "r"((int)q));
}

// sum_k x_k y_k rounded to 62 fraction bits less than the factors have together; CX, CY: conjugate that
// factor
template <bool CX, bool CY>
__device__ __forceinline__ void fx_dot3(const int4 x[3], const int4 y0, const int4 y1, const int4 y2, long long& re,
                                        long long& im) {
    long long A = 0, B = 0, C = 0, D = 0;
    const int4 ys[3] = {y0, y1, y2};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int4 a = x[k], y = ys[k];
        // re = ar br - ai bi, im = ar bi + ai br with the signs of conjugated imaginary parts: n is the
        // negated imaginary part of the first factor, used where a minus sign is left
        const int n1 = fx_neg(a.z), n0 = fx_neg(a.w);
        const bool minus = CX == CY;  // sign of ai bi in re
        fx_macc(a.x, a.y, y.x, y.y, A, B);
        fx_macc(minus ? n1 : a.z, minus ? n0 : a.w, y.z, y.w, A, B);
        // im: the sign of bi is CY's, of ai CX's; with CY the sum is accumulated negated and turned below
        fx_macc(a.x, a.y, y.z, y.w, C, D);
        fx_macc(minus ? a.z : n1, minus ? a.w : n0, y.x, y.y, C, D);
    }
    re = A + (B >> 31);
    im = C + (D >> 31);
    if (CY) im = -im;
}

// One staple, row by row: T_i = a_i B^dag with a_i row i of A (LOWER: of A^dag), 58 fraction bits, and
// S_i += T_i C^dag (LOWER: T_i C), 56 fraction bits.  Only a row of A and of T is held at a time.
template <bool LOWER, class SRC>
__device__ __forceinline__ void fx_staple(const SRC A, const SRC B, const SRC C, long long S[18]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        int4 a[3], t[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) a[k] = A.at(LOWER ? 3 * k + i : 3 * i + k);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long re, im;
            fx_dot3<LOWER, true>(a, B.at(3 * j), B.at(3 * j + 1), B.at(3 * j + 2), re, im);
            fx_limbs(re, t[j].x, t[j].y);
            fx_limbs(im, t[j].z, t[j].w);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long re, im;
            constexpr int sk = LOWER ? 3 : 1;
            const int q = LOWER ? j : 3 * j;
            fx_dot3<false, !LOWER>(t, C.at(q), C.at(q + sk), C.at(q + 2 * sk), re, im);
            S[2 * (3 * i + j)] += re;
            S[2 * (3 * i + j) + 1] += im;
        }
    }
}

// Links (external layout, n = 4 V of them) into limbs (unless out is null) and their marks; flags->bad for a
// link outside the fixed-point range
__global__ void __launch_bounds__(kBSG) split_links_kernel(const double2* __restrict__ U, size_t n, int4* __restrict__ out,
                                                           GaugeFlags* __restrict__ flags, unsigned char* __restrict__ weak) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    float row[3] = {0.f, 0.f, 0.f}, col[3] = {0.f, 0.f, 0.f};
    bool big = false;
    int large = 0;  // entries of 2^-6 and more: three in a matrix with one such entry per row
    if (i < n) {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double2 u = U[i * 9 + k];
            const int m = max(__double2hiint(u.x) & 0x7fffffff, __double2hiint(u.y) & 0x7fffffff);
            big = big || m >= 0x3ff80000;  // 1.5, and non-finite values
            large += m >= kWeakEntry;
            const int4 q = fx_split_entry(u);
            if (out) out[(size_t)k * n + i] = q;
            const float a = (float)q.x * 0x1p-29f, b = (float)q.z * 0x1p-29f;
            const float t = fmaf(a, a, b * b);
            row[k / 3] += t;
            col[k % 3] += t;
        }
        float worst = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) worst = fmaxf(worst, fmaxf(fabsf(row[k] - 1.f), fabsf(col[k] - 1.f)));
        if (big || !(worst < 0x1p-15f)) atomicOr(&flags->bad, 1);
        weak[i] = large <= 3;
    }
    const unsigned marked = __ballot_sync(0xffffffffu, i < n && large <= 3);
    if ((threadIdx.x & 31) == 0 && marked) atomicAdd(&flags->nweak, __popc(marked));
}

// One thread per unmarked link (mu, s), as gauge_force_kernel: Pi (optional) and per-block sums of Re tr(U Sigma)
template <class SRC>
__global__ void __launch_bounds__(kBSG, 2) gauge_force_fx_kernel(GaugeLex g, const void* __restrict__ U,
                                                                 const GaugeFlags* __restrict__ flags,
                                                                 const unsigned char* __restrict__ weak, double beta,
                                                                 double2* __restrict__ F, double* __restrict__ part) {
    if (gauge_all_fp64(*flags, 4 * g.V)) return;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    double retr = 0.0;
    if (i < 4 * g.V && !weak[i]) {
        const int mu = (int)(i / g.V);
        const size_t s = i - (size_t)mu * g.V;
        int c[4];
        size_t r = s;
        for (int d = 0; d < 4; ++d) {
            c[d] = (int)(r % g.L[d]);
            r /= g.L[d];
        }
        long long S[18];
#pragma unroll
        for (int k = 0; k < 18; ++k) S[k] = 0;
        const size_t xm = gauge_shift(g, c, s, mu, +1);
#pragma unroll 1
        for (int nu = 0; nu < 4; ++nu) {
            if (nu == mu) continue;
            const size_t xn = gauge_shift(g, c, s, nu, +1), xb = gauge_shift(g, c, s, nu, -1);
            int cb[4] = {c[0], c[1], c[2], c[3]};
            cb[nu] = c[nu] == 0 ? g.L[nu] - 1 : c[nu] - 1;
            const size_t xmb = gauge_shift(g, cb, xb, mu, +1);  // x + mu - nu
            const SRC a(U, g.V, nu, xm), b(U, g.V, mu, xn), c0(U, g.V, nu, s);
            fx_staple<false>(a, b, c0, S);  // U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+
            const SRC al(U, g.V, nu, xmb), bl(U, g.V, mu, xb), cl(U, g.V, nu, xb);
            fx_staple<true>(al, bl, cl, S);  // U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu)
        }
        FxM Sm;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            fx_limbs(S[2 * k] << 2, Sm.e[k].x, Sm.e[k].y);
            fx_limbs(S[2 * k + 1] << 2, Sm.e[k].z, Sm.e[k].w);
        }
        // O = U Sigma with 56 fraction bits
        const SRC own(U, g.V, mu, s);
        FxM u;
#pragma unroll
        for (int k = 0; k < 9; ++k) u.e[k] = own.at(k);
        long long O[18];
#pragma unroll
        for (int k = 0; k < 9; ++k)
            fx_dot3<false, false>(u.e + 3 * (k / 3), Sm.e[k % 3], Sm.e[3 + k % 3], Sm.e[6 + k % 3], O[2 * k], O[2 * k + 1]);
        retr = __ll2double_rn(O[0] + O[8] + O[16]) * 0x1p-56;
        if (F) {
            // Pi = -(beta/3) ta(O): off-diagonal (O - O^+)/2, diagonal i (Im O_aa - Im tr O / 3)
            const double f = -beta / 3.0 * 0x1p-56, fh = 0.5 * f;
            double2* o = F + ((size_t)mu * g.V + s) * 9;
            const double d0 = __ll2double_rn(O[1]), d1 = __ll2double_rn(O[9]), d2 = __ll2double_rn(O[17]);
            const double im3 = (d0 + d1 + d2) / 3.0;
            o[0] = make_double2(0.0, f * (d0 - im3));
            o[4] = make_double2(0.0, f * (d1 - im3));
            o[8] = make_double2(0.0, f * (d2 - im3));
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = a + 1; b < 3; ++b) {
                    const double re = fh * __ll2double_rn(O[2 * (3 * a + b)] - O[2 * (3 * b + a)]);
                    const double im = fh * __ll2double_rn(O[2 * (3 * a + b) + 1] + O[2 * (3 * b + a) + 1]);
                    o[3 * a + b] = make_double2(re, im);
                    o[3 * b + a] = make_double2(-re, im);
                }
        }
    }
    __shared__ double sm[kBSG / 32];
    retr = warp_sum(retr);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sm[wid] = retr;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < kBSG / 32; ++k) t += sm[k];
        part[blockIdx.x] = t;
    }
}

}  // namespace

cudaError_t launch_gauge_force_fx(const GaugeLex& g, const double2* U, const GaugeWork& w, double beta, double2* F,
                                  double* partials, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(w.flags, 0, sizeof(GaugeFlags), st);
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)((4 * g.V + kBSG - 1) / kBSG);
    note_launch();
    split_links_kernel<<<nb, kBSG, 0, st>>>(U, 4 * g.V, (int4*)w.limbs, w.flags, w.weak);
    note_launch();
    if (w.limbs) gauge_force_fx_kernel<Limbs><<<nb, kBSG, 0, st>>>(g, w.limbs, w.flags, w.weak, beta, F, partials);
    else gauge_force_fx_kernel<Direct><<<nb, kBSG, 0, st>>>(g, U, w.flags, w.weak, beta, F, partials);
    return cudaGetLastError();
}

}  // namespace odwf
