// The FP64-accuracy hops in block fixed point (fx.cuh): one thread per 5D site, the fused hop of
// kernels.cuh with its epilogues.  The input is a fixed-point field; a non-dagger hop reads
// chi = B psi, shifted once per site by the kernel that produced it.
//
// What bounds it: the FP64 pipe of the epilogues (about 130 to 220 operations per 5D site at 2 per
// clock and SM: 42 to 60% busy) and the latency of the integer stencil (1728 multiply-adds at 32 per
// clock and SM) with the 12 warps per SM that 168 registers leave.  16^3x32x16, one system, the four
// hops of S^dag S: 0.57 / 0.69 / 0.61 / 0.49 ms; the FP64 stencil they replace, 1334 to 1700 FP64
// operations per 5D site, took 2.6 to 3.0 ms each.  Four blocks per SM (128 registers) spill.
#pragma once

#include "fx.cuh"
#include "kernels.h"

namespace odwf {

constexpr int kFxThreads = 128;
constexpr int kFxMinBlocks = 3;
constexpr int kFxSite = 73;  // int4 words of a site's staged links (8 x 9, one more to spread the banks)

// Epilogue flags beyond kernels.cuh's: z and out formats are fixed by the epilogue
enum : int { FX_ZFX = 1 << 20, FX_OUTFX = 1 << 21, FX_OUTB = 1 << 22 };

// ---------------------------------------------------------------- bidiagonal operators
// bidiag_apply with one product and one multiply-add per real in both directions
__device__ __forceinline__ void fx_bidiag(double v[24], const double* a, const double* b, double r, int s, int ns,
                                          bool dag) {
    const int sm = (s + ns - 1) & (ns - 1), sp = (s + 1) & (ns - 1);
    const double as = a[s];
    // coefficients of the neighbours in s: up from sm (dag: sp), down from sp (dag: sm)
    const int su = dag ? sp : sm, sd = dag ? sm : sp;
    double cu = dag ? b[sp] : b[s], cd = dag ? b[sm] : b[s];
    if (s == (dag ? ns - 1 : 0)) cu *= -r;
    if (s == (dag ? 0 : ns - 1)) cd *= -r;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const double u = shfl_idx(v[k], su, ns), d = shfl_idx(v[12 + k], sd, ns);
        v[k] = fma(as, v[k], cu * u);
        v[12 + k] = fma(as, v[12 + k], cd * d);
    }
}

// ---------------------------------------------------------------- M^-1 along s
// The cyclic bidiagonal solves of minv_apply as serial recurrences: the block's spinors are turned
// in shared memory so that a thread walks the Ns values of one real of one site, w = inv_d v + al w,
// then adds A fac w_last (the corner).  Three FP64 operations per real against six of the log2 Ns
// shuffle scan, and the division of fac once per block.
//   tab: inv_d[Ns], then for each of the four recurrences (M^-1 up, M^-1 down, M^-dag up, M^-dag down)
//   al[Ns] = -c_s / d_s and A[Ns], its running product in the order of the recurrence.
// buf: (blockDim / Ns) * 24 columns of Ns + 1 doubles.  Every thread of the block must call.
__device__ __forceinline__ void fx_minv(double v[24], double* buf, const double* tab, double fac, int s, int ns,
                                        int lg_ns, bool dag) {
    double* mine = buf + (size_t)(threadIdx.x >> lg_ns) * 24 * (ns + 1) + s;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 24; ++k) mine[k * (ns + 1)] = v[k];
    __syncthreads();
    const int ncol = (blockDim.x >> lg_ns) * 24;
    // with 1.5 columns per thread, alternate blocks give the second one to the other warps (schedulers)
    for (int c = threadIdx.x ^ ((blockIdx.x & 1) * (blockDim.x >> 1)); c < ncol; c += blockDim.x) {
        const int down = (c % 24) >= 12;
        const double* al = tab + ns * (1 + 2 * ((dag ? 2 : 0) + down));
        const int step = (down != 0) == dag ? 1 : -1;  // M^-1: up forward, down backward; M^-dag the reverse
        int i = step > 0 ? 0 : ns - 1;
        double* p = buf + c * (ns + 1);
        double w = 0.0;
#pragma unroll 8
        for (int n = 0; n < ns; ++n, i += step) {
            w = fma(__ldg(al + i), w, __ldg(tab + i) * p[i]);
            p[i] = w;
        }
        const double wc = fac * w;
        for (int n = 0; n < ns; ++n) p[n] = fma(__ldg(al + ns + n), wc, p[n]);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 24; ++k) v[k] = mine[k * (ns + 1)];
}

// fac = -r / (1 + r A_last); A_last, the product of all al, is the same for the four recurrences
__device__ __forceinline__ double fx_corner(const double* tab, double r, int ns) {
    return -r / fma(r, __ldg(tab + 3 * ns - 1), 1.0);
}

// ---------------------------------------------------------------- the stencil
// (1 + sg gamma_mu) projection of one colour, limb by limb: h = up + sg G dn for both spins,
// (h0.re, h0.im, h1.re, h1.im); |h| < 2^60
template <int MU, bool PLUS>
__device__ __forceinline__ void fx_project(const int4& u0, const int4& u1, const int4& d0, const int4& d1,
                                           FxLimbs h[4]) {
    const FxLimbs u[4] = {{u0.x, u0.y}, {u0.z, u0.w}, {u1.x, u1.y}, {u1.z, u1.w}};
    const FxLimbs d[4] = {{d0.x, d0.y}, {d0.z, d0.w}, {d1.x, d1.y}, {d1.z, d1.w}};
    // G d: mu 0 (-i d1, -i d0), 1 (-d1, d0), 2 (-i d0, i d1), 3 (d0, d1): source real and whether it
    // enters with a minus sign
    constexpr int src[4][4] = {{3, 2, 1, 0}, {2, 3, 0, 1}, {1, 0, 3, 2}, {0, 1, 2, 3}};
    constexpr bool neg[4][4] = {{false, true, false, true}, {true, true, false, false}, {false, true, true, false},
                                {false, false, false, false}};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const FxLimbs g = d[src[MU][i]];
        h[i].hi = (neg[MU][i] == PLUS) ? u[i].hi - g.hi : u[i].hi + g.hi;
        h[i].lo = (neg[MU][i] == PLUS) ? u[i].lo - g.lo : u[i].lo + g.lo;
    }
}

// lower spins of the colour: acc += sg G^dag w, w = (w0, w1) complex
template <int MU, bool PLUS>
__device__ __forceinline__ void fx_lower(const long long w[4], long long& a0r, long long& a0i, long long& a1r,
                                         long long& a1i) {
    // G^dag w: mu 0 (i w1, i w0), 1 (w1, -w0), 2 (i w0, -i w1), 3 (w0, w1)
    long long g[4];
    bool n[4];
    if (MU == 0) { g[0] = w[3]; g[1] = w[2]; g[2] = w[1]; g[3] = w[0]; n[0] = true; n[1] = false; n[2] = true; n[3] = false; }
    else if (MU == 1) { g[0] = w[2]; g[1] = w[3]; g[2] = w[0]; g[3] = w[1]; n[0] = n[1] = false; n[2] = n[3] = true; }
    else if (MU == 2) { g[0] = w[1]; g[1] = w[0]; g[2] = w[3]; g[3] = w[2]; n[0] = true; n[1] = false; n[2] = false; n[3] = true; }
    else { g[0] = w[0]; g[1] = w[1]; g[2] = w[2]; g[3] = w[3]; n[0] = n[1] = n[2] = n[3] = false; }
    a0r = (n[0] == PLUS) ? a0r - g[0] : a0r + g[0];
    a0i = (n[1] == PLUS) ? a0i - g[1] : a0i + g[1];
    a1r = (n[2] == PLUS) ? a1r - g[2] : a1r + g[2];
    a1i = (n[3] == PLUS) ? a1i - g[3] : a1i + g[3];
}

// One direction: acc += [w ; sg G^dag w], w = (U h) >> sh, U staged as nine (re1, re0, im1, im0)
template <int MU, bool PLUS>
__device__ __forceinline__ void fx_dir(const int4* __restrict__ p, int ns, const int4* U, int sh,
                                       long long acc[24]) {
    FxLimbs h[3][4];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int4 u0 = __ldg(p + c * ns), u1 = __ldg(p + (3 + c) * ns), d0 = __ldg(p + (6 + c) * ns),
                   d1 = __ldg(p + (9 + c) * ns);
        fx_project<MU, PLUS>(u0, u1, d0, d1, h[c]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        long long A[4] = {0, 0, 0, 0}, B[4];  // leading and cross sums; B starts at the rounding half unit
#pragma unroll
        for (int i = 0; i < 4; ++i) B[i] = 1ll << 30;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 u = U[3 * a + b];
            const int m1 = fx_neg(u.z), m0 = fx_neg(u.w);
#pragma unroll
            for (int sp = 0; sp < 2; ++sp) {
                const FxLimbs x = h[b][2 * sp], y = h[b][2 * sp + 1];
                A[2 * sp] = fx_mad(u.x, x.hi, fx_mad(m1, y.hi, A[2 * sp]));
                A[2 * sp + 1] = fx_mad(u.x, y.hi, fx_mad(u.z, x.hi, A[2 * sp + 1]));
                B[2 * sp] = fx_mad(u.x, x.lo, fx_mad(u.y, x.hi, fx_mad(m1, y.lo, fx_mad(m0, y.hi, B[2 * sp]))));
                B[2 * sp + 1] = fx_mad(u.x, y.lo, fx_mad(u.y, y.hi, fx_mad(u.z, x.lo, fx_mad(u.w, x.hi, B[2 * sp + 1]))));
            }
        }
        long long w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = (A[i] + (B[i] >> 31)) >> sh;
        acc[2 * a] += w[0];
        acc[2 * a + 1] += w[1];
        acc[6 + 2 * a] += w[2];
        acc[6 + 2 * a + 1] += w[3];
        fx_lower<MU, PLUS>(w, acc[12 + 2 * a], acc[12 + 2 * a + 1], acc[18 + 2 * a], acc[18 + 2 * a + 1]);
    }
}

// The stencil in FP64 for one 5D site, for neighbours or links outside the fixed-point range
static __device__ __noinline__ void fx_hop_slow(const HopParams<double>& P, const void* in, const int* ex, int h, int s,
                                         bool dag, double* y) {
    for (int k = 0; k < 24; ++k) y[k] = 0.0;
    const int* nb = P.nbr + ((size_t)P.p_out * P.g.Vh + h) * 8;
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
        const int raw = nb[j], mu = j >> 1, hn = checked_index(raw & 0x7fffffff, P.g.Vh, P.bounds_flag, kBoundsNeighbour);
        double v[24], hp[12], u[18], w[12];
        fx_load_double(in, ex, (size_t)hn, s, P.ns, v);
        const double sg = ((j & 1) == 0) == dag ? 1.0 : -1.0;
        project(mu, sg, v, hp);
        const size_t idx = (j & 1) == 0 ? ((size_t)(P.p_out * 4 + mu) * P.g.Vh + h)
                                        : ((size_t)((1 - P.p_out) * 4 + mu) * P.g.Vh + hn);
        LinkIO<LinkD18, double>::load(P.links_d, idx, u);
        su3_mul(u, hp, w, (j & 1) != 0);
        if (raw < 0)
            for (int k = 0; k < 12; ++k) w[k] = -w[k];
        accumulate(mu, sg, w, y);
    }
}

// index of the link of direction j at site h (parity p_out) with neighbour hn
__device__ __forceinline__ size_t fx_link_index(const HopParams<double>& P, int j, int h, int hn) {
    return (j & 1) ? (size_t)((1 - P.p_out) * 4 + (j >> 1)) * P.g.Vh + hn : (size_t)(P.p_out * 4 + (j >> 1)) * P.g.Vh + h;
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
    extern __shared__ __align__(16) int4 s_links[];

    const int sys = blockIdx.y + P.sys_base;
    if (P.gate && P.st[sys].status != P.need_status) return;  // uniform over the block
    if (P.prof_count && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(P.prof_count, 1ull);

    const int ns = P.ns;
    const size_t gi = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int s = (int)(gi & (size_t)(ns - 1));
    const size_t hh = gi >> P.lg_ns;
    const bool valid = hh < (size_t)P.g.Vh;
    const int h = valid ? (int)hh : 0;  // threads past the last site read site 0's neighbours and store nothing
    const double r = P.r_sys[sys];

    int nb[8];
    {
        const int4* tp = reinterpret_cast<const int4*>(P.nbr + ((size_t)P.p_out * P.g.Vh + h) * 8);
        const int4 n0 = __ldg(tp), n1 = __ldg(tp + 1);
        const int raw[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) nb[j] = checked_index(raw[j] & 0x7fffffff, P.g.Vh, P.bounds_flag, kBoundsNeighbour);
    }
    // the site's eight links into shared memory, 72 elements over its Ns lanes: the adjoint for a
    // backward hop, negated (the -1 of -1/2 W) except across the antiperiodic boundary
    int4* my_links = s_links + (threadIdx.x >> P.lg_ns) * kFxSite;
    const int4* lk = reinterpret_cast<const int4*>(P.links);
    for (int i = s; i < 72; i += ns) {
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
    __syncwarp();

    const int4* in = reinterpret_cast<const int4*>(P.in.d(sys)) + chunk_slot(s, ns);
    const int* ex = reinterpret_cast<const int*>(P.in.n(sys));
    int e[8], M = kFxZero;
    bool slow = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int en = __ldg(ex + (size_t)nb[j] * ns + s), eu = __ldg(P.link_ex + fx_link_index(P, j, h, nb[j]));
        slow |= en == kFxRaw || eu == kFxRaw;
        e[j] = en + eu;
        M = max(M, e[j]);
    }
    long long acc[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] = 0;
#define ODWF_FX_DIR(MU_, DIR_)                                                                            \
    fx_dir<MU_, (DIR_ == 0) == DAG>(in + (size_t)nb[2 * MU_ + DIR_] * (12 * ns), ns,                      \
                                    my_links + 9 * (2 * MU_ + DIR_), min(M - e[2 * MU_ + DIR_], 63), acc)
    ODWF_FX_DIR(0, 0); ODWF_FX_DIR(0, 1);
    ODWF_FX_DIR(1, 0); ODWF_FX_DIR(1, 1);
    ODWF_FX_DIR(2, 0); ODWF_FX_DIR(2, 1);
    ODWF_FX_DIR(3, 0); ODWF_FX_DIR(3, 1);
#undef ODWF_FX_DIR
    // -1/2 W psi (or -1/2 W^dag psi) = acc 2^(M + 2) / 2
    double v[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) v[k] = fx_to_double(acc[k], M + 1);
    if (slow || ((M < kFxMinExp || M >= kFxMaxExp) && M > kFxZero / 2)) {
        double y[24];
        fx_hop_slow(P, P.in.d(sys), ex, h, s, DAG, y);
#pragma unroll
        for (int k = 0; k < 24; ++k) v[k] = -0.5 * y[k];
    }

    // the links are read: their shared memory now holds the recurrences of M^-1 (fx_minv)
    double* buf = reinterpret_cast<double*>(s_links);
    __shared__ double s_fac;
    if (HOPOP != OP_ID || POST != 0) {
        if (threadIdx.x == 0) s_fac = fx_corner(P.tab5, r, ns);
        __syncthreads();
    }
    const double fac = s_fac;

    if (DAG) fx_bidiag(v, P.cf.rho, P.cf.sigma, r, s, ns, true);  // B^dag: H^dag psi
    if (HOPOP == OP_MINV) fx_minv(v, buf, P.tab5, fac, s, ns, P.lg_ns, false);
    if (HOPOP == OP_MINVDAG) fx_minv(v, buf, P.tab5, fac, s, ns, P.lg_ns, true);
    if (ZOP != ZOP_NONE) {
        double z[24];
        if (F & FX_ZFX) fx_load_double(P.z.d(sys), reinterpret_cast<const int*>(P.z.n(sys)), (size_t)h, s, ns, z);
        else SpinorIO<SpF64, double>::load(P.z.d(sys), nullptr, (size_t)h, s, ns, z);
        if (ZOP == ZOP_M) fx_bidiag(z, P.cf.d, P.cf.e, r, s, ns, false);
        if (ZOP == ZOP_MDAG) fx_bidiag(z, P.cf.d, P.cf.e, r, s, ns, true);
#pragma unroll
        for (int k = 0; k < 24; ++k) v[k] = NEG ? z[k] - v[k] : z[k] + v[k];
    }
    double nrm = 0.0;
    if (NORM && valid) {
#pragma unroll
        for (int k = 0; k < 24; ++k) nrm = fma(v[k], v[k], nrm);
    }
    if (POST == OP_MINV) fx_minv(v, buf, P.tab5, fac, s, ns, P.lg_ns, false);
    if (POST == OP_MINVDAG) fx_minv(v, buf, P.tab5, fac, s, ns, P.lg_ns, true);
    if (F & FX_OUTB) fx_bidiag(v, P.cf.rho, P.cf.sigma, r, s, ns, false);

    if (valid) {
        if (CG) {
            // v = A p;  r <- r - alpha A p;  x <- x + alpha p;  nrm = |r|^2
            const double alpha = P.st[sys].alpha;
            double w[24];
            SpinorIO<SpF64, double>::load(P.cg_r.d(sys), nullptr, (size_t)h, s, ns, w);
#pragma unroll
            for (int k = 0; k < 24; ++k) {
                w[k] = fma(-alpha, v[k], w[k]);
                nrm = fma(w[k], w[k], nrm);
            }
            SpinorIO<SpF64, double>::store(P.cg_r.d(sys), nullptr, (size_t)h, s, ns, w);
            SpinorIO<SpF64, double>::load(P.cg_x.d(sys), nullptr, (size_t)h, s, ns, w);
            SpinorIO<SpF64, double>::load(P.cg_p.d(sys), nullptr, (size_t)h, s, ns, v);
#pragma unroll
            for (int k = 0; k < 24; ++k) w[k] = fma(alpha, v[k], w[k]);
            SpinorIO<SpF64, double>::store(P.cg_x.d(sys), nullptr, (size_t)h, s, ns, w);
        } else {
            if (RESID) {
                double b[24];
                SpinorIO<SpF64, double>::load(P.b.d(sys), nullptr, (size_t)h, s, ns, b);
#pragma unroll
                for (int k = 0; k < 24; ++k) {
                    v[k] = b[k] - v[k];
                    nrm = fma(v[k], v[k], nrm);
                }
            }
            if (F & FX_OUTFX) fx_store(P.out.d(sys), reinterpret_cast<int*>(P.out.n(sys)), (size_t)h, s, ns, v);
            else SpinorIO<SpF64, double>::store(P.out.d(sys), nullptr, (size_t)h, s, ns, v);
        }
    }
    if (REDUCE) reduce_and_finalize(nrm, P.partials, P.counters, P.st, sys, FIN, P.part_stride);
}

// Threads per block: 128, or 64 while that leaves fewer than two blocks for each of the 152 SMs
// (a small lattice then spreads over twice the SMs) and for Ns = 2, whose staged links fill shared memory.
inline int fx_threads(size_t n5, int ns) { return ns == 2 || n5 < (size_t)kFxThreads * 304 ? 64 : kFxThreads; }
// dynamic shared memory of a block: its staged links or the recurrences' columns, whichever is larger
inline size_t fx_smem(int bs, int ns, bool links) {
    const size_t cols = (size_t)(bs / ns) * 24 * (ns + 1) * sizeof(double);
    const size_t lk = links ? (size_t)(bs / ns) * kFxSite * sizeof(int4) : 0;
    return cols > lk ? cols : lk;
}

template <int F>
cudaError_t hop_fx(const HopParams<double>& P, int nsys, cudaStream_t st) {
    const size_t n = (size_t)P.g.Vh * P.ns;
    const int bs = fx_threads(n, P.ns);
    note_launch();
    hop_fx_kernel<F><<<dim3(blocks_for(n, bs), nsys), bs, fx_smem(bs, P.ns, true), st>>>(P);
    return cudaGetLastError();
}

}  // namespace odwf
