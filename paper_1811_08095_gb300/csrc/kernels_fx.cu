// Fixed-point hops (kernels_fx.cuh): the non-dagger epilogues and the site-local kernel that
// writes a hop's input.
#include "kernels_fx.cuh"

namespace odwf {

cudaError_t launch_hop_fx_dag(const HopParams<double>& P, Epi e, int nsys, cudaStream_t st);  // kernels_fx_dag.cu

cudaError_t launch_hop_fx(const HopParams<double>& P, Epi e, int nsys, cudaStream_t st) {
    switch (e) {
        case Epi::MINV: return hop_fx<EPI_MINV | FX_OUTB | FX_OUTFX>(P, nsys, st);
        case Epi::SCHUR: return hop_fx<EPI_SCHUR>(P, nsys, st);
        case Epi::SCHUR_NORM_MDINV: return hop_fx<EPI_SCHUR_NORM_MDINV | FX_OUTFX>(P, nsys, st);
        case Epi::SCHUR_MDINV: return hop_fx<EPI_SCHUR_NORM_MDINV_STORE | FX_OUTFX>(P, nsys, st);
        case Epi::FULL: return hop_fx<EPI_FULL>(P, nsys, st);
        case Epi::PLAIN: return hop_fx<EPI_PLAIN>(P, nsys, st);
        case Epi::ZMINUS_POSTMINV: return hop_fx<EPI_ZMINUS_POSTMINV>(P, nsys, st);
        default: return launch_hop_fx_dag(P, e, nsys, st);
    }
}

// out = op(in) of an FP64 field into the fixed-point format, two threads per 5D site as the hops
__global__ void __launch_bounds__(kFxThreads) m5_fx_kernel(FieldRef in, FieldRef out, Geom g, int p, int ns, int lg_ns,
                                                           const double* r_sys, int sys_base, FxOp op,
                                                           const double* tab5, const SysState* gate_st, int need) {
    extern __shared__ __align__(16) double s_cols[];
    __shared__ double s_fac;
    const int sys = blockIdx.y + sys_base;
    if (gate_st && gate_st[sys].status != need) return;
    const size_t gi = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const FxLane t(threadIdx.x, ns, lg_ns);
    const int a = t.a, s = t.s;
    const size_t hh = gi >> (lg_ns + 1);
    const bool valid = hh < (size_t)g.Vh;
    const int h = valid ? (int)hh : 0;
    const int site = threadIdx.x >> (lg_ns + 1), sites = blockDim.x >> (lg_ns + 1);
    const double r = r_sys[sys];
    double v[12];
    FxF64(in, sys, g, p, h, s, a, ns).load(v);
    if (op != FxOp::ID) {
        double* mine = s_cols + site * 24 * (ns + 1);
        if (op != FxOp::B && threadIdx.x == 0) s_fac = fx_corner(tab5, r, ns);
        __syncthreads();
        const double fac = s_fac;
        if (op == FxOp::B) fx_turn<C_ONEL>(v, s_cols, mine, s_cols, tab5, r, fac, a, s, sites, ns);
        else if (op == FxOp::MINVDAG) fx_turn<C_MINVDAG>(v, s_cols, mine, s_cols, tab5, r, fac, a, s, sites, ns);
        else fx_turn<C_MINV | C_OUTL>(v, s_cols, mine, s_cols, tab5, r, fac, a, s, sites, ns);
    }
    fx_store(out.d(sys), reinterpret_cast<int*>(out.n(sys)), (size_t)h, t, ns, valid, v);
}

cudaError_t launch_m5_fx(const FieldRef& in, const FieldRef& out, const Geom& g, int p, int ns, const double* r_sys,
                         int sys_base, int nsys, FxOp op, const double* tab5, cudaStream_t st,
                         const SysState* gate_st, int need) {
    const size_t n = (size_t)g.Vh * ns;
    const int bs = fx_threads(n);
    note_launch();
    m5_fx_kernel<<<dim3(blocks_for(2 * n, bs), nsys), bs, op == FxOp::ID ? 0 : fx_smem(bs, ns, 1, false), st>>>(
        in, out, g, p, ns, lg2(ns), r_sys, sys_base, op, tab5, gate_st, need);
    return cudaGetLastError();
}

// FP64 links into fixed point (fx.cuh), one thread per link.  The exponent leaves room for eight
// directions in a 63-bit sum: with the largest entry below 2^e and every row and column sum of
// |re| + |im| at most 2.5 2^e (SU(3): sqrt 6), a product component stays below 5 times the
// neighbour's largest.
__global__ void __launch_bounds__(128) links_fx_kernel(const double2* __restrict__ d18, int4* __restrict__ out,
                                                       int* __restrict__ ex, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double2 u[9];
    int mx = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        u[k] = d18[i * 9 + k];
        mx = max(mx, max(__double2hiint(u[k].x) & 0x7fffffff, __double2hiint(u[k].y) & 0x7fffffff));
    }
    const int emax = mx >> 20;
    const bool raw = emax == 0x7ff || (emax < kFxMinField && mx > 0);  // non-finite, or below 2^-958
    const int e = emax < kFxMinField ? 2046 : emax;                    // a zero link: everything shifted out
    long long q[18];
    unsigned row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        q[2 * k] = fx_from_double<7>(u[k].x, e);
        q[2 * k + 1] = fx_from_double<7>(u[k].y, e);
        const unsigned a = (unsigned)abs((int)(q[2 * k] >> 31)) + (unsigned)abs((int)(q[2 * k + 1] >> 31));
        row[k / 3] += a;
        col[k % 3] += a;
    }
    const unsigned big = max(max(max(row[0], row[1]), row[2]), max(max(col[0], col[1]), col[2]));
    const int more = big > 1342177280u ? 2 : 0;  // 2.5 x 2^29
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const FxLimbs re = fx_split(q[2 * k] >> more), im = fx_split(q[2 * k + 1] >> more);
        out[i * 9 + k] = make_int4(re.hi, re.lo, im.hi, im.lo);
    }
    ex[i] = raw ? kFxHard : emax < kFxMinField ? kFxZero : emax - 1022 + more;
}

cudaError_t launch_links_fx(const void* d18, void* fx, size_t n_links, cudaStream_t st) {
    note_launch();
    links_fx_kernel<<<blocks_for(n_links, 128), 128, 0, st>>>((const double2*)d18, (int4*)fx,
                                                              (int*)((char*)fx + n_links * 144), n_links);
    return cudaGetLastError();
}

}  // namespace odwf
