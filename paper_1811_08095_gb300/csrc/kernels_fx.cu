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

// out = op(in) of an FP64 field into the fixed-point format
__global__ void __launch_bounds__(128) m5_fx_kernel(FieldRef in, FieldRef out, size_t n_sites, int ns, int lg_ns,
                                                    const double* r_sys, int sys_base, FxOp op,
                                                    const __grid_constant__ Coef5<double> cf, const SysState* gate_st,
                                                    int need) {
    const int sys = blockIdx.y + sys_base;
    if (gate_st && gate_st[sys].status != need) return;
    const size_t gi = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int s = (int)(gi & (size_t)(ns - 1));
    const size_t h = gi >> lg_ns;
    const bool valid = h < n_sites;
    const double r = r_sys[sys];
    double v[24];
    if (valid) {
        SpinorIO<SpF64, double>::load(in.d(sys), nullptr, h, s, ns, v);
    } else {
#pragma unroll
        for (int k = 0; k < 24; ++k) v[k] = 0.0;
    }
    if (op == FxOp::MINVDAG) minv_apply(v, cf, r, s, ns, true);
    if (op == FxOp::B_MINV) minv_apply(v, cf, r, s, ns, false);
    if (op == FxOp::B || op == FxOp::B_MINV) fx_bidiag(v, cf.rho, cf.sigma, r, s, ns, false);
    if (valid) fx_store(out.d(sys), reinterpret_cast<int*>(out.n(sys)), h, s, ns, v);
}

cudaError_t launch_m5_fx(const FieldRef& in, const FieldRef& out, size_t n_sites, int ns, const double* r_sys,
                         int sys_base, int nsys, FxOp op, const Coef5<double>& cf, cudaStream_t st,
                         const SysState* gate_st, int need) {
    note_launch();
    m5_fx_kernel<<<dim3(blocks_for(n_sites * ns, 128), nsys), 128, 0, st>>>(in, out, n_sites, ns, lg2(ns), r_sys,
                                                                            sys_base, op, cf, gate_st, need);
    return cudaGetLastError();
}

}  // namespace odwf
