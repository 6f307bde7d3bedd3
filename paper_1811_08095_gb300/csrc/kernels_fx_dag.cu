// Fixed-point hops (kernels_fx.cuh): the adjoint epilogues.
#include "kernels_fx.cuh"

namespace odwf {

cudaError_t launch_hop_fx_dag(const HopParams<double>& P, Epi e, int nsys, cudaStream_t st) {
    switch (e) {
        case Epi::D_MINVDAG: return hop_fx<EPID_MINVDAG | FX_OUTFX>(P, nsys, st);
        case Epi::D_NORMAL: return hop_fx<EPID_NORMAL | FX_ZFX>(P, nsys, st);
        case Epi::D_NORMAL_CG: return hop_fx<EPID_NORMAL_CG | FX_ZFX>(P, nsys, st);
        case Epi::D_NORMAL_RESID: return hop_fx<EPID_NORMAL_RESID | FX_ZFX>(P, nsys, st);
        case Epi::D_ZMINUS: return hop_fx<EPID_ZMINUS>(P, nsys, st);
        case Epi::D_FULL: return hop_fx<EPID_FULL>(P, nsys, st);
        case Epi::D_PLAIN: return hop_fx<EPID_PLAIN>(P, nsys, st);
        case Epi::D_ZMINUS_POSTMINVDAG: return hop_fx<EPID_ZMINUS_POSTMINVDAG>(P, nsys, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace odwf
