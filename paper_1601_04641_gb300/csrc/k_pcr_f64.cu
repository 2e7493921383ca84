// FP64 line solves by truncated cyclic reduction (gp_pcr.cuh): the Cartesian
// sweeps of every form, and the axial condensate's radial sweep.
#include "gp_pcr.cuh"

namespace gpcn {

namespace {
template <class F> cudaError_t by_kind(Kind k, const SweepArgs &a, const PcrArgs &p, cudaStream_t s) {
    switch (k) {
    case K_X: return p.rhs ? launch_pcr<F, K_X, true>(a, p, s) : launch_pcr<F, K_X, false>(a, p, s);
    case K_Y: return launch_pcr<F, K_Y, false>(a, p, s);
    case K_Z: return launch_pcr<F, K_Z, false>(a, p, s);
    }
    return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t launch_sweep_pcr(Form form, Kind kind, const SweepArgs &a, const PcrArgs &p, cudaStream_t s) {
    if (a.n_lines <= 0) return cudaSuccess;
    switch (form) {
    case F_IMAG_REAL: return by_kind<FImagReal<double>>(kind, a, p, s);
    case F_IMAG_CPLX: return by_kind<FImagCplx<double>>(kind, a, p, s);
    case F_REALTIME: return by_kind<FRealTime<double>>(kind, a, p, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace gpcn
