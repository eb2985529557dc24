// Packed Legendre synthesis of FP32 plans (legendre_pk.cuh).
#include "legendre_pk.cuh"

namespace gsl {

cudaError_t launch_leg_fwd_pk_dd(const Plan &p, int rpt, const void *src, void *ring, double wpos, bool ring_dd, cudaStream_t st);

// rpt: rings per thread 1, 2 or 4 (spin 0 pairs two rings, so 1 runs as 2)
cudaError_t launch_leg_fwd_pk(const Plan &p, int rpt, const void *src, void *ring, int nm, double wpos, bool ring_dd,
                              cudaStream_t st)
{
    if (p.prec != LENS_FP32)
        return nm == 1 ? launch_leg_fwd_pk_dd(p, rpt, src, ring, wpos, ring_dd, st) : cudaErrorInvalidValue;
    if (nm == 1) return fwd_pk_rpt<PkF, 1>(p, rpt, src, ring, wpos, false, st);
    if (nm == 2) return fwd_pk_rpt<PkF, 2>(p, rpt, src, ring, wpos, false, st);
    return nm == 4 ? fwd_pk_rpt<PkF, 4>(p, rpt, src, ring, wpos, false, st) : cudaErrorInvalidValue;
}

}  // namespace gsl
