// Packed Legendre synthesis and adjoint of FP64 plans, double-float (legendre_pk.cuh).
#include "legendre_pk.cuh"

namespace gsl {

cudaError_t launch_leg_fwd_pk_dd(const Plan &p, int rpt, const void *src, void *ring, double wpos, bool ring_dd, cudaStream_t st)
{
    return fwd_pk_rpt<PkD, 1>(p, rpt, src, ring, wpos, ring_dd, st);
}

cudaError_t launch_leg_adj_pk_dd(const Plan &p, int rpt, const void *ring, void *alm, double wpos, void *fx,
                                 cudaStream_t st)
{
    return adj_pk_rpt<PkD>(p, rpt, ring, alm, wpos, fx, st);
}

}  // namespace gsl
