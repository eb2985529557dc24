// Packed Legendre adjoint of FP32 plans (legendre_pk.cuh).
#include "legendre_pk.cuh"

namespace gsl {

cudaError_t launch_leg_adj_pk_dd(const Plan &p, int rpt, const void *ring, void *alm, double wpos, void *fx,
                                 cudaStream_t st);

cudaError_t launch_leg_adj_pk(const Plan &p, int rpt, const void *ring, void *alm, double wpos, void *fx, cudaStream_t st)
{
    return p.prec == LENS_FP32 ? adj_pk_rpt<PkF>(p, rpt, ring, alm, wpos, fx, st)
                               : launch_leg_adj_pk_dd(p, rpt, ring, alm, wpos, fx, st);
}

}  // namespace gsl
