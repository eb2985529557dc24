// FP64 interpolation (nufft.cuh).
#include "nufft.cuh"

namespace gsl {

cudaError_t interp_f64(const Plan &p, const void *grid, void *map, cudaStream_t st)
{
    return p.spin ? interp_dispatch<double, true>(p, grid, map, st) : interp_dispatch<double, false>(p, grid, map, st);
}

}  // namespace gsl
