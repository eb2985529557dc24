// FP64 spreading (nufft.cuh).
#include "nufft.cuh"
#include "nufft_strip.cuh"

namespace gsl {

cudaError_t spread_f64(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    return p.spin ? spread_dispatch<double, true>(p, map, grid, st) : spread_dispatch<double, false>(p, map, grid, st);
}

}  // namespace gsl
