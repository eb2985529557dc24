// FP32 interpolation and spreading (nufft.cuh).
#include "nufft.cuh"
#include "nufft_strip.cuh"

namespace gsl {

cudaError_t interp_f32(const Plan &p, const void *grid, void *map, cudaStream_t st)
{
    return p.spin ? interp_dispatch<float, true>(p, grid, map, st) : interp_dispatch<float, false>(p, grid, map, st);
}

cudaError_t spread_f32(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    return p.spin ? spread_dispatch<float, true>(p, map, grid, st) : spread_dispatch<float, false>(p, map, grid, st);
}

}  // namespace gsl
