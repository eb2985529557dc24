// Double-float real numbers with operators, and complex numbers of them: the synthesis transforms of fft.cuh and
// torus.cu run with T = dfl in FP64 plans with restart values, where FP64 butterflies waited for GB300's FP64 pipe
// (1/60 of the FP32 rate), as long as the plan's truncation error hides their rounding (plan.cu: not with W = 16 on small
// grids).  lmax 2048, spin 2: theta 2.68 -> 0.65 ms, phi 2.45 -> 0.60 ms; the error of a synthesis against
// 64-bit sums is unchanged (epsilon 1e-10, lmax 512 to 4096: within 0.05%).  Operations are those of common.cuh's df32 (sums by
// two-sum, ~2^-46 relative; not renormalised); factors of +-1 and 1/2 are plain floats.  Not for the adjoint: there the
// deconvolution comes last and amplifies the transforms' rounding noise (5e-13 of the a_lm).
#pragma once

#include "common.cuh"

namespace gsl {

struct dfl {
    float h, l;
    __host__ __device__ constexpr dfl() : h(0.f), l(0.f) {}
    __host__ __device__ constexpr dfl(float h_, float l_) : h(h_), l(l_) {}
    __host__ __device__ explicit constexpr dfl(double d) : h((float)d), l((float)(d - (double)(float)d)) {}
};
struct __align__(16) dfl2 {
    dfl x, y;
};
template <> struct cplx_of<dfl> { using type = dfl2; };

// Type of an exact factor (+-1, 1/2) in front of a T
template <typename T> struct sign_of { using type = T; };
template <> struct sign_of<dfl> { using type = float; };
template <typename T> using sgn = typename sign_of<T>::type;

__device__ __forceinline__ dfl to_dfl(df32 a) { return {a.h, a.l}; }
__device__ __forceinline__ df32 to_df(dfl a) { return {a.h, a.l}; }
__device__ __forceinline__ dfl operator-(dfl a) { return {-a.h, -a.l}; }
__device__ __forceinline__ dfl operator+(dfl a, dfl b) { return to_dfl(df_sub_u(to_df(a), df32{-b.h, -b.l})); }
__device__ __forceinline__ dfl operator-(dfl a, dfl b) { return to_dfl(df_sub_u(to_df(a), to_df(b))); }
__device__ __forceinline__ dfl operator*(dfl a, dfl b) { return to_dfl(df_mul(to_df(a), to_df(b))); }
__device__ __forceinline__ dfl operator*(float f, dfl a) { return {f * a.h, f * a.l}; }  // f a power of two, +-
__device__ __forceinline__ dfl operator*(dfl a, float f) { return f * a; }
__device__ __forceinline__ dfl operator*(int f, dfl a) { return (float)f * a; }
// a b + c, as df_fma of common.cuh
__device__ __forceinline__ dfl dfl_fma(dfl a, dfl b, dfl c)
{
    const float s = __fadd_rn(c.h, __fmul_rn(a.h, b.h));
    const float bb = __fsub_rn(s, c.h);
    const float ec = __fsub_rn(c.h, __fsub_rn(s, bb));
    const float ep = __fmaf_rn(a.h, b.h, -bb);
    const float lo = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, c.l));
    return {s, __fadd_rn(lo, __fadd_rn(ec, ep))};
}
__device__ __forceinline__ dfl2 mkc(dfl r, dfl i) { return {r, i}; }
__device__ __forceinline__ dfl2 cadd(dfl2 a, dfl2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ dfl2 csub(dfl2 a, dfl2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ dfl2 cmul(dfl2 a, dfl2 b) { return {dfl_fma(-a.y, b.y, a.x * b.x), dfl_fma(a.y, b.x, a.x * b.y)}; }
__device__ __forceinline__ dfl2 cmulc(dfl2 a, dfl2 b) { return {dfl_fma(a.y, b.y, a.x * b.x), dfl_fma(-a.x, b.y, a.y * b.x)}; }
__device__ __forceinline__ dfl2 cscale(dfl2 a, dfl s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ dfl2 cscale(dfl2 a, float s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ dfl2 cmul_i(dfl2 a) { return {-a.y, a.x}; }
__device__ __forceinline__ dfl2 cmul_mi(dfl2 a) { return {a.y, -a.x}; }

__device__ __forceinline__ double dfl_value(dfl a) { return (double)a.h + (double)a.l; }

// elements of device tables
__device__ __forceinline__ float2 ldc(const float2 *p) { return __ldg(p); }
__device__ __forceinline__ double2 ldc(const double2 *p) { return __ldg(p); }
__device__ __forceinline__ dfl2 ldc(const dfl2 *p)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return {dfl(v.x, v.y), dfl(v.z, v.w)};
}

}  // namespace gsl
