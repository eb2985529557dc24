// Pairs of FP32 numbers in one 64-bit register (Blackwell's f32x2 instructions).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace gsl {
namespace {

using pk = unsigned long long;  // two FP32 numbers: low word first

__device__ __forceinline__ pk pk_make(float a, float b)
{
    pk r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 pk_get(pk v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ pk pk_fma(pk a, pk b, pk c)
{
    pk r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ pk pk_mul(pk a, pk b)
{
    pk r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pk pk_add(pk a, pk b)
{
    pk r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pk pk_sub(pk a, pk b)
{
    pk r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Double-float arithmetic on pairs (df32 of common.cuh, operation for operation)
struct __align__(16) D2 {
    pk h, l;
};
__device__ __forceinline__ D2 d2_mul(D2 a, D2 b)
{
    const pk p = pk_mul(a.h, b.h);
    const pk np = p ^ 0x8000000080000000ull;
    pk e = pk_fma(a.h, b.h, np);
    e = pk_fma(a.h, b.l, e);
    e = pk_fma(a.l, b.h, e);
    return {p, e};
}
__device__ __forceinline__ D2 d2_add_u(D2 a, D2 b)
{
    const pk s = pk_add(a.h, b.h);
    const pk bb = pk_sub(s, a.h);
    pk err = pk_add(pk_sub(a.h, pk_sub(s, bb)), pk_sub(b.h, bb));
    err = pk_add(err, pk_add(a.l, b.l));
    return {s, err};
}
// The product of two pairs as two scalar instructions (the same pipe time): ptxas contracts mul.rn.f32x2
// followed by add.rn.f32x2 into one fma, which the error terms below cannot have.
__device__ __forceinline__ pk pk_mul_alone(pk a, pk b)
{
    const float2 x = pk_get(a), y = pk_get(b);
    return pk_make(__fmul_rn(x.x, y.x), __fmul_rn(x.y, y.y));
}
// a b + c in 10 operations (mul then add: 12, and two negations): the two-sum of c.h and p = fl(a.h b.h) gives
// s, bb = fl(s - c.h) and c' = s - bb exactly; the error of s is (c.h - c') + (p - bb), and with the product's own
// error a.h b.h - p the second part becomes a.h b.h - bb, one fma.
__device__ __forceinline__ D2 d2_fma(D2 a, D2 b, D2 c)
{
    const pk s = pk_add(c.h, pk_mul_alone(a.h, b.h));
    const pk nbb = pk_sub(c.h, s);
    const pk ec = pk_sub(c.h, pk_add(s, nbb));
    const pk ep = pk_fma(a.h, b.h, nbb);
    pk lo = pk_fma(a.h, b.l, c.l);
    lo = pk_fma(a.l, b.h, lo);
    return {s, pk_add(lo, pk_add(ec, ep))};
}
__device__ __forceinline__ D2 d2_norm(D2 a)
{
    const pk h = pk_add(a.h, a.l);
    const pk bb = pk_sub(h, a.h);
    return {h, pk_add(pk_sub(a.h, pk_sub(h, bb)), pk_sub(a.l, bb))};
}
}  // namespace
}  // namespace gsl
