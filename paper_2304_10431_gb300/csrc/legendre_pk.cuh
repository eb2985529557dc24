// Legendre synthesis and adjoint with restart values, in packed pairs of FP32 numbers.
//
// The sums and the recursion are those of legendre.cu; plans with restart values (FP32 plans at
// epsilon >= 1e-5, FP64 plans at epsilon >= 5e-11) run them here.  Blackwell's f32x2
// instructions (fma / add / mul on a 64-bit register holding two FP32 numbers) do two lanes' worth of
// work per issue slot at the same rounding, and the Legendre steps were bound by instruction issue
// (12 FP32 instructions per ring and degree for spin s, the loads and the loop around them), so every
// value here is a pair:
//   spin s:  (+s value, -s value) of one ring,
//   spin 0:  the values of two rings (32 rings apart).
// Measured on GB300 (FP32 FMA per clock and SM): fma.rn.f32x2 125 with an operand shared by neighbouring
// instructions, 84 with three distinct ones (as the scalar instruction: the register file delivers two operands
// per lane and clock), add / mul.rn.f32x2 125; negating an operand costs two logic instructions (31-50), so
// no operand is ever negated in the loop.  Instead:
//   * the plain step mu_l = c_l mu_{l-1} - mu_{l-2} carries nu_l = sigma_l mu_l with the signs
//     sigma = (-, -, +, +) repeating over the degrees of a block (sigma_l = -sigma_{l-2}), which turns it into
//     nu_l = (sigma_l sigma_{l-1} c_l) nu_{l-1} + nu_{l-2}: one fma; sigma_l sigma_{l-1} (-, +, ...) is folded into
//     the step entry, sigma_l into the coefficients (forward) or the flush (adjoint).  A block of 8
//     degrees begins and ends with sigma = +, so restart values are stored unsigned;
//   * the sign rel = (-1)^(l - lf) of the mirrored ring is folded into the coefficient pairs.
//
// One warp owns 32 RPT rings of one order and works alone (no CTA barrier): it brings the step
// entries and the coefficients of 64 degrees into its shared memory in the form the loop reads
// (duplicated, signed, scaled; one 16-byte broadcast load gives two operands), so neither a
// coefficient pass over the a_lm nor duplicated tables in device memory are needed, and the loop has
// no global loads but the restart values.  Degrees beyond lmax are staged as zeros, so the last
// block needs no tail.  States away from the scale 2^0 (evanescent rings) take the SCALED block,
// which rescales every four degrees (four steps grow a value by at most 2^34).
//
// Time per launch at lmax 4096, before (scalar instructions, coefficient pass, rings per thread adjacent) and
// after, ms: FP32 spin 0 synthesis 4.35 -> 3.0, adjoint 5.26 -> 4.6; spin 2 11.4 -> 7.6, 13.6 -> 10.1; FP64 spin 0
// 19.2 -> 16.3, 27.0 -> 21.8; spin 2 63.6 -> 51.3, 100.7 -> 70.4.  The loops are bound by register operands
// (FP32: the FMA pipe is busy 63% of the cycles against 67% with three operand reads each) and, in double-float, by the
// FMA pipe.  Tried and not kept: skipping the 32-ring groups of a warp that are still evanescent
// (8-16% fewer ring-degrees, but a second copy of the block: spin 2 7.5 -> 7.9 ms).
//
// Arithmetic: PkF, FP32 (FP32 plans; rings below ck.jb in Reinsch's form, the others in the monic plain
// form), and PkD, double-float pairs (FP64 plans; monic form, every operation of common.cuh's
// df32 on two lanes).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "legendre_rec.cuh"
#include "pk.cuh"

namespace gsl {
namespace {

constexpr int kStage = 64;  // degrees staged at a time
constexpr float kUpF = 0x1p20f;  // a scaled state moves up one exponent from this magnitude on
enum { kSpin0 = 0, kSpinS = 1, kGrad = 2 };

// FP32 arithmetic on pairs
struct PkF {
    using V = pk;       // a pair of values, coefficients or sums
    using X = pk;       // cos theta (or 1 - cos theta) of the pair's rings
    using S = float;    // one value
    using C2 = float2;  // ring coefficient
    using R = float;
    static __device__ __forceinline__ V zero() { return 0ull; }
    static __device__ __forceinline__ V make(S a, S b) { return pk_make(a, b); }
    static __device__ __forceinline__ void get(V v, S &a, S &b)
    {
        const float2 t = pk_get(v);
        a = t.x;
        b = t.y;
    }
    static __device__ __forceinline__ V mac(V acc, V k, V v) { return pk_fma(k, v, acc); }
    static __device__ __forceinline__ V vscale(V v, pk f) { return pk_mul(v, f); }
    static __device__ __forceinline__ V norm(V v) { return v; }
    static __device__ __forceinline__ S sadd(S a, S b) { return a + b; }
    static __device__ __forceinline__ S ssub(S a, S b) { return a - b; }
    static __device__ __forceinline__ S ssgn(S a, float sg) { return a * sg; }
    static __device__ __forceinline__ R out(S a) { return a; }
    static __device__ __forceinline__ S in(float v) { return v; }
    static __device__ __forceinline__ S shfl(S v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
    static __device__ __forceinline__ float mag(S a) { return fabsf(a); }
};

struct PkD {
    using V = D2;
    struct X { D2 v; };
    using S = df32;
    using C2 = double2;
    using R = double;
    static __device__ __forceinline__ V zero() { return {0ull, 0ull}; }
    static __device__ __forceinline__ V make(S a, S b) { return {pk_make(a.h, b.h), pk_make(a.l, b.l)}; }
    static __device__ __forceinline__ void get(V v, S &a, S &b)
    {
        const float2 h = pk_get(v.h), l = pk_get(v.l);
        a = {h.x, l.x};
        b = {h.y, l.y};
    }
    static __device__ __forceinline__ V mac(V acc, V k, V v) { return d2_fma(k, v, acc); }
    static __device__ __forceinline__ V vscale(V v, pk f) { return {pk_mul(v.h, f), pk_mul(v.l, f)}; }
    static __device__ __forceinline__ V norm(V v) { return d2_norm(v); }
    static __device__ __forceinline__ S sadd(S a, S b) { return df_add_u(a, b); }
    static __device__ __forceinline__ S ssub(S a, S b) { return df_sub_u(a, b); }
    static __device__ __forceinline__ S ssgn(S a, float sg) { return df_scale_pow2(a, sg); }
    static __device__ __forceinline__ R out(S a) { return (double)a.h + (double)a.l; }
    static __device__ __forceinline__ S in(double v) { return df_split(v); }
    static __device__ __forceinline__ S shfl(S v, int off)
    {
        return {__shfl_xor_sync(0xffffffffu, v.h, off), __shfl_xor_sync(0xffffffffu, v.l, off)};
    }
    static __device__ __forceinline__ float mag(S a) { return fabsf(a.h); }
};

// ---------------------------------------------------------------- staged step entries
// Per degree two entries, s4 (16 bytes) and s2 (8 bytes):
//   PkF plain, spin s   s4 = (a, a, t, -t)      a, t = alpha_l, tau_l times sigma_l sigma_{l-1}
//   PkF plain, spin 0   s2 = (a, a)
//   PkF Reinsch         s4 = (-A, -A, -K, -K-), s2 = (B, B); K- = K + 2 AT (spin 0: K)
//   PkD, spin s         s4 = (t.h, -t.h, t.l, -t.l), s2 = (a.h, a.l)
//   PkD, spin 0         s4 = (a.h, a.h, a.l, a.l)
struct StageMem {
    float4 *s4;
    float2 *s2;
};

template <class A, int MODE, bool REIN>
__device__ __forceinline__ void stage_step(const StageMem &sm, int i, const void *rec, int64_t idx, bool live, int dl)
{
    const float sg = (dl & 1) ? 1.f : -1.f;  // sigma_l sigma_{l-1}
    if constexpr (REIN) {
        const float4 c = live ? __ldg((const float4 *)rec + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float km = MODE == kSpin0 ? c.w : __fmaf_rn(2.f, c.z, c.w);
        sm.s4[i] = make_float4(-c.x, -c.x, -c.w, -km);
        sm.s2[i] = make_float2(c.y, c.y);
    } else if constexpr (MODE == kSpin0) {
        float2 c = live ? __ldg((const float2 *)rec + idx) : make_float2(0.f, 0.f);
        c.x *= sg;
        c.y *= sg;
        if constexpr (std::is_same<A, PkF>::value) sm.s2[i] = make_float2(c.x, c.x);
        else sm.s4[i] = make_float4(c.x, c.x, c.y, c.y);
    } else {
        float4 c = live ? __ldg((const float4 *)rec + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
        c.x *= sg; c.y *= sg; c.z *= sg; c.w *= sg;
        if constexpr (std::is_same<A, PkF>::value) {
            sm.s4[i] = make_float4(c.x, c.x, c.z, -c.z);
        } else {
            sm.s4[i] = make_float4(c.z, -c.z, c.w, -c.w);
            sm.s2[i] = make_float2(c.x, c.y);
        }
    }
}

__device__ __forceinline__ ulonglong2 ld4(const float4 *p) { return *reinterpret_cast<const ulonglong2 *>(p); }
__device__ __forceinline__ pk ld2(const float2 *p) { return *reinterpret_cast<const pk *>(p); }

// ---------------------------------------------------------------- ring states
// NR pairs per thread; w[1] holds the newest value (Reinsch: w[1] the value, w[0] the difference).
// E: exponents (base 2^60) of the pair's two states, zero in unscaled blocks.
template <class A, int MODE, bool REIN, int NR> struct Pairs {
    using V = typename A::V;
    V w[2][NR];
    pk x[NR];                     // PkF: (x, x') ; PkD: spin s (x.h, x.l) of the ring, spin 0 the high words
    pk xl[NR];                    // PkD spin 0: the low words
    int Ea[NR], Eb[NR];
    static constexpr int RPT = MODE == kSpin0 ? 2 * NR : NR;  // rings per thread
    // ring of slot k of this thread: wb + 32 k + lane
    __device__ __forceinline__ void geom(const RingTab &rt, int r0, int nnorth)
    {
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            float2 v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int r = r0 + 32 * (MODE == kSpin0 ? 2 * u + q : u);
                v[q] = make_float2(0.f, 0.f);
                if (r < nnorth) {
                    if constexpr (REIN) v[q].x = __ldg(rt.y1 + r);
                    else v[q] = __ldg(rt.xdf + r);
                }
            }
            xl[u] = 0ull;
            if constexpr (std::is_same<A, PkF>::value) {
                x[u] = pk_make(v[0].x, v[1].x);
            } else if constexpr (MODE == kSpin0) {
                x[u] = pk_make(v[0].x, v[1].x);
                xl[u] = pk_make(v[0].y, v[1].y);
            } else {
                x[u] = pk_make(v[0].x, v[0].y);
            }
            Ea[u] = 0;
            Eb[u] = 0;
            w[0][u] = A::zero();
            w[1][u] = A::zero();
        }
    }
    // states before degree lf + K k, from row k of the restart values; true if any is scaled
    __device__ __forceinline__ bool restart(const CkTab &ck, int64_t row, int r0, int nnorth, float i0, float i1)
    {
        bool sc = false;
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            if constexpr (MODE == kSpin0) {
                typename A::S a[2], b[2];
                int e[2] = {0, 0};
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int r = r0 + 32 * (2 * u + q);
                    a[q] = {};
                    b[q] = {};
                    if (r >= nnorth) continue;
                    if constexpr (std::is_same<A, PkF>::value) {
                        const float2 v = __ldg((const float2 *)ck.v + row + r);
                        a[q] = REIN ? v.x : v.x * i0;
                        b[q] = REIN ? v.y : v.y * i1;
                    } else {
                        const float4 v = __ldg((const float4 *)ck.v + row + r);
                        a[q] = {v.x, v.y};
                        b[q] = {v.z, v.w};
                    }
                    e[q] = __ldg((const short *)ck.e + row + r);
                }
                w[0][u] = A::make(a[0], a[1]);
                w[1][u] = A::make(b[0], b[1]);
                Ea[u] = e[0];
                Eb[u] = e[1];
            } else {
                const int r = r0 + 32 * u;
                if (r < nnorth) {
                    const short2 e = __ldg((const short2 *)ck.e + row + r);
                    if constexpr (std::is_same<A, PkF>::value) {
                        float4 v = __ldg((const float4 *)ck.v + row + r);
                        if (!REIN) { v.x *= i0; v.y *= i1; v.z *= i0; v.w *= i1; }
                        w[0][u] = pk_make(v.x, v.z);
                        w[1][u] = pk_make(v.y, v.w);
                    } else {
                        const float4 p = __ldg((const float4 *)ck.v + 2 * (row + r));
                        const float4 n = __ldg((const float4 *)ck.v + 2 * (row + r) + 1);
                        w[0][u] = {pk_make(p.x, n.x), pk_make(p.y, n.y)};
                        w[1][u] = {pk_make(p.z, n.z), pk_make(p.w, n.w)};
                    }
                    Ea[u] = e.x;
                    Eb[u] = e.y;
                }
            }
            sc = sc || Ea[u] != 0 || Eb[u] != 0;
        }
        return __any_sync(0xffffffffu, sc);
    }
    __device__ __forceinline__ void renorm()
    {
        if constexpr (!std::is_same<A, PkF>::value) {
#pragma unroll
            for (int u = 0; u < NR; ++u) {
                w[0][u] = A::norm(w[0][u]);
                w[1][u] = A::norm(w[1][u]);
            }
        }
    }
    // one degree (position i of the stage), the newest value into word NW
    template <int NW> __device__ __forceinline__ void advance(const StageMem &sm, int i)
    {
        if constexpr (std::is_same<A, PkF>::value) {
            if constexpr (REIN) {
                const ulonglong2 c = ld4(sm.s4 + i);
                const pk B = ld2(sm.s2 + i);
#pragma unroll
                for (int u = 0; u < NR; ++u) {
                    const pk nd = pk_fma(c.x, x[u], c.y);  // -(K + A (1 - x))
                    w[0][u] = pk_fma(B, w[0][u], pk_mul(nd, w[1][u]));
                    w[1][u] = pk_add(w[1][u], w[0][u]);
                }
            } else if constexpr (MODE == kSpin0) {
                const pk a = ld2(sm.s2 + i);
#pragma unroll
                for (int u = 0; u < NR; ++u) w[NW][u] = pk_fma(pk_mul(a, x[u]), w[1 - NW][u], w[NW][u]);
            } else {
                const ulonglong2 c = ld4(sm.s4 + i);
#pragma unroll
                for (int u = 0; u < NR; ++u) w[NW][u] = pk_fma(pk_fma(c.x, x[u], c.y), w[1 - NW][u], w[NW][u]);
            }
        } else {
            if constexpr (MODE == kSpin0) {
                const ulonglong2 c = ld4(sm.s4 + i);
#pragma unroll
                for (int u = 0; u < NR; ++u) {
                    const D2 ax = d2_mul(D2{c.x, c.y}, D2{x[u], xl[u]});
                    w[NW][u] = d2_fma(ax, w[1 - NW][u], w[NW][u]);
                }
            } else {
                const ulonglong2 c = ld4(sm.s4 + i);
                const float2 al = sm.s2[i];
#pragma unroll
                for (int u = 0; u < NR; ++u) {
                    const float2 xv = pk_get(x[u]);
                    const df32 ax = df_mul(df32{al.x, al.y}, df32{xv.x, xv.y});
                    const D2 y = d2_add_u(D2{pk_make(ax.h, ax.h), pk_make(ax.l, ax.l)}, D2{c.x, c.y});
                    w[NW][u] = d2_fma(y, w[1 - NW][u], w[NW][u]);
                }
            }
        }
    }
    // rescale the states whose newest value (word NW; Reinsch: w[1]) has grown past 2^20 (2^-40 at E = -1):
    // legendre values stay below one over much of the sphere, so a threshold of 2^60 kept most rings scaled
    template <int NW> __device__ __forceinline__ void rescale()
    {
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            typename A::S a, b;
            A::get(w[REIN ? 1 : NW][u], a, b);
            const bool ga = Ea[u] < 0 && A::mag(a) > kUpF, gb = Eb[u] < 0 && A::mag(b) > kUpF;
            const pk f = pk_make(ga ? kSmallF : 1.f, gb ? kSmallF : 1.f);
            w[0][u] = A::vscale(w[0][u], f);
            w[1][u] = A::vscale(w[1][u], f);
            Ea[u] += ga ? 1 : 0;
            Eb[u] += gb ? 1 : 0;
        }
    }
    static __device__ __forceinline__ float fac(int E) { return E == 0 ? 1.0f : (E == -1 ? kSmallF : 0.0f); }
    __device__ __forceinline__ pk factor(int u) const { return pk_make(fac(Ea[u]), fac(Eb[u])); }
    __device__ __forceinline__ bool any_scaled() const
    {
        bool sc = false;
#pragma unroll
        for (int u = 0; u < NR; ++u) sc = sc || Ea[u] != 0 || Eb[u] != 0;
        return __any_sync(0xffffffffu, sc);
    }
};

// 1 / (c.x + c.y) rounded to FP32 (the residual of the high word's reciprocal with the low word included)
__device__ __forceinline__ float inverse(float2 c)
{
    const float r = __frcp_rn(c.x);
    return __fmaf_rn(r, __fmaf_rn(-c.y, r, __fmaf_rn(-c.x, r, 1.f)), r);
}

// sign sigma of the degree dl = l - lf (plain form); rel = (-1)^dl
__device__ __forceinline__ float sigma_of(int dl) { return (dl & 2) ? 1.f : -1.f; }

// coefficient pair arrays of one degree: spin s four pairs, spin 0 / gradient-only two
template <int MODE> constexpr int kNC = MODE == kSpinS ? 4 : 2;

// ---------------------------------------------------------------- forward
// The prepared (scaled) coefficient of a degree: PkF from the a_lm themselves (c: the monic
// scale times the order weight), PkD from the prepared df32 table.
template <class A, int MODE> struct Coef {
    typename A::S ar, ai, br, bi;
};

// c (a + b) for c = c.x + c.y, one rounding (to within 2^-22 of a tie): the sum as a two-sum pair
__device__ __forceinline__ float scaled_sum(float2 c, float a, float b)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return __fmaf_rn(c.x, s, __fmaf_rn(c.x, e, c.y * s));
}

template <class A, int MODE>
__device__ __forceinline__ Coef<A, MODE> load_coef(const void *src, int64_t nalm, int64_t idx, float2 c, bool m0, float sgs)
{
    Coef<A, MODE> k;
    if constexpr (std::is_same<A, PkF>::value) {
        float2 g = __ldg((const float2 *)src + idx);
        if (m0) g.y = 0.f;
        if constexpr (MODE == kSpinS) {
            float2 q = __ldg((const float2 *)src + nalm + idx);
            if (m0) q.y = 0.f;
            k.ar = scaled_sum(c, g.x, -q.y);
            k.ai = scaled_sum(c, g.y, q.x);
            k.br = sgs * scaled_sum(c, g.x, q.y);
            k.bi = sgs * scaled_sum(c, q.x, -g.y);
        } else {
            k.ar = __fmaf_rn(c.x, g.x, c.y * g.x);
            k.ai = __fmaf_rn(c.x, g.y, c.y * g.y);
            k.br = k.ar;
            k.bi = k.ai;
        }
    } else {
        const float4 a = __ldg((const float4 *)src + idx);
        k.ar = {a.x, a.y};
        k.ai = {a.z, a.w};
        k.br = k.ar;
        k.bi = k.ai;
        if constexpr (MODE == kSpinS) {
            const float4 b = __ldg((const float4 *)src + nalm + idx);
            k.br = {b.x, b.y};
            k.bi = {b.z, b.w};
        }
    }
    return k;
}

// pairs of one degree: spin s (a, rel a) re, im, (rel b, b) re, im; otherwise (a, a) re, im; times sg
template <class A, int MODE>
__device__ __forceinline__ void coef_pairs(const Coef<A, MODE> &k, float sg, float rel, typename A::V *out)
{
    if constexpr (MODE == kSpinS) {
        out[0] = A::make(A::ssgn(k.ar, sg), A::ssgn(k.ar, sg * rel));
        out[1] = A::make(A::ssgn(k.ai, sg), A::ssgn(k.ai, sg * rel));
        out[2] = A::make(A::ssgn(k.br, sg * rel), A::ssgn(k.br, sg));
        out[3] = A::make(A::ssgn(k.bi, sg * rel), A::ssgn(k.bi, sg));
    } else {
        out[0] = A::make(A::ssgn(k.ar, sg), A::ssgn(k.ar, sg));
        out[1] = A::make(A::ssgn(k.ai, sg), A::ssgn(k.ai, sg));
    }
}

// the staged pairs of one degree and map, by 16-byte loads
template <int NC> __device__ __forceinline__ void load_pairs(const pk *c, pk (&k)[NC])
{
#pragma unroll
    for (int q = 0; q < NC; q += 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(c + q);
        k[q] = v.x;
        k[q + 1] = v.y;
    }
}
template <int NC> __device__ __forceinline__ void load_pairs(const D2 *c, D2 (&k)[NC])
{
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(c + q);
        k[q] = {v.x, v.y};
    }
}

// bytes of shared memory per warp: step entries, then (forward) coefficient pairs
template <class A, int MODE, int NM> __host__ __device__ constexpr size_t fwd_pk_smem()
{
    return kStage * (sizeof(float4) + sizeof(float2) + NM * kNC<MODE> * sizeof(typename A::V));
}

template <class A, int MODE, int NM, int NR>
struct FwdSums {
    // spin s: (north +m, south +m) re, im, (south -m, north -m) re, im;
    // otherwise the pair's sums over rel = +1 degrees re, im, rel = -1 degrees re, im
    typename A::V s[NM][NR][4];
};

template <class A, int MODE, bool REIN, int NR, int NM, bool SCALED>
__device__ __forceinline__ void fwd_pk_block(Pairs<A, MODE, REIN, NR> &st, FwdSums<A, MODE, NM, NR> &acc,
                                             const StageMem &sm, const typename A::V *cf, int i0)
{
    using V = typename A::V;
    pk f[NR];
    if (SCALED) {
#pragma unroll
        for (int u = 0; u < NR; ++u) f[u] = st.factor(u);
    }
#pragma unroll
    for (int j = 0; j < kBlk; ++j) {
        if (j & 1) st.template advance<1>(sm, i0 + j);
        else st.template advance<0>(sm, i0 + j);
        if (SCALED && (j == 3 || j == 7)) {
            st.template rescale<1>();
#pragma unroll
            for (int u = 0; u < NR; ++u) f[u] = st.factor(u);
        }
        V v[NR];
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            v[u] = st.w[REIN ? 1 : (j & 1)][u];
            if (SCALED) v[u] = A::vscale(v[u], f[u]);
        }
#pragma unroll
        for (int b = 0; b < NM; ++b) {
            V k[kNC<MODE>];
            load_pairs(cf + ((i0 + j) * NM + b) * kNC<MODE>, k);
#pragma unroll
            for (int q = 0; q < kNC<MODE>; ++q) {
                const int t = MODE == kSpinS ? q : q + 2 * (j & 1);
#pragma unroll
                for (int u = 0; u < NR; ++u) acc.s[b][u][t] = A::mac(acc.s[b][u][t], k[q], v[u]);
            }
        }
    }
}

template <class A, int MODE, bool REIN, int NR, int NM>
__device__ __forceinline__ void fwd_pk_body(const void *__restrict__ src, const void *__restrict__ rec,
                                            const RingTab &rt, typename A::C2 *__restrict__ ring, int lmax, int mmax,
                                            int spin, int ntheta, int nnorth, int64_t nalm, int64_t ring_stride,
                                            float wpos, bool ring_dd, const CkTab &ck, int wb, unsigned char *smem)
{
    using V = typename A::V;
    using S = typename A::S;
    constexpr int RPT = Pairs<A, MODE, REIN, NR>::RPT;
    constexpr bool F32 = std::is_same<A, PkF>::value;
    const int lane = threadIdx.x & 31;
    const int m = blockIdx.y;
    const int s = MODE == kSpin0 ? 0 : spin;
    const int l0 = m > s ? m : s;
    const int lf = l0 + 1;
    const int64_t base = alm_base(lmax, m);
    const int64_t mstride = (int64_t)(MODE == kSpinS ? 2 : 1) * nalm;  // one map's a_lm
    const float wm = F32 ? (m > 0 ? wpos : 1.f) : 1.f;
    const float sgs = (s & 1) ? -1.f : 1.f;
    const int r0 = wb + lane;

    StageMem sm;
    sm.s4 = reinterpret_cast<float4 *>(smem);
    V *cf = reinterpret_cast<V *>(sm.s4 + kStage);
    sm.s2 = reinterpret_cast<float2 *>(cf + kStage * NM * kNC<MODE>);

    FwdSums<A, MODE, NM, NR> acc;
#pragma unroll
    for (int b = 0; b < NM; ++b)
#pragma unroll
        for (int u = 0; u < NR; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc.s[b][u][q] = A::zero();

    Pairs<A, MODE, REIN, NR> st;
    st.geom(rt, r0, nnorth);
    const int K = ck_interval(ck, m);
    const int nck = ck_count(lmax, lf, K);
    const int ndeg = lmax + 1 - lf;  // degrees after l0
    const int64_t ckrow = __ldg(ck.base + m) - nnorth;  // row of the start values
    int kj = 0x7fff;
    if (lane < RPT && wb + 32 * lane < nnorth) kj = __ldg(ck.kstart + (int64_t)m * ck.ngrp + (wb >> 5) + lane);
    kj = __reduce_min_sync(0xffffffffu, kj);
    bool scaled = false;
    if (kj == 0) {  // degree l0 itself (rel = -1): from the start values
        scaled = st.restart(ck, ckrow, r0, nnorth, 1.f, 1.f);
#pragma unroll
        for (int b = 0; b < NM; ++b) {
            // c_{l0} = 1: the coefficient in the plain normalisation serves both forms
            const Coef<A, MODE> k = load_coef<A, MODE>((const char *)src + b * mstride * sizeof(float2), nalm, base + l0,
                                                       make_float2(wm, 0.f), m == 0, sgs);
            V c[kNC<MODE>];
            coef_pairs<A, MODE>(k, 1.f, -1.f, c);
#pragma unroll
            for (int u = 0; u < NR; ++u) {
                const V v = A::vscale(st.w[1][u], st.factor(u));
#pragma unroll
                for (int q = 0; q < kNC<MODE>; ++q) {
                    const int t = MODE == kSpinS ? q : q + 2;
                    acc.s[b][u][t] = A::mac(acc.s[b][u][t], c[q], v);
                }
            }
        }
    }
    const int d0 = kj * K;
    for (int cs = d0 & ~(kStage - 1); cs < ndeg; cs += kStage) {
        __syncwarp();
#pragma unroll 1
        for (int i = lane; i < kStage; i += 32) {
            const int dl = cs + i;
            const bool live = dl < ndeg;
            const int64_t idx = base + lf + dl;
            stage_step<A, MODE, REIN>(sm, i, rec, idx, live, dl);
            const float rel = (dl & 1) ? -1.f : 1.f, sg = REIN ? 1.f : sigma_of(dl);
            float2 c = F32 && !REIN && live ? __ldg(ck.cs + idx) : make_float2(1.f, 0.f);
            c.x *= wm;
            c.y *= wm;
#pragma unroll
            for (int b = 0; b < NM; ++b) {
                Coef<A, MODE> k = {};
                if (live)
                    k = load_coef<A, MODE>((const char *)src + b * mstride * sizeof(float2), nalm, idx, c, m == 0, sgs);
                V pr[kNC<MODE>];
                coef_pairs<A, MODE>(k, sg, rel, pr);
#pragma unroll
                for (int q = 0; q < kNC<MODE>; ++q) cf[(i * NM + b) * kNC<MODE> + q] = pr[q];
            }
        }
        __syncwarp();
        const int de = min(cs + kStage, ndeg);
#pragma unroll 1
        for (int d = max(cs, d0); d < de; d += kBlk) {
            if ((d & (K - 1)) == 0 && d != 0) {
                const int k = d / K;
                if (k <= nck) {
                    float i0 = 1.f, i1 = 1.f;
                    if (F32 && !REIN) {
                        i0 = inverse(__ldg(ck.cs + base + lf + d - 2));
                        i1 = inverse(__ldg(ck.cs + base + lf + d - 1));
                    }
                    scaled = st.restart(ck, ckrow + (int64_t)k * nnorth, r0, nnorth, i0, i1);
                }
            }
            st.renorm();
            if constexpr (!F32) {
#pragma unroll
                for (int u = 0; u < NR; ++u)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc.s[0][u][q] = A::norm(acc.s[0][u][q]);
            }
            if (scaled) {
                fwd_pk_block<A, MODE, REIN, NR, NM, true>(st, acc, sm, cf, d - cs);
                scaled = st.any_scaled();
            } else {
                fwd_pk_block<A, MODE, REIN, NR, NM, false>(st, acc, sm, cf, d - cs);
            }
        }
    }

    // write: spin 0 column m; spin s columns mmax + m and mmax - m, with the minus sign
    const float s0 = ((lf - m) & 1) ? -1.f : 1.f, ms0 = -s0;
    auto put = [&](typename A::C2 *col, int j, S re, float sr, S im, float si) {
        re = A::ssgn(re, sr);
        im = A::ssgn(im, si);
        if constexpr (!F32) {
            if (ring_dd) {
                reinterpret_cast<float4 *>(col)[j] = make_float4(re.h, re.l, im.h, im.l);
                return;
            }
        }
        col[j] = mkc(A::out(re), A::out(im));
    };
#pragma unroll
    for (int b = 0; b < NM; ++b) {
        typename A::C2 *rb = ring + b * ring_stride;
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            S r[4][2];
#pragma unroll
            for (int q = 0; q < 4; ++q) A::get(acc.s[b][u][q], r[q][0], r[q][1]);
            if constexpr (MODE == kSpin0) {
                typename A::C2 *col = rb + (int64_t)m * ntheta;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int jn = r0 + 32 * (2 * u + q), js = ntheta - 1 - jn;
                    if (jn >= nnorth) continue;
                    put(col, jn, A::sadd(r[0][q], r[2][q]), 1.f, A::sadd(r[1][q], r[3][q]), 1.f);
                    if (js != jn) put(col, js, A::ssub(r[0][q], r[2][q]), s0, A::ssub(r[1][q], r[3][q]), s0);
                }
            } else {
                const int jn = r0 + 32 * u, js = ntheta - 1 - jn;
                if (jn >= nnorth) continue;
                typename A::C2 *colp = rb + (int64_t)(mmax + m) * ntheta, *colq = rb + (int64_t)(mmax - m) * ntheta;
                if constexpr (MODE == kSpinS) {
                    put(colp, jn, r[0][0], -1.f, r[1][0], -1.f);
                    if (js != jn) put(colp, js, r[0][1], ms0, r[1][1], ms0);
                    if (m > 0) {
                        put(colq, jn, r[2][1], -1.f, r[3][1], -1.f);
                        if (js != jn) put(colq, js, r[2][0], ms0, r[3][0], ms0);
                    }
                } else {
                    // b = (-1)^s conj a: the four spin-s sums from the sums of a s-lambda and a (-s)lambda
                    // over rel = +1 (r[0], r[1]) and rel = -1 (r[2], r[3]) degrees
                    put(colp, jn, A::sadd(r[0][0], r[2][0]), -1.f, A::sadd(r[1][0], r[3][0]), -1.f);
                    if (js != jn) put(colp, js, A::ssub(r[0][1], r[2][1]), ms0, A::ssub(r[1][1], r[3][1]), ms0);
                    if (m > 0) {
                        put(colq, jn, A::sadd(r[0][1], r[2][1]), -sgs, A::sadd(r[1][1], r[3][1]), sgs);
                        if (js != jn)
                            put(colq, js, A::ssub(r[0][0], r[2][0]), sgs * ms0, A::ssub(r[1][0], r[3][0]), -(sgs * ms0));
                    }
                }
            }
        }
    }
}

// src: PkF the a_lm of the call (NM maps), PkD the prepared df32 coefficients.
// rec_s: step table of Reinsch's form; rec_a: df32 (alpha, tau) table.
template <class A, int MODE, int NR, int NM>
__global__ void __launch_bounds__(128) k_leg_fwd_pk(const void *__restrict__ src, const void *__restrict__ rec_s,
                                                    const void *__restrict__ rec_a, RingTab rt,
                                                    typename A::C2 *__restrict__ ring, int lmax, int mmax, int spin,
                                                    int ntheta, int nnorth, int64_t nalm, int64_t ring_stride,
                                                    float wpos, int ring_dd, CkTab ck)
{
    extern __shared__ __align__(16) unsigned char pk_smem[];
    constexpr int RPT = MODE == kSpin0 ? 2 * NR : NR;
    const int wid = threadIdx.x >> 5;
    const int wb = (blockIdx.x * (blockDim.x >> 5) + wid) * 32 * RPT;  // first ring of the warp
    if (wb >= nnorth) return;
    unsigned char *mem = pk_smem + wid * fwd_pk_smem<A, MODE, NM>();
    if constexpr (std::is_same<A, PkF>::value) {
        if (wb < ck.jb)
            return fwd_pk_body<A, MODE, true, NR, NM>(src, rec_s, rt, ring, lmax, mmax, spin, ntheta, nnorth, nalm,
                                                      ring_stride, wpos, false, ck, wb, mem);
    }
    fwd_pk_body<A, MODE, false, NR, NM>(src, rec_a, rt, ring, lmax, mmax, spin, ntheta, nnorth, nalm, ring_stride, wpos,
                                        ring_dd != 0, ck, wb, mem);
}

// ---------------------------------------------------------------- adjoint
// Per degree a lane adds its rings' products into kVals sums (spin s: U.re, U.im, V.re, V.im; otherwise
// re, im) and stores them in its row of the warp's shared memory; after 8 degrees the warp adds the 32
// rows column-wise: a lane reads 16-byte quads of some of the rows (spin s 8 rows of one
// degree's quad, otherwise 4 rows of two degrees' quad), adds them and combines with the lanes of
// the other rows by a transpose-reduce of the quad.
// Row stride: NV + 4 floats (quads of consecutive rows in distinct banks for 16-byte accesses); PkD keeps
// the low words in a second plane.
template <int MODE> constexpr int kVals = MODE == kSpinS ? 4 : 2;
template <int MODE> constexpr int kRow = kBlk * kVals<MODE> + 4;
template <class A, int MODE> __host__ __device__ constexpr size_t adj_pk_smem()
{
    return kStage * (sizeof(float4) + sizeof(float2)) +
           (std::is_same<A, PkF>::value ? 1 : 2) * 32 * kRow<MODE> * sizeof(float);
}

template <class A> struct Quad {
    typename A::V a, b;  // values 0, 1 and 2, 3
};
__device__ __forceinline__ void quad_load(Quad<PkF> &q, const float *p, int)
{
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
    q.a = v.x;
    q.b = v.y;
}
__device__ __forceinline__ void quad_load(Quad<PkD> &q, const float *p, int plane)
{
    const ulonglong2 h = *reinterpret_cast<const ulonglong2 *>(p), l = *reinterpret_cast<const ulonglong2 *>(p + plane);
    q.a = {h.x, l.x};
    q.b = {h.y, l.y};
}
__device__ __forceinline__ pk vadd(pk a, pk b) { return pk_add(a, b); }
__device__ __forceinline__ D2 vadd(D2 a, D2 b) { return d2_add_u(a, b); }
__device__ __forceinline__ float sel(bool c, float a, float b) { return c ? a : b; }
__device__ __forceinline__ df32 sel(bool c, df32 a, df32 b) { return {c ? a.h : b.h, c ? a.l : b.l}; }

// Adds the value val of degree l, component c (spin s: U.re, U.im, V.re, V.im with `other` the V / U of the
// same degree; otherwise re, im) times wl (order weight, monic scale, sigma) into a_lm / G, C.
// fx: deterministic plans, fixed-point sums in units of 1 / fxu.
template <class A, int MODE>
__device__ __forceinline__ void put_alm(typename A::S val, typename A::S other, int c, int64_t i, int64_t nalm, bool m0,
                                        double wl, float wlf, float sgs, typename A::R *out, unsigned long long *fx,
                                        double fxu)
{
    int64_t dst = 2 * i + c;
    bool drop = m0 && c == 1;
    if constexpr (MODE == kSpinS) {
        //   G.re = -(U.re + sgs V.re)/2   G.im = -(U.im - sgs V.im)/2
        //   C.re = -(U.im + sgs V.im)/2   C.im =  (U.re - sgs V.re)/2
        drop = m0 && (c == 1 || c == 2);
        if (c == 0) val = A::ssgn(A::sadd(val, A::ssgn(other, sgs)), -0.5f);
        else if (c == 1) val = A::ssgn(A::sadd(val, A::ssgn(other, -sgs)), -0.5f);
        else if (c == 2) { val = A::ssgn(A::sadd(other, A::ssgn(val, -sgs)), 0.5f); dst = 2 * (nalm + i) + 1; }
        else { val = A::ssgn(A::sadd(other, A::ssgn(val, sgs)), -0.5f); dst = 2 * (nalm + i); }
    }
    if (drop) return;
    if constexpr (std::is_same<A, PkF>::value) {
        if (fx) atomicAdd(fx + dst, (unsigned long long)__float2ll_rn(val * wlf * (float)fxu));
        else atomicAdd(out + dst, val * wlf);
    } else {
        const double v = A::out(val) * wl;
        if (fx) atomicAdd(fx + dst, (unsigned long long)__double2ll_rn(v * fxu));
        else atomicAdd(out + dst, v);
    }
}

template <class A, int MODE, bool REIN, int NR, bool SCALED>
__device__ __forceinline__ void adj_pk_block(Pairs<A, MODE, REIN, NR> &st,
                                             const typename A::V (&in)[NR][4], const StageMem &sm, int i0, float *row,
                                             int plane)
{
    using V = typename A::V;
    using S = typename A::S;
    pk f[NR];
    if (SCALED) {
#pragma unroll
        for (int u = 0; u < NR; ++u) f[u] = st.factor(u);
    }
#pragma unroll
    for (int j = 0; j < kBlk; ++j) {
        if (j & 1) st.template advance<1>(sm, i0 + j);
        else st.template advance<0>(sm, i0 + j);
        if (SCALED && (j == 3 || j == 7)) {
            st.template rescale<1>();
#pragma unroll
            for (int u = 0; u < NR; ++u) f[u] = st.factor(u);
        }
        V t[kVals<MODE>];
#pragma unroll
        for (int q = 0; q < kVals<MODE>; ++q) t[q] = A::zero();
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            V v = st.w[REIN ? 1 : (j & 1)][u];
            if (SCALED) v = A::vscale(v, f[u]);
#pragma unroll
            for (int q = 0; q < kVals<MODE>; ++q)
                t[q] = A::mac(t[q], in[u][MODE == kSpinS ? q : q + 2 * (j & 1)], v);
        }
        // spin s: U = lo + rel hi, V = rel lo + hi; otherwise lo + hi
        S o[kVals<MODE>];
#pragma unroll
        for (int q = 0; q < kVals<MODE>; ++q) {
            S a, b;
            A::get(t[q], a, b);
            if (MODE == kSpinS && (j & 1)) o[q] = q < 2 ? A::ssub(a, b) : A::ssub(b, a);
            else o[q] = A::sadd(a, b);
        }
        float *p = row + j * kVals<MODE>;
        if constexpr (std::is_same<A, PkF>::value) {
            if constexpr (MODE == kSpinS) *reinterpret_cast<float4 *>(p) = make_float4(o[0], o[1], o[2], o[3]);
            else *reinterpret_cast<float2 *>(p) = make_float2(o[0], o[1]);
        } else {
            if constexpr (MODE == kSpinS) {
                *reinterpret_cast<float4 *>(p) = make_float4(o[0].h, o[1].h, o[2].h, o[3].h);
                *reinterpret_cast<float4 *>(p + plane) = make_float4(o[0].l, o[1].l, o[2].l, o[3].l);
            } else {
                *reinterpret_cast<float2 *>(p) = make_float2(o[0].h, o[1].h);
                *reinterpret_cast<float2 *>(p + plane) = make_float2(o[0].l, o[1].l);
            }
        }
    }
}

template <class A, int MODE, bool REIN, int NR>
__device__ __forceinline__ void adj_pk_body(const typename A::C2 *__restrict__ ring, const void *__restrict__ rec,
                                            const RingTab &rt, typename A::C2 *__restrict__ alm, int lmax, int mmax,
                                            int spin, int ntheta, int nnorth, int64_t nalm, double wpos,
                                            const double *__restrict__ scale, unsigned long long *fx,
                                            const double *__restrict__ fxs, const CkTab &ck, int wb,
                                            unsigned char *smem)
{
    using V = typename A::V;
    using S = typename A::S;
    using R = typename A::R;
    constexpr int RPT = Pairs<A, MODE, REIN, NR>::RPT;
    constexpr bool F32 = std::is_same<A, PkF>::value;
    constexpr int NVAL = kVals<MODE>, ROW = kRow<MODE>, plane = 32 * ROW;
    const int lane = threadIdx.x & 31;
    const int m = blockIdx.y;
    const int s = MODE == kSpin0 ? 0 : spin;
    const int l0 = m > s ? m : s;
    const int lf = l0 + 1;
    const int64_t base = alm_base(lmax, m);
    const float sgs = (s & 1) ? -1.f : 1.f;
    const float s0 = ((lf - m) & 1) ? -1.f : 1.f;
    const double wm = (m > 0 ? wpos : 1.0) * (MODE == kGrad ? -0.5 : 1.0);
    const float wmf = (float)wm;
    const double fxu = fx ? fxs[1 + m] : 0.0;
    const int r0 = wb + lane;
    R *out = reinterpret_cast<R *>(alm);

    StageMem sm;
    sm.s4 = reinterpret_cast<float4 *>(smem);
    sm.s2 = reinterpret_cast<float2 *>(sm.s4 + kStage);
    float *red = reinterpret_cast<float *>(sm.s2 + kStage);
    float *row = red + lane * ROW;

    // inputs.  spin s: (H_m(N), s0 H_m(S)) re, im and (s0 H_-m(S), H_-m(N)) re, im; spin 0: per ring H_N + H_S or
    // H_N - H_S for rel = +1 then rel = -1 degrees; gradient-only: see AdjIn of legendre.cu
    V in[NR][4];
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        if constexpr (MODE == kSpin0) {
            S e[2][4];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int jn = r0 + 32 * (2 * u + q), js = ntheta - 1 - jn;
                typename A::C2 n = mkc(R(0), R(0)), t = n;
                if (jn < nnorth) {
                    n = ring[(int64_t)m * ntheta + jn];
                    if (js != jn) t = ring[(int64_t)m * ntheta + js];
                }
                const S nr = A::in(n.x), ni = A::in(n.y), sr = A::in(t.x), si = A::in(t.y);
                // rel = s0 (-1)^(l - m): the sum for s0 = +1, the difference for s0 = -1
                const S pr = A::sadd(nr, sr), pi = A::sadd(ni, si), dr = A::ssub(nr, sr), di = A::ssub(ni, si);
                e[q][0] = s0 > 0 ? pr : dr; e[q][1] = s0 > 0 ? pi : di;
                e[q][2] = s0 > 0 ? dr : pr; e[q][3] = s0 > 0 ? di : pi;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) in[u][q] = A::make(e[0][q], e[1][q]);
        } else {
            const int jn = r0 + 32 * u, js = ntheta - 1 - jn;
            typename A::C2 hn = mkc(R(0), R(0)), hs = hn, gn = hn, gs = hn;
            if (jn < nnorth) {
                const typename A::C2 *cp = ring + (int64_t)(mmax + m) * ntheta, *cq = ring + (int64_t)(mmax - m) * ntheta;
                hn = cp[jn];
                gn = cq[jn];
                if (js != jn) { hs = cp[js]; gs = cq[js]; }
            }
            const S hnr = A::in(hn.x), hni = A::in(hn.y), hsr = A::ssgn(A::in(hs.x), s0), hsi = A::ssgn(A::in(hs.y), s0);
            const S gnr = A::in(gn.x), gni = A::in(gn.y), gsr = A::ssgn(A::in(gs.x), s0), gsi = A::ssgn(A::in(gs.y), s0);
            if constexpr (MODE == kSpinS) {
                in[u][0] = A::make(hnr, hsr);
                in[u][1] = A::make(hni, hsi);
                in[u][2] = A::make(gsr, gnr);
                in[u][3] = A::make(gsi, gni);
            } else {
                const S agsr = A::ssgn(gsr, sgs), agsi = A::ssgn(gsi, sgs), agnr = A::ssgn(gnr, sgs), agni = A::ssgn(gni, sgs);
                in[u][0] = A::make(A::sadd(hnr, agsr), A::sadd(hsr, agnr));
                in[u][1] = A::make(A::ssub(hni, agsi), A::ssub(hsi, agni));
                in[u][2] = A::make(A::ssub(hnr, agsr), A::ssub(agnr, hsr));
                in[u][3] = A::make(A::sadd(hni, agsi), A::ssgn(A::sadd(hsi, agni), -1.f));
            }
        }
    }

    Pairs<A, MODE, REIN, NR> st;
    st.geom(rt, r0, nnorth);
    const int K = ck_interval(ck, m);
    const int nck = ck_count(lmax, lf, K);
    const int ndeg = lmax + 1 - lf;
    const int64_t ckrow = __ldg(ck.base + m) - nnorth;
    int kj = 0x7fff;
    if (lane < RPT && wb + 32 * lane < nnorth) kj = __ldg(ck.kstart + (int64_t)m * ck.ngrp + (wb >> 5) + lane);
    kj = __reduce_min_sync(0xffffffffu, kj);
    bool scaled = false;
    if (kj == 0) {  // degree l0 (rel = -1, c_{l0} = 1) from the start values: one reduction by shuffles
        scaled = st.restart(ck, ckrow, r0, nnorth, 1.f, 1.f);
        V t[NVAL];
#pragma unroll
        for (int q = 0; q < NVAL; ++q) t[q] = A::zero();
#pragma unroll
        for (int u = 0; u < NR; ++u) {
            const V v = A::vscale(st.w[1][u], st.factor(u));
#pragma unroll
            for (int q = 0; q < NVAL; ++q) t[q] = A::mac(t[q], in[u][MODE == kSpinS ? q : q + 2], v);
        }
        S o[NVAL];
#pragma unroll
        for (int q = 0; q < NVAL; ++q) {
            S a, b;
            A::get(t[q], a, b);
            o[q] = MODE != kSpinS ? A::sadd(a, b) : (q < 2 ? A::ssub(a, b) : A::ssub(b, a));
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) o[q] = A::sadd(o[q], A::shfl(o[q], off));
        }
        if (lane < NVAL) {
            S v = o[0], w = o[0];
            if constexpr (MODE == kSpinS) {
                v = lane == 0 ? o[0] : lane == 1 ? o[1] : lane == 2 ? o[2] : o[3];
                w = lane == 0 ? o[2] : lane == 1 ? o[3] : lane == 2 ? o[0] : o[1];
            } else {
                v = lane == 0 ? o[0] : o[1];
            }
            put_alm<A, MODE>(v, w, lane, base + l0, nalm, m == 0, wm, wmf, sgs, out, fx, fxu);
        }
    }
    const int d0 = kj * K;
    for (int cs = d0 & ~(kStage - 1); cs < ndeg; cs += kStage) {
        __syncwarp();
#pragma unroll
        for (int i = lane; i < kStage; i += 32)
            stage_step<A, MODE, REIN>(sm, i, rec, base + lf + cs + i, cs + i < ndeg, cs + i);
        __syncwarp();
        const int de = min(cs + kStage, ndeg);
#pragma unroll 1
        for (int d = max(cs, d0); d < de; d += kBlk) {
            if ((d & (K - 1)) == 0 && d != 0) {
                const int k = d / K;
                if (k <= nck) {
                    float i0 = 1.f, i1 = 1.f;
                    if (F32 && !REIN) {
                        i0 = inverse(__ldg(ck.cs + base + lf + d - 2));
                        i1 = inverse(__ldg(ck.cs + base + lf + d - 1));
                    }
                    scaled = st.restart(ck, ckrow + (int64_t)k * nnorth, r0, nnorth, i0, i1);
                }
            }
            st.renorm();
            if (scaled) {
                adj_pk_block<A, MODE, REIN, NR, true>(st, in, sm, d - cs, row, plane);
                scaled = st.any_scaled();
            } else {
                adj_pk_block<A, MODE, REIN, NR, false>(st, in, sm, d - cs, row, plane);
            }
            __syncwarp();
            // column sums: lanes of one quad column are NQ apart
            constexpr int NQ = kBlk * NVAL / 4, NG = 32 / NQ, NROW = 32 / NG;  // quads, row groups, rows a lane adds
            const int q = lane & (NQ - 1), g = lane / NQ;
            Quad<A> sum;
            quad_load(sum, red + g * NROW * ROW + 4 * q, plane);
#pragma unroll
            for (int i = 1; i < NROW; ++i) {
                Quad<A> t;
                quad_load(t, red + (g * NROW + i) * ROW + 4 * q, plane);
                sum.a = vadd(sum.a, t.a);
                sum.b = vadd(sum.b, t.b);
            }
            __syncwarp();  // the rows are rewritten by the next block
            S v0, v1, v2, v3;
            A::get(A::norm(sum.a), v0, v1);
            A::get(A::norm(sum.b), v2, v3);
            // transpose-reduce: bit 4 of the lane keeps values 2, 3; bit 3 keeps the odd one of the two
            const bool up = lane & 16, uq = lane & 8;
            S ka = sel(up, v2, v0), kb = sel(up, v3, v1);
            ka = A::sadd(ka, A::shfl(sel(up, v0, v2), 16));
            kb = A::sadd(kb, A::shfl(sel(up, v1, v3), 16));
            S v = sel(uq, kb, ka);
            v = A::sadd(v, A::shfl(sel(uq, ka, kb), 8));
            if constexpr (NQ == 4) v = A::sadd(v, A::shfl(v, 4));  // eight row groups: one more stage
            int j, c;
            if constexpr (NVAL == 4) {
                c = (up ? 2 : 0) + (uq ? 1 : 0);
                j = q;
            } else {  // quad q: degrees 2q (values 0, 1) and 2q + 1 (values 2, 3)
                c = uq ? 1 : 0;
                j = 2 * q + (up ? 1 : 0);
            }
            S other = v;
            if constexpr (MODE == kSpinS) other = A::shfl(v, 16);  // U <-> V of the same degree
            const int dl = d + j;
            if (dl < ndeg && (NQ == 8 || !(lane & 4))) {
                const int64_t i = base + lf + dl;
                double wl = 0.0;
                float wlf = wmf;
                if constexpr (F32) {
                    if (!REIN) wlf *= __ldg(ck.cs + i).x * sigma_of(dl);
                } else {
                    wl = wm * __ldg(scale + i) * (double)sigma_of(dl);
                }
                put_alm<A, MODE>(v, other, c, i, nalm, m == 0, wl, wlf, sgs, out, fx, fxu);
            }
        }
    }
}

template <class A, int MODE, int NR>
__global__ void __launch_bounds__(128) k_leg_adj_pk(const typename A::C2 *__restrict__ ring,
                                                    const void *__restrict__ rec_s, const void *__restrict__ rec_a,
                                                    RingTab rt, typename A::C2 *__restrict__ alm, int lmax, int mmax,
                                                    int spin, int ntheta, int nnorth, int64_t nalm, double wpos,
                                                    const double *__restrict__ scale, unsigned long long *fx,
                                                    const double *__restrict__ fxs, CkTab ck)
{
    extern __shared__ __align__(16) unsigned char pk_smem[];
    constexpr int RPT = MODE == kSpin0 ? 2 * NR : NR;
    const int wid = threadIdx.x >> 5;
    const int wb = (blockIdx.x * (blockDim.x >> 5) + wid) * 32 * RPT;
    if (wb >= nnorth) return;
    unsigned char *mem = pk_smem + wid * adj_pk_smem<A, MODE>();
    if constexpr (std::is_same<A, PkF>::value) {
        if (wb < ck.jb)
            return adj_pk_body<A, MODE, true, NR>(ring, rec_s, rt, alm, lmax, mmax, spin, ntheta, nnorth, nalm, wpos,
                                                  scale, fx, fxs, ck, wb, mem);
    }
    adj_pk_body<A, MODE, false, NR>(ring, rec_a, rt, alm, lmax, mmax, spin, ntheta, nnorth, nalm, wpos, scale, fx, fxs,
                                    ck, wb, mem);
}

// ---------------------------------------------------------------- launches
// CTAs of up to four warps (a warp works alone, so the CTA shape only packs them); grid.y = order, low
// orders (the longest) first.
struct PkShape {
    dim3 grid, block;
};
PkShape pk_shape(const Plan &p, int rpt)
{
    const int nw = (p.nnorth + 32 * rpt - 1) / (32 * rpt);
    const int chunks = (nw + 3) / 4;
    const int warps = (nw + chunks - 1) / chunks;
    return {dim3(chunks, p.mmax + 1), dim3(32 * warps)};
}

template <class A, int MODE, int NR, int NM>
cudaError_t fwd_pk(const Plan &p, const void *src, void *ring, double wpos, bool ring_dd, cudaStream_t st)
{
    const PkShape sh = pk_shape(p, MODE == kSpin0 ? 2 * NR : NR);
    const size_t smem = sh.block.x / 32 * fwd_pk_smem<A, MODE, NM>();
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_leg_fwd_pk<A, MODE, NR, NM>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_leg_fwd_pk<A, MODE, NR, NM><<<sh.grid, sh.block, smem, st>>>(
        src, p.rec_s, p.prec == LENS_FP32 ? p.rec_a : p.rec_a_df, p.rings, (typename A::C2 *)ring, p.lmax, p.mmax,
        p.spin, p.ntheta, p.nnorth, p.nalm, (int64_t)p.ncol * p.ntheta, (float)wpos, ring_dd ? 1 : 0, p.ck);
    return cudaGetLastError();
}

template <class A, int MODE, int NR>
cudaError_t adj_pk(const Plan &p, const void *ring, void *alm, double wpos, void *fx, cudaStream_t st)
{
    const PkShape sh = pk_shape(p, MODE == kSpin0 ? 2 * NR : NR);
    const size_t smem = sh.block.x / 32 * adj_pk_smem<A, MODE>();
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_leg_adj_pk<A, MODE, NR>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k_leg_adj_pk<A, MODE, NR><<<sh.grid, sh.block, smem, st>>>(
        (const typename A::C2 *)ring, p.rec_s, p.prec == LENS_FP32 ? p.rec_a : p.rec_a_df, p.rings,
        (typename A::C2 *)alm, p.lmax, p.mmax, p.spin, p.ntheta, p.nnorth, p.nalm, wpos, p.scale,
        (unsigned long long *)fx, p.fx_scale, p.ck);
    return cudaGetLastError();
}

template <class A, int NM>
cudaError_t fwd_pk_rpt(const Plan &p, int rpt, const void *src, void *ring, double wpos, bool ring_dd, cudaStream_t st)
{
    if (!p.spin) return rpt <= 2 ? fwd_pk<A, kSpin0, 1, NM>(p, src, ring, wpos, ring_dd, st) : fwd_pk<A, kSpin0, 2, NM>(p, src, ring, wpos, ring_dd, st);
    if constexpr (NM == 1) {
        if (p.grad) {
            if (rpt == 1) return fwd_pk<A, kGrad, 1, 1>(p, src, ring, wpos, ring_dd, st);
            return rpt == 2 ? fwd_pk<A, kGrad, 2, 1>(p, src, ring, wpos, ring_dd, st) : fwd_pk<A, kGrad, 4, 1>(p, src, ring, wpos, ring_dd, st);
        }
    }
    if constexpr (NM < 4) {
        if (rpt == 1) return fwd_pk<A, kSpinS, 1, NM>(p, src, ring, wpos, ring_dd, st);
        if (rpt == 2 || NM == 2) return fwd_pk<A, kSpinS, 2, NM>(p, src, ring, wpos, ring_dd, st);
    }
    if constexpr (NM == 1) return fwd_pk<A, kSpinS, 4, 1>(p, src, ring, wpos, ring_dd, st);
    return cudaErrorInvalidValue;
}

template <class A>
cudaError_t adj_pk_rpt(const Plan &p, int rpt, const void *ring, void *alm, double wpos, void *fx, cudaStream_t st)
{
    if (!p.spin) return rpt <= 2 ? adj_pk<A, kSpin0, 1>(p, ring, alm, wpos, fx, st) : adj_pk<A, kSpin0, 2>(p, ring, alm, wpos, fx, st);
    if (p.grad) {
        if (rpt == 1) return adj_pk<A, kGrad, 1>(p, ring, alm, wpos, fx, st);
        return rpt == 2 ? adj_pk<A, kGrad, 2>(p, ring, alm, wpos, fx, st) : adj_pk<A, kGrad, 4>(p, ring, alm, wpos, fx, st);
    }
    if (rpt == 1) return adj_pk<A, kSpinS, 1>(p, ring, alm, wpos, fx, st);
    return rpt == 2 ? adj_pk<A, kSpinS, 2>(p, ring, alm, wpos, fx, st) : adj_pk<A, kSpinS, 4>(p, ring, alm, wpos, fx, st);
}

}  // namespace
}  // namespace gsl
