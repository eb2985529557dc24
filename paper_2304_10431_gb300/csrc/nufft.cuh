// Non-uniform FFT steps (Sect. 3 "NUFFT": type 2 for the forward operator,
// type 1 for the adjoint) on the oversampled torus grid.
//
// Kernel: exponential of semicircle, psi(z) = exp(beta (sqrt(1 - (2z/W)^2) - 1))
// for |z| < W/2 (grid units), zero outside.  A point at grid coordinates
// (u, v) = (theta N1 / 2pi, phi N2 / 2pi) touches the W x W cells
// i0 + a, j0 + b with i0 = ceil(u - W/2), j0 = ceil(v - W/2), a, b < W:
//   type 2:  f = sum_ab psi(u - i0 - a) psi(v - j0 - b) g[i0 + a, j0 + b]
//   type 1:  g[i0 + a, j0 + b] += psi(u - i0 - a) psi(v - j0 - b) f
// The two use the same weights, so they are exact transposes.
//
// Points are prepared once per plan (Sect. 4: the geometry is reused): cell
// offset into the row-padded grid, fractional offsets (u - i0, v - j0) from
// FP64 coordinates, the spin phase e^{i s chi}, a permutation that sorts
// points by grid tile (of the first tap), within a tile by cell row and column where that pays (launch_prep_points), so that
// neighbouring threads share grid rows and cells, and the first sorted point of every tile.
// Interpolation runs one thread per sorted point and reads its taps
// through L1: sorted neighbours share rows, so the tile stays cached (staging
// the tile and its halo in shared memory first measured 1.36x slower for
// spin 0 at lmax 4096).  Sorted by row and column, and by aligned pairs (k_interp32): lmax 4096, 50M points, FP32, spin 0
// 1.17 -> 0.77 ms, spin 2 2.08 -> 1.56 ms.
// Spreading: FP64 plans with double-float weights and FP32 plans with W >= 8 (spin 0: W >= 10) or epsilon < 1e-5 by strips in
// registers (nufft_strip.cuh); the others one CTA per 32 x 32 tile: its points add their W x W taps into the tile and its halo, (32 + W - 1) x (32 + W - 1)
// integers held in shared memory, and the CTA then adds the non-zero cells into the grid with one global atomic each.
//
// Deterministic plans (LENS_DETERMINISTIC) spread in 64-bit fixed point: every
// tap value is scaled by a power of two 2^k and rounded to an integer, and the
// shared-memory and global atomics add integers, exactly and so in any order.
// k is chosen per call so that no cell can exceed 2^62: a cell receives at
// most Kmax points (the largest point count of a tile and its left, upper and
// upper-left neighbours, whose taps are the only ones that reach it), each
// contributing |x| psi psi <= max |x|.  A conversion pass then writes the
// grid in the plan's precision.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "pk.cuh"

namespace gsl {
namespace {

constexpr int kSpreadThreads = 64;
// FP64 tiles hold 64-bit cells (31 KB at W = 13, seven CTAs per SM): 256 threads keep
// more warps in flight per tile
constexpr int kSpreadThreads64 = 256;

// the ES kernel of tap offset z (FP64 plans)
template <typename T> __device__ __forceinline__ T es_kernel(T z, T twoW, T beta)
{
    const T t = z * twoW;
    const T q = T(1) - t * t;
    return q > T(0) ? exp(beta * (sqrt(q) - T(1))) : T(0);
}

// FP32 plans: the kernel weight of tap a by Horner's rule in t = 2 frac - (W - 1) from the plan's
// polynomial coefficients (W + 1 fused multiply-adds; interpolation and spreading read the same
// coefficients, so the pair stay exact transposes of each other)
template <int W> __device__ __forceinline__ float ker_poly(const KerPoly &kp, int a, float t)
{
    float acc = kp.c[a * (W + 2) + W + 1];
#pragma unroll
    for (int k = W; k >= 0; --k) acc = fmaf(acc, t, kp.c[a * (W + 2) + k]);
    return acc;
}

// fixed-point term: v 2^k (exact, 2^k a power of two) rounded to an integer
__device__ __forceinline__ unsigned long long to_fx(float v, float sc) { return (unsigned long long)__float2ll_rn(v * sc); }
__device__ __forceinline__ unsigned long long to_fx(double v, double sc)
{
    return (unsigned long long)__double2ll_rn(v * sc);
}

__device__ __forceinline__ df32 ld_df(const float2 *p)
{
    const float2 v = __ldg(p);
    return {v.x, v.y};
}
// double-float weights of sorted point p: theta tap a, phi tap b
template <int W> __device__ __forceinline__ const float *dd_weights(const double *wts, int64_t p)
{
    return reinterpret_cast<const float *>(wts) + p * dd_words(W);
}
template <int W> __device__ __forceinline__ df32 dd_theta(const float *w, int a)
{
    if ((W & 1) && a == W - 1) return ld_df(reinterpret_cast<const float2 *>(w + 2 * a));
    const float *q = w + 4 * (a >> 1) + (a & 1);
    return {__ldg(q), __ldg(q + 2)};
}
template <int W> __device__ __forceinline__ df32 dd_phi(const float *w, int b)
{
    return ld_df(reinterpret_cast<const float2 *>(w + 2 * W) + b);
}

// PRE: 0 evaluate the kernel, 1 read the double weights, 2 the double-float pairs
template <typename T, int W, int PRE>
__device__ __forceinline__ void tap_weights(T (&wa)[W], T (&wb)[W], const cplx<T> &f, const double *wts, int64_t p,
                                            T beta, const KerPoly &kp)
{
    if (PRE == 1) {
        const double *w = wts + p * 2 * W;
#pragma unroll
        for (int a = 0; a < W; ++a) {
            wa[a] = (T)__ldg(w + a);
            wb[a] = (T)__ldg(w + W + a);
        }
    } else if (PRE == 2) {
        const float *w = dd_weights<W>(wts, p);
#pragma unroll
        for (int a = 0; a < W; ++a) {
            wa[a] = (T)df_value(dd_theta<W>(w, a));
            wb[a] = (T)df_value(dd_phi<W>(w, a));
        }
    } else if constexpr (std::is_same<T, float>::value) {
        const float tx = fmaf(2.f, f.x, -(float)(W - 1)), ty = fmaf(2.f, f.y, -(float)(W - 1));
#pragma unroll
        for (int a = 0; a < W; ++a) {
            wa[a] = ker_poly<W>(kp, a, tx);
            wb[a] = ker_poly<W>(kp, a, ty);
        }
    } else {
        const T twoW = T(2) / T(W);
#pragma unroll
        for (int a = 0; a < W; ++a) {
            wa[a] = es_kernel<T>(f.x - T(a), twoW, beta);
            wb[a] = es_kernel<T>(f.y - T(a), twoW, beta);
        }
    }
}

template <typename T, int W, bool SPIN, int PRE>
__global__ void __launch_bounds__(256) k_interp(const void *__restrict__ grid, const uint32_t *__restrict__ cell,
                                                const cplx<T> *__restrict__ frac, const int32_t *__restrict__ perm,
                                                const cplx<T> *__restrict__ phase, const double *__restrict__ wts,
                                                T *__restrict__ map, int64_t n, int pitch, T beta,
                                                const __grid_constant__ KerPoly kp)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t c0 = cell[p];
    T wa[W], wb[W];
    tap_weights<T, W, PRE>(wa, wb, PRE ? cplx<T>{} : frac[p], wts, p, beta, kp);
    const int32_t dst = perm[p];
    if (!SPIN) {
        const T *g = (const T *)grid + c0;
        T acc = T(0);
#pragma unroll
        for (int a = 0; a < W; ++a) {
            T r = T(0);
#pragma unroll
            for (int b = 0; b < W; ++b) r += wb[b] * __ldg(g + (int64_t)a * pitch + b);
            acc += wa[a] * r;
        }
        map[dst] = acc;
    } else {
        const cplx<T> *g = (const cplx<T> *)grid + c0;
        T ax = T(0), ay = T(0);
#pragma unroll
        for (int a = 0; a < W; ++a) {
            T rx = T(0), ry = T(0);
#pragma unroll
            for (int b = 0; b < W; ++b) {
                const cplx<T> v = __ldg(g + (int64_t)a * pitch + b);
                rx += wb[b] * v.x;
                ry += wb[b] * v.y;
            }
            ax += wa[a] * rx;
            ay += wa[a] * ry;
        }
        const cplx<T> ph = phase[p];
        map[dst] = ax * ph.x - ay * ph.y;
        map[n + dst] = ax * ph.y + ay * ph.x;
    }
}

// FP32 plans: the W taps of a row by aligned pairs of cells (spin s 16-byte loads of two complex cells, spin 0 8-byte
// loads of two real ones), the weights shifted by one cell where the first tap lies in the second half of its pair;
// (W + 2) / 2 loads a row instead of W.  The sums were bound by the L1 data stage (92% of its wavefronts: lanes of
// neighbouring points hit the same banks with 4- and 8-byte loads); with the points sorted by row and column the 8 lanes of a
// 16-byte load's quarter lie within ~13 cells.  The extra cell of a pair may be one past the row's wrap columns: k_phi_fwd
// writes zeros there.  Spin s sums in tap order, as before (its bits do not change).
template <int W, bool SPIN>
__global__ void __launch_bounds__(256) k_interp32(const float *__restrict__ grid, const uint32_t *__restrict__ cell,
                                                  const float2 *__restrict__ frac, const int32_t *__restrict__ perm,
                                                  const float2 *__restrict__ phase, float *__restrict__ map, int64_t n,
                                                  int pitch, const __grid_constant__ KerPoly kp)
{
    constexpr int NPR = (W + 2) / 2;  // pairs that cover W cells from either half of a pair
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const uint32_t c0 = cell[p];  // row * pitch + column, pitch even: its parity is the column's
    const bool odd = c0 & 1;
    float wa[W], wb[W];
    tap_weights<float, W, 0>(wa, wb, frac[p], nullptr, p, 0.f, kp);
    float ws[2 * NPR];
#pragma unroll
    for (int k = 0; k < 2 * NPR; ++k) {
        const float e = k < W ? wb[k < W ? k : 0] : 0.f, o = k > 0 && k - 1 < W ? wb[k > 0 && k - 1 < W ? k - 1 : 0] : 0.f;
        ws[k] = odd ? o : e;
    }
    const int32_t dst = perm[p];
    if constexpr (!SPIN) {
        const float *g = grid + (c0 & ~1u);
        pk w2[NPR];
#pragma unroll
        for (int k = 0; k < NPR; ++k) w2[k] = pk_make(ws[2 * k], ws[2 * k + 1]);
        pk acc = 0ull;
#pragma unroll
        for (int a = 0; a < W; ++a) {
            pk r = 0ull;
#pragma unroll
            for (int k = 0; k < NPR; ++k)
                r = pk_fma(w2[k], __ldg(reinterpret_cast<const pk *>(g + (int64_t)a * pitch) + k), r);
            acc = pk_fma(pk_make(wa[a], wa[a]), r, acc);
        }
        const float2 v = pk_get(acc);
        map[dst] = v.x + v.y;
    } else {
        const float *g = grid + 2 * (int64_t)(c0 & ~1u);
        pk acc = 0ull;
#pragma unroll
        for (int a = 0; a < W; ++a) {
            pk r = 0ull;
#pragma unroll
            for (int k = 0; k < NPR; ++k) {
                const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(g + 2 * (int64_t)a * pitch) + k);
                r = pk_fma(pk_make(ws[2 * k], ws[2 * k]), v.x, r);
                r = pk_fma(pk_make(ws[2 * k + 1], ws[2 * k + 1]), v.y, r);
            }
            acc = pk_fma(pk_make(wa[a], wa[a]), r, acc);
        }
        const float2 s = pk_get(acc), ph = phase[p];
        map[dst] = s.x * ph.x - s.y * ph.y;
        map[n + dst] = s.x * ph.y + s.y * ph.x;
    }
}

// FP64 plans with point weights: the same sums in double-float arithmetic on the FP32 pipe.  The grid holds
// double-float pairs (k_phi_fwd writes them for these plans: float2 per real, spin s float4 (re h, im h, re l, im l)); a
// term is one d2_fma (pk.cuh) of both components of a column, or for spin 0 of two rows; row sums are
// normalised before the theta weights; ~2^-46 relative per term.
// A warp brings the weights of its 32 points (contiguous in the table) through shared memory with coalesced 16-byte
// loads, each point's row padded to an odd number of 16-byte words (conflict-free LDS.128).  Bound by the L1
// data stage (92% busy: the grid loads, whose lanes cover about three rows of a tile); FMA pipe 58%.  Spin 2,
// lmax 2048, 12.6M points, W = 13 (FP64 eps 1e-10): 3.09 ms with the weights read by each thread (3W loads of 32 separate
// lines) and scalar sums, 2.87 with the weights staged, 2.05 with packed sums; spin 0: 1.45 staged, 1.38 packed.
// Four CTAs per SM (128 registers): 2.05 ms; three 2.13, five 2.08, six 2.17.
constexpr int kInterpDD = 128;  // threads per CTA
template <int W, bool SPIN>
__global__ void __launch_bounds__(kInterpDD, 4) k_interp_dd(const void *__restrict__ grid, const uint32_t *__restrict__ cell,
                                                            const int32_t *__restrict__ perm,
                                                            const double2 *__restrict__ phase,
                                                            const double *__restrict__ wts, double *__restrict__ map,
                                                            int64_t n, int pitch)
{
    constexpr int NP = dd_pairs(W), Q = dd_words(W) / 4, S = Q | 1;  // 16-byte words per point and per row
    __shared__ float4 sw[kInterpDD * S];
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * kInterpDD + threadIdx.x, p0 = p - lane;
    float4 *wrow = sw + (threadIdx.x - lane) * S;
    const int words = (int)min((int64_t)32, n - p0) * Q;
    const float4 *wg = reinterpret_cast<const float4 *>(wts) + p0 * Q;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const int i = k * 32 + lane;
        if (i < words) wrow[i / Q * S + i % Q] = __ldg(wg + i);
    }
    __syncwarp();
    if (p >= n) return;
    const uint32_t c0 = cell[p];
    const int32_t dst = perm[p];
    const float4 *w = wrow + lane * S;
    // phi weights; an odd W's first one shares its 16 bytes with the last theta weight
    constexpr int O = W & 1;
    df32 wb[W];
    const float4 mid = O ? w[W / 2] : make_float4(0.f, 0.f, 0.f, 0.f);
    if (O) wb[0] = {mid.z, mid.w};
#pragma unroll
    for (int i = 0; i < W / 2; ++i) {
        const float4 v = w[W / 2 + O + i];
        wb[2 * i + O] = {v.x, v.y};
        wb[2 * i + O + 1] = {v.z, v.w};
    }
    if (!SPIN) {
        const float2 *g = reinterpret_cast<const float2 *>(grid) + c0;
        D2 acc = {0ull, 0ull};  // rows in pairs; an odd W's last row twice, the second time with weight zero
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 *ga = g + (int64_t)(2 * i) * pitch, *gb = 2 * i + 1 < W ? ga + pitch : ga;
            D2 r = {0ull, 0ull};
#pragma unroll
            for (int b = 0; b < W; ++b) {
                const float2 x = __ldg(ga + b), y = __ldg(gb + b);
                r = d2_fma(D2{pk_make(x.x, y.x), pk_make(x.y, y.y)}, D2{pk_make(wb[b].h, wb[b].h), pk_make(wb[b].l, wb[b].l)}, r);
            }
            D2 wa;
            if (2 * i + 1 < W) {
                const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(w)[i];
                wa = {v.x, v.y};
            } else {
                wa = {pk_make(mid.x, 0.f), pk_make(mid.y, 0.f)};
            }
            acc = d2_fma(d2_norm(r), wa, acc);
        }
        const float2 sh = pk_get(acc.h), sl = pk_get(acc.l);
        map[dst] = df_value(df32{sh.x, sl.x}) + df_value(df32{sh.y, sl.y});
    } else {
        // both components in one packed instruction (grid: re h, im h, re l, im l)
        const ulonglong2 *g = reinterpret_cast<const ulonglong2 *>(grid) + c0;
        D2 acc = {0ull, 0ull};
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float4 wa = w[i];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int a = 2 * i + k;
                if (a >= W) continue;
                D2 r = {0ull, 0ull};
#pragma unroll
                for (int b = 0; b < W; ++b) {
                    const ulonglong2 v = __ldg(g + (int64_t)a * pitch + b);
                    r = d2_fma(D2{v.x, v.y}, D2{pk_make(wb[b].h, wb[b].h), pk_make(wb[b].l, wb[b].l)}, r);
                }
                const df32 t = 2 * i + 1 == W ? df32{wa.x, wa.y} : k ? df32{wa.y, wa.w} : df32{wa.x, wa.z};
                acc = d2_fma(d2_norm(r), D2{pk_make(t.h, t.h), pk_make(t.l, t.l)}, acc);
            }
        }
        const float2 sh = pk_get(acc.h), sl = pk_get(acc.l);
        const double2 ph = phase[p];
        const double x = df_value(df32{sh.x, sl.x}), y = df_value(df32{sh.y, sl.y});
        map[dst] = x * ph.x - y * ph.y;
        map[n + dst] = x * ph.y + y * ph.x;
    }
}

// one thread per sorted point, one global atomic per tap (deterministic FP64 plans):
// fixed-point integers into the grid memory (scale *fxs)
template <typename T, bool FX> struct Acc {
    using type = T;
};
template <typename T> struct Acc<T, true> {
    using type = unsigned long long;
};
template <typename T, bool FX>
__device__ __forceinline__ void acc_add(typename Acc<T, FX>::type *dst, T v, T sc)
{
    if constexpr (FX) atomicAdd(dst, to_fx(v, sc));
    else atomicAdd(dst, v);
}

template <typename T, int W, bool SPIN, int PRE>
__global__ void __launch_bounds__(256) k_spread_direct(void *__restrict__ grid, const uint32_t *__restrict__ cell,
                                                       const cplx<T> *__restrict__ frac,
                                                       const int32_t *__restrict__ perm,
                                                       const cplx<T> *__restrict__ phase,
                                                       const double *__restrict__ wts, const T *__restrict__ map,
                                                       int64_t n, int pitch, T beta, const double *__restrict__ fxs,
                                                       const __grid_constant__ KerPoly kp)
{
    using G = typename Acc<T, true>::type;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const T sc = (T)fxs[0];
    const uint32_t c0 = cell[p];
    T wa[W], wb[W];
    tap_weights<T, W, PRE>(wa, wb, PRE ? cplx<T>{} : frac[p], wts, p, beta, kp);
    const int32_t src = perm[p];
    if (!SPIN) {
        const T x = map[src];
        G *g = (G *)grid + c0;
#pragma unroll
        for (int a = 0; a < W; ++a) {
            const T xa = wa[a] * x;
#pragma unroll
            for (int b = 0; b < W; ++b) acc_add<T, true>(g + (int64_t)a * pitch + b, xa * wb[b], sc);
        }
    } else {
        // e^{-i s chi} (Q + i U)
        const cplx<T> ph = phase[p];
        const T q = map[src], u = map[n + src];
        const T zx = ph.x * q + ph.y * u, zy = ph.x * u - ph.y * q;
        G *g = (G *)grid + 2 * (int64_t)c0;
#pragma unroll
        for (int a = 0; a < W; ++a) {
            const T xa = wa[a] * zx, ya = wa[a] * zy;
#pragma unroll
            for (int b = 0; b < W; ++b) {
                G *q2 = g + 2 * ((int64_t)a * pitch + b);
                acc_add<T, true>(q2, xa * wb[b], sc);
                acc_add<T, true>(q2 + 1, ya * wb[b], sc);
            }
        }
    }
}

// FX: fixed-point integers in shared memory and in the grid (scale *fxs).
// IT (integer tiles; FP32 plans at epsilon >= 1e-5 and FP64 plans, not FX):
// the tile accumulates in fixed point in shared memory, 32-bit integers for
// FP32 plans (integer atomics there run ~3x the rate of float atomics) and
// 64-bit for FP64 plans (no FP64 atomics in the inner loop), in units of 1/u
// with u = 2^k per tile, k the largest integer with kmax_t max|x| u <= 2^30
// (FP64: 2^62): kmax_t (plan time) is the most of the tile's points whose
// W x W windows cover one cell and max|x| (per call) the map's largest |value|
// (|Q| + |U| for spin s), taps |psi| <= 1, so no cell sum can overflow.  Every
// term is rounded once (to 2^-k; FP64: relative 2^-62 of the tile's bound);
// the flush converts back for one global atomic per non-zero cell.  A map
// with a non-finite value makes the whole tile NaN.
// Where kPassFrom or more points reach one cell, the tile is spread and flushed kPassPoints points at a time, by
// gridDim.y CTAs in turn: tile_kmax holds at most 65535, and the unit would grow with the pile (FP32, a map of one sign, 300,000 points in one cell: 7e-5 of the
// a_lm; with the passes 6e-7 at 150,000).  FP32: even skies reach 1024 points only above 20 per cell, where the flush of a
// pass starts to cost.
template <typename T> constexpr uint32_t kPassFrom = sizeof(T) == 4 ? 1024 : 65535;
template <typename T> constexpr uint32_t kPassPoints = sizeof(T) == 4 ? 512 : 65535;
template <typename T, bool FX, bool IT> struct SAcc { using type = typename Acc<T, FX>::type; };
template <> struct SAcc<float, false, true> { using type = int; };
template <> struct SAcc<double, false, true> { using type = long long; };
__device__ __forceinline__ int tile_int(float v) { return __float2int_rn(v); }
__device__ __forceinline__ long long tile_int(double v) { return __double2ll_rn(v); }
__device__ __forceinline__ void tile_add(int *dst, int v) { atomicAdd(dst, v); }
__device__ __forceinline__ void tile_add(long long *dst, long long v)
{
    atomicAdd(reinterpret_cast<unsigned long long *>(dst), (unsigned long long)v);  // two's complement sum
}

// PILE: some tile has kPassFrom or more points in a cell (FP32 plans run the variant without passes otherwise: with a loop of
// passes around the body spin 0, lmax 512, W = 9 took 56.5 us for 53.4).
template <typename T, int W, bool SPIN, int PRE, bool FX, bool IT = false, bool PILE = sizeof(T) == 8>
__global__ void __launch_bounds__(sizeof(T) == 8 ? kSpreadThreads64 : kSpreadThreads) k_spread(void *__restrict__ grid, const uint32_t *__restrict__ cell,
                                                           const cplx<T> *__restrict__ frac,
                                                           const int32_t *__restrict__ perm,
                                                           const cplx<T> *__restrict__ phase,
                                                           const double *__restrict__ wts, const T *__restrict__ map,
                                                           int64_t n, int pitch, int R, int ntc,
                                                           const uint32_t *__restrict__ tile_start, T beta,
                                                           const double *__restrict__ fxs,
                                                           int tile_r, int sorted, const unsigned short *__restrict__ tile_kmax,
                                                           const unsigned long long *__restrict__ maxbits,
                                                           const __grid_constant__ KerPoly kp)
{
    static_assert(!(IT && FX), "fixed-point tiles or fixed-point grid");
    using G = typename SAcc<T, FX, IT>::type;
    constexpr int TC = kTileC + W - 1, NC = SPIN ? 2 : 1;
    const int TR = tile_r + W - 1;  // tile rows (16, 32 or 64) plus the kernel halo
    extern __shared__ __align__(16) unsigned char spread_smem[];
    G *buf = reinterpret_cast<G *>(spread_smem);  // TR x TC cells x NC planes
    const int t = blockIdx.x;
    const uint32_t p0 = tile_start[t], p1 = tile_start[t + 1];
    if (p0 == p1) return;
    T sc = FX ? (T)fxs[0] : T(1);
    bool bad = false;  // IT: non-finite map value
    bool pile = false;
    if constexpr (IT) {
        constexpr int kBits = sizeof(T) == 4 ? 30 : 62;  // tile sums of |terms| below 2^kBits
        pile = PILE && tile_kmax[t] >= kPassFrom<T>;
        const double bound =
            (double)(pile ? kPassPoints<T> : tile_kmax[t]) * __longlong_as_double((long long)*maxbits);
        if (!(bound < 1e300)) bad = true;  // infinity or NaN in the map
        else if (bound > 0.0) sc = (T)ldexp(1.0, kBits - (ilogb(bound) + 1));  // bound < 2^(ilogb+1)
        pile = pile && !bad;
    }
    if (PILE && blockIdx.y > 0 && !pile) return;
    const int r0 = (t / ntc) * tile_r, c0 = (t % ntc) * kTileC;
    // points pb .. pe - 1, which reach the tile rows lo .. hi - 1
    const auto pass = [&](uint32_t pb, uint32_t pe, int lo, int hi) {
        for (int i = lo * TC + threadIdx.x; i < hi * TC; i += blockDim.x) {
            buf[i] = G(0);
            if (SPIN) buf[TR * TC + i] = G(0);
        }
        __syncthreads();
        // (points in sorted order: spin 2, lmax 2048, W = 7: 0.69 ms; a run of points per thread, for fewer of a warp's taps in
        // one bank, 0.77, runs per group of four threads 0.78: the loads then no longer coalesce)
        for (uint32_t p = pb + threadIdx.x; p < (bad ? pb : pe); p += blockDim.x) {
            const uint32_t c = cell[p];
            const int lr = (int)(c / (uint32_t)pitch) - r0, lc = (int)(c % (uint32_t)pitch) - c0;
            if ((unsigned)lr >= (unsigned)tile_r || (unsigned)lc >= (unsigned)kTileC) continue;  // not this tile's
            const int32_t src = perm[p];
            // spin s: two planes (real parts, then imaginary parts), so that the lanes'
            // atomics of one plane spread over all 32 banks
            G *b0 = buf + (lr * TC + lc);
            T wa[W], wb[W];
            tap_weights<T, W, PRE>(wa, wb, PRE ? cplx<T>{} : frac[p], wts, p, beta, kp);
            // IT: the power-of-two unit sc is applied to the point's value first (exact)
            if (!SPIN) {
                const T x = IT ? map[src] * sc : map[src];
#pragma unroll
                for (int a = 0; a < W; ++a) {
                    const T xa = wa[a] * x;
#pragma unroll
                    for (int b = 0; b < W; ++b) {
                        if constexpr (IT) tile_add(b0 + a * TC + b, tile_int(xa * wb[b]));
                        else acc_add<T, FX>(b0 + a * TC + b, xa * wb[b], sc);
                    }
                }
            } else {
                // e^{-i s chi} (Q + i U)
                const cplx<T> ph = phase[p];
                const T q = map[src], u = map[n + src];
                T zx = ph.x * q + ph.y * u, zy = ph.x * u - ph.y * q;
                if constexpr (IT) { zx *= sc; zy *= sc; }
#pragma unroll
                for (int a = 0; a < W; ++a) {
                    const T xa = wa[a] * zx, ya = wa[a] * zy;
#pragma unroll
                    for (int b = 0; b < W; ++b) {
                        G *q2 = b0 + (a * TC + b);
                        if constexpr (IT) {
                            tile_add(q2, tile_int(xa * wb[b]));
                            tile_add(q2 + TR * TC, tile_int(ya * wb[b]));
                        } else {
                            acc_add<T, FX>(q2, xa * wb[b], sc);
                            acc_add<T, FX>(q2 + TR * TC, ya * wb[b], sc);
                        }
                    }
                }
            }
        }
        __syncthreads();
        if constexpr (IT) {
            T *g = (T *)grid;
            const T inv = bad ? T(NAN) : T(1) / sc;
            for (int i = lo * TC + threadIdx.x; i < hi * TC; i += blockDim.x) {
                const int gr = r0 + i / TC, gc = c0 + i % TC;
                if (gr >= R || gc >= pitch) continue;
                const int64_t o = (int64_t)gr * pitch + gc;
                if (!SPIN) {
                    const G v = buf[i];
                    if (v != 0 || bad) atomicAdd(g + o, (T)v * inv);
                } else {
                    const G vx = buf[i], vy = buf[TR * TC + i];
                    if (vx != 0 || bad) atomicAdd(g + 2 * o, (T)vx * inv);
                    if (vy != 0 || bad) atomicAdd(g + 2 * o + 1, (T)vy * inv);
                }
            }
        } else {
            G *g = (G *)grid;
            for (int i = lo * TC + threadIdx.x; i < hi * TC; i += blockDim.x) {
                const int gr = r0 + i / TC, gc = c0 + i % TC;
                if (gr >= R || gc >= pitch) continue;
                const int64_t o = (int64_t)gr * pitch + gc;
                if (!SPIN) {
                    const G v = buf[i];
                    if (v != G(0)) atomicAdd(g + o, v);
                } else {
                    const G vx = buf[i], vy = buf[TR * TC + i];
                    if (vx != G(0)) atomicAdd(g + 2 * o, vx);
                    if (vy != G(0)) atomicAdd(g + 2 * o + 1, vy);
                }
            }
        }
    };
    if (!PILE || !pile) {
        pass(p0, p1, 0, TR);
        return;
    }
    constexpr uint32_t step = kPassPoints<T>;
    for (uint32_t pb = p0 + blockIdx.y * step; pb < p1; pb += gridDim.y * step) {
        const uint32_t pe = min(p1, pb + step);
        int lo = 0, hi = TR;
        if (sorted) {
            lo = max((int)(cell[pb] / (uint32_t)pitch) - r0, 0);
            hi = min((int)(cell[pe - 1] / (uint32_t)pitch) - r0 + W, TR);
        }
        pass(pb, pe, lo, hi);
        __syncthreads();  // the next pass clears the tile
    }
}

template <int W, bool SPIN> cudaError_t spread_strip(const Plan &p, const void *map, void *grid, cudaStream_t st);
template <int W, bool SPIN> cudaError_t spread_strip32(const Plan &p, const void *map, void *grid, cudaStream_t st);

template <typename T, bool SPIN, int W>
cudaError_t interp_w(const Plan &p, const void *grid, void *map, cudaStream_t st)
{
    const int thr = 256;
    const int64_t blocks = (p.npts + thr - 1) / thr;
    if (blocks == 0) return cudaSuccess;
    const auto run = [&](auto kern) {
        kern<<<(unsigned)blocks, thr, 0, st>>>(grid, p.cell, (const cplx<T> *)p.frac, p.perm, (const cplx<T> *)p.phase,
                                               p.wts, (T *)map, p.npts, p.pitch, (T)p.beta, p.kpoly);
        return cudaGetLastError();
    };
    if constexpr (std::is_same<T, double>::value) {
        if (p.wts && p.wts_dd) {  // double-float taps on the double-float grid k_phi_fwd wrote
            k_interp_dd<W, SPIN><<<(unsigned)((p.npts + kInterpDD - 1) / kInterpDD), kInterpDD, 0, st>>>(
                grid, p.cell, p.perm, (const double2 *)p.phase, p.wts, (double *)map, p.npts, p.pitch);
            return cudaGetLastError();
        }
        if (p.wts) return run(k_interp<T, W, SPIN, 1>);
        return run(k_interp<T, W, SPIN, 0>);
    } else {
        k_interp32<W, SPIN><<<(unsigned)blocks, thr, 0, st>>>((const float *)grid, p.cell, (const float2 *)p.frac, p.perm,
                                                              (const float2 *)p.phase, (float *)map, p.npts, p.pitch, p.kpoly);
        return cudaGetLastError();
    }
}

template <bool SPIN> constexpr int kStripW = strip_support(SPIN);

template <typename T, bool SPIN, int W>
cudaError_t spread_w(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    if (p.npts == 0) return cudaSuccess;
    const double *fxs = p.fx_scale;
    const size_t cells = (size_t)(p.tile_r + W - 1) * (kTileC + W - 1) * (SPIN ? 2 : 1);
    const auto run = [&](auto kern, size_t esz) {
        const size_t sm = cells * esz;
        cudaError_t e2 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e2 != cudaSuccess) return e2;
        kern<<<dim3((unsigned)p.ntiles, (unsigned)p.parts), sizeof(T) == 8 ? kSpreadThreads64 : kSpreadThreads, sm, st>>>(
            grid, p.cell, (const cplx<T> *)p.frac, p.perm, (const cplx<T> *)p.phase, p.wts, (const T *)map, p.npts,
            p.pitch, p.R, p.ntile_c, p.tile_start, (T)p.beta, fxs, p.tile_r, p.sorted ? 1 : 0, p.tile_kmax, p.maxbits, p.kpoly);
        return cudaGetLastError();
    };
    if constexpr (std::is_same<T, double>::value) {
        if (!p.det) {
            if (p.strip) return spread_strip<W, SPIN>(p, map, grid, st);
            // 64-bit integer tiles
            if (p.wts) return run(k_spread<T, W, SPIN, 1, false, true>, 8);
            return run(k_spread<T, W, SPIN, 0, false, true>, 8);
        }
        const unsigned blocks = (unsigned)((p.npts + 255) / 256);
        const cplx<T> *fr = (const cplx<T> *)p.frac, *ph = (const cplx<T> *)p.phase;
        const auto direct = [&](auto kern) {
            kern<<<blocks, 256, 0, st>>>(grid, p.cell, fr, p.perm, ph, p.wts, (const T *)map, p.npts, p.pitch,
                                         (T)p.beta, fxs, p.kpoly);
            return cudaGetLastError();
        };
        if (p.wts) return p.wts_dd ? direct(k_spread_direct<T, W, SPIN, 2>) : direct(k_spread_direct<T, W, SPIN, 1>);
        return direct(k_spread_direct<T, W, SPIN, 0>);
    } else {
        if (p.det) return run(k_spread<T, W, SPIN, 0, true>, 8);
        if (p.strip) return spread_strip32<W, SPIN>(p, map, grid, st);
        if constexpr (W < kStripW<SPIN>)
            return p.piles ? run(k_spread<T, W, SPIN, 0, false, true, true>, 4) : run(k_spread<T, W, SPIN, 0, false, true, false>, 4);
        else return cudaErrorInvalidValue;  // such plans spread by strips
    }
}

template <typename T, bool SPIN>
cudaError_t interp_dispatch(const Plan &p, const void *grid, void *map, cudaStream_t st)
{
    switch (p.W) {
    case 4: return interp_w<T, SPIN, 4>(p, grid, map, st);
    case 5: return interp_w<T, SPIN, 5>(p, grid, map, st);
    case 6: return interp_w<T, SPIN, 6>(p, grid, map, st);
    case 7: return interp_w<T, SPIN, 7>(p, grid, map, st);
    case 8: return interp_w<T, SPIN, 8>(p, grid, map, st);
    case 9: return interp_w<T, SPIN, 9>(p, grid, map, st);
    case 10: return interp_w<T, SPIN, 10>(p, grid, map, st);
    case 11: return interp_w<T, SPIN, 11>(p, grid, map, st);
    case 12: return interp_w<T, SPIN, 12>(p, grid, map, st);
    case 13: return interp_w<T, SPIN, 13>(p, grid, map, st);
    case 14: return interp_w<T, SPIN, 14>(p, grid, map, st);
    case 15: return interp_w<T, SPIN, 15>(p, grid, map, st);
    case 16: return interp_w<T, SPIN, 16>(p, grid, map, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T, bool SPIN>
cudaError_t spread_dispatch(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    switch (p.W) {
    case 4: return spread_w<T, SPIN, 4>(p, map, grid, st);
    case 5: return spread_w<T, SPIN, 5>(p, map, grid, st);
    case 6: return spread_w<T, SPIN, 6>(p, map, grid, st);
    case 7: return spread_w<T, SPIN, 7>(p, map, grid, st);
    case 8: return spread_w<T, SPIN, 8>(p, map, grid, st);
    case 9: return spread_w<T, SPIN, 9>(p, map, grid, st);
    case 10: return spread_w<T, SPIN, 10>(p, map, grid, st);
    case 11: return spread_w<T, SPIN, 11>(p, map, grid, st);
    case 12: return spread_w<T, SPIN, 12>(p, map, grid, st);
    case 13: return spread_w<T, SPIN, 13>(p, map, grid, st);
    case 14: return spread_w<T, SPIN, 14>(p, map, grid, st);
    case 15: return spread_w<T, SPIN, 15>(p, map, grid, st);
    case 16: return spread_w<T, SPIN, 16>(p, map, grid, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace gsl
