// Spreading of FP64 plans with double-float weights (epsilon >= 5e-11) and of FP32 plans with W >= 8 (spin 0: W >= 10; or epsilon < 1e-5),
// not deterministic: tiles swept row by row in registers.
//
// One warp owns a tile of tile_r rows x (33 - W) columns, so the W-wide windows of its points cover 32
// columns: lane c holds column c of the W rows that the points of one cell row touch, as sums of row pairs
// (f32x2 instructions).  The points are sorted by cell row (plan creation); after the points of a
// row, its grid row receives nothing more from this tile: the lane adds it into the grid with one atomic and
// the window moves down a row.  No shared-memory accumulation: the tiles of 64-bit integers that this replaces
// were bound by shared-memory atomics (1.1 taps per clock and SM; lmax 4096, 50M points, W = 13: spin 0 24.2 ms, spin 2
// 45.7, now 9.6 and 17.0).  A point costs the whole warp W/2 multiply-adds of a pair (an odd W's last row is scalar: half
// of one), whatever part of the 32 columns it covers (W = 13: 41%).
//
// Sums are double-float (d2_fma, ~2^-47 of the partial sums), of values scaled by the power of two that brings the
// tile's largest one near 1.  Tried and not kept: high words offset by a bound of the cell's sum, where a term takes 6
// instructions instead of 10; their rounding errors are relative to that bound (4e-12 of the a_lm at 1.2
// points per cell, against 5e-13 for the integer tiles).
//
// Weights arrive by bulk copies of 16 points (contiguous in the table) into shared memory, double-buffered on
// mbarriers; a wait that gives up sets FLAG_TIMEOUT, the warp waits for its other copy in flight and returns.
#pragma once

#include "nufft.cuh"
#include "pk.cuh"

namespace gsl {
namespace {

constexpr int kStripWarps = 4;   // warps (tiles) per CTA
constexpr int kStripBatch = 16;  // points per weight copy (FP64)

template <int W> __host__ __device__ constexpr size_t strip_warp_smem()
{
    // two weight buffers, values (float4), offsets (int), two mbarriers
    return 2 * kStripBatch * dd_words(W) * sizeof(float) + kStripBatch * (sizeof(float4) + sizeof(int)) + 16;
}

// Points of tile t for this CTA row: blockIdx.y-th part of `part` points (a tile with more points than that is shared
// by several warps, each sweeping the rows of its part); false if there are none.
__device__ __forceinline__ bool strip_points(const uint32_t *__restrict__ tile_start, int t, uint32_t part, uint32_t &p0,
                                             uint32_t &p1)
{
    const uint32_t a = tile_start[t], b = tile_start[t + 1], off = blockIdx.y * part;
    if (b - a <= off) return false;
    p0 = a + off;
    p1 = min(b, p0 + part);
    return true;
}

template <int W, bool SPIN>
__global__ void __launch_bounds__(32 * kStripWarps)
k_spread_strip(double *__restrict__ grid, const uint32_t *__restrict__ cell, const int32_t *__restrict__ perm,
               const double2 *__restrict__ phase, const double *__restrict__ wts, const double *__restrict__ map,
               int64_t n, int pitch, int R, int ntc, int ntiles, const uint32_t *__restrict__ tile_start, int tile_r,
               uint32_t part, unsigned *__restrict__ status)
{
    constexpr int NP = W / 2, NC = SPIN ? 2 : 1, TC = 33 - W;  // row pairs; an odd W's last row by itself
    constexpr bool ODD = W & 1;
    constexpr uint32_t WBYTES = dd_words(W) * sizeof(float);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int t = blockIdx.x * kStripWarps + wid;
    if (t >= ntiles) return;
    uint32_t p0, p1;
    if (!strip_points(tile_start, t, part, p0, p1)) return;
    extern __shared__ __align__(16) unsigned char strip_smem[];
    unsigned char *mem = strip_smem + wid * strip_warp_smem<W>();
    float4 *sval = reinterpret_cast<float4 *>(mem + 2 * kStripBatch * WBYTES);
    int *soff = reinterpret_cast<int *>(sval + kStripBatch);
    uint64_t *bar = reinterpret_cast<uint64_t *>(soff + kStripBatch);
    if (lane == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        fence_async_shared();
    }
    __syncwarp();
    const int nb = (int)((p1 - p0 + kStripBatch - 1) / kStripBatch);
    auto fetch = [&](int k) {  // weights of batch k into buffer k & 1
        if (lane == 0) {
            const uint32_t q = p0 + k * kStripBatch, cnt = min((uint32_t)kStripBatch, p1 - q);
            mbar_expect_tx(bar + (k & 1), cnt * WBYTES);
            bulk_copy_g2s(mem + (k & 1) * kStripBatch * WBYTES, reinterpret_cast<const char *>(wts) + (size_t)q * WBYTES,
                          cnt * WBYTES, bar + (k & 1));
        }
    };
    fetch(0);

    // the tile's largest |value| (spin s: |Q| + |U|, whose exponent range is the values' own; squares would lose
    // maps above 1e154 and below 1e-162) as the bits of a non-negative double
    unsigned long long mx = 0;
    for (uint32_t p = p0 + lane; p < p1; p += 32) {
        const int32_t src = perm[p];
        const double q = fabs(map[src]), v = SPIN ? q + fabs(map[n + src]) : q;
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        mx = b > mx ? b : mx;  // infinities and NaNs order above the finite values
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        mx = o > mx ? o : mx;
    }
    const double top = __longlong_as_double((long long)mx);
    const bool bad = !(top < 1e300);  // infinity or NaN: the tile becomes NaN
    int ex = bad || top == 0.0 ? 0 : -ilogb(top);
    ex = min(max(ex, -1000), 1000);
    const double sc = ldexp(1.0, ex), inv = bad ? NAN : ldexp(1.0, -ex);

    const int r0 = (t / ntc) * tile_r, c0 = (t % ntc) * TC;
    D2 S[NC][NP];
    df32 last[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        last[c] = {0.f, 0.f};
#pragma unroll
        for (int i = 0; i < NP; ++i) S[c][i] = {0ull, 0ull};
    }
    int cur = 0;  // tile row of the window's first row
    const int gc = c0 + lane;
    auto next_row = [&]() {  // add the window's first row into the grid, move down
        const int gr = r0 + cur;
        bool any = bad;
        df32 v[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            v[c] = {pk_get(S[c][0].h).x, pk_get(S[c][0].l).x};
            any = any || v[c].h != 0.f || v[c].l != 0.f;
        }
        if (any && gr < R && gc < pitch) {
            double *g = grid + ((int64_t)gr * pitch + gc) * NC;
#pragma unroll
            for (int c = 0; c < NC; ++c) atomicAdd(g + c, df_value(v[c]) * inv);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                S[c][i].h = pk_make(pk_get(S[c][i].h).y, i + 1 < NP ? pk_get(S[c][i + 1 < NP ? i + 1 : i].h).x : last[c].h);
                S[c][i].l = pk_make(pk_get(S[c][i].l).y, i + 1 < NP ? pk_get(S[c][i + 1 < NP ? i + 1 : i].l).x : last[c].l);
            }
            last[c] = {0.f, 0.f};
        }
        ++cur;
    };

    bool ok = true;
    for (int k = 0; k < nb; ++k) {
        if (k + 1 < nb) fetch(k + 1);  // its buffer was last read in batch k - 1 (all lanes past the barrier below)
        const uint32_t q0 = p0 + k * kStripBatch;
        const int cnt = (int)min((uint32_t)kStripBatch, p1 - q0);
        if (lane < cnt) {
            const uint32_t p = q0 + lane, c = cell[p];
            const int lr = (int)(c / (uint32_t)pitch) - r0, lc = (int)(c % (uint32_t)pitch) - c0;
            const bool mine = (unsigned)lr < (unsigned)tile_r && (unsigned)lc < (unsigned)TC;
            const int32_t src = perm[p];
            df32 x, y = {0.f, 0.f};
            if constexpr (!SPIN) {
                x = df_split(map[src] * sc);
            } else {
                const double2 ph = phase[p];
                const double qv = map[src], u = map[n + src];
                x = df_split((ph.x * qv + ph.y * u) * sc);
                y = df_split((ph.x * u - ph.y * qv) * sc);
            }
            soff[lane] = mine && !bad ? lr << 8 | lc : -1;
            sval[lane] = make_float4(x.h, x.l, y.h, y.l);
        }
        if (!mbar_wait_warp(bar + (k & 1), (k >> 1) & 1)) {
            if (k + 1 < nb) mbar_wait_warp(bar + ((k + 1) & 1), ((k + 1) >> 1) & 1);
            ok = false;
            break;
        }
        __syncwarp();
        const float *wbuf = reinterpret_cast<const float *>(mem + (k & 1) * kStripBatch * WBYTES);
        // the next point's offset, value and column weight are loaded while a point is summed
        int so = soff[0];
        float4 xv = sval[0];
        auto column = [&](int q, int o) {
            const int b = lane - (o & 255);
            return o >= 0 && (unsigned)b < (unsigned)W
                       ? *reinterpret_cast<const float2 *>(wbuf + q * dd_words(W) + 2 * W + 2 * b)
                       : make_float2(0.f, 0.f);
        };
        float2 wb = column(0, so);
#pragma unroll 1
        for (int q = 0; q < cnt; ++q) {
            const float *w = wbuf + q * dd_words(W);
            const int row = so >> 8;  // (-1 for a point of no tile: no row to move to, weights zero)
            D2 v[NC];
            df32 t[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                t[c] = df_mul(df32{wb.x, wb.y}, c == 0 ? df32{xv.x, xv.y} : df32{xv.z, xv.w});
                v[c] = {pk_make(t[c].h, t[c].h), pk_make(t[c].l, t[c].l)};
            }
            const int qn = min(q + 1, cnt - 1);
            so = soff[qn];
            xv = sval[qn];
            wb = column(qn, so);
            while (cur < row) next_row();
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const ulonglong2 wa = *reinterpret_cast<const ulonglong2 *>(w + 4 * i);
#pragma unroll
                for (int c = 0; c < NC; ++c) S[c][i] = d2_fma(D2{wa.x, wa.y}, v[c], S[c][i]);
            }
            if constexpr (ODD) {
                const float2 wa = *reinterpret_cast<const float2 *>(w + 4 * NP);
#pragma unroll
                for (int c = 0; c < NC; ++c) last[c] = df_fma(df32{wa.x, wa.y}, t[c], last[c]);
            }
        }
        // keep the low words below an ulp of the sums (2,000 points in one cell, unnormalised: 2e-12 of the a_lm)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
#pragma unroll
            for (int i = 0; i < NP; ++i) S[c][i] = d2_norm(S[c][i]);
            if constexpr (ODD) last[c] = df_renorm(last[c]);
        }
        __syncwarp();  // the buffers are rewritten by the next batch
    }
    if (!ok && lane == 0) atomicOr(status, FLAG_TIMEOUT);
    const int end = min(tile_r + W - 1, bad ? 1 << 20 : cur + W);  // rows the last points reach
    while (cur < end) next_row();
}

// FP32 plans with W >= 8 (spin 0: W >= 10; or epsilon < 1e-5): the same sweep with FP32 sums.  Each lane evaluates the 2W polynomial weights
// of one point of a batch of 32 into shared memory (the coefficients come from the constant bank); then the warp
// takes the points in turn.  Bound by issue: for both components of spin s about 50 instructions a point at W = 8 and 60 at
// W = 10, where the tiles of 32-bit integers in shared memory (nufft.cuh) cost 2 W^2 atomics.  The rule stands in plan.cu
// with both sides measured (spin 2, lmax 4096, 50M points, W = 8: tiles 3.34 ms, strips 2.66).  Sums of up to 4096 points of a
// warp (more in piles above 262,144 points) are plain FP32: 1e-6 of the a_lm for 300,000 points in one cell (integer tiles
// in one pass: 5e-5 to 4e-4).  Two tiles of 17 - W columns per warp, one per half,
// were tried for the lanes a point leaves idle: 2.83 ms, and the narrow tiles cost the interpolation 0.2-0.4 ms.
template <int W> __host__ __device__ constexpr size_t strip32_warp_smem()
{
    // per point: value twice (float4), theta weights (padded to 16 bytes), tile row and column (int2), phi weights; one
    // slot more than the 32 points, which the loop's look-ahead reads
    return (33 * (4 + 4 * ((W + 3) / 4) + 2 + W) * sizeof(float) + 15) / 16 * 16;
}

template <int W, bool SPIN>
__global__ void __launch_bounds__(32 * kStripWarps)
k_spread_strip32(float *__restrict__ grid, const uint32_t *__restrict__ cell, const float2 *__restrict__ frac,
                 const int32_t *__restrict__ perm, const float2 *__restrict__ phase, const float *__restrict__ map,
                 int64_t n, int pitch, int R, int ntc, int ntiles, const uint32_t *__restrict__ tile_start, int tile_r,
                 uint32_t part, const __grid_constant__ KerPoly kp)
{
    constexpr int NP = (W + 1) / 2, NC = SPIN ? 2 : 1, TC = 33 - W, WA = 4 * ((W + 3) / 4);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int t = blockIdx.x * kStripWarps + wid;
    if (t >= ntiles) return;
    uint32_t p0, p1;
    if (!strip_points(tile_start, t, part, p0, p1)) return;
    extern __shared__ __align__(16) unsigned char strip_smem[];
    float4 *sval = reinterpret_cast<float4 *>(strip_smem + wid * strip32_warp_smem<W>());  // (x, x, y, y)
    float *swa = reinterpret_cast<float *>(sval + 33);                                     // [33][WA]
    int2 *soff = reinterpret_cast<int2 *>(swa + 33 * WA);                                  // (row, column)
    float *swb = reinterpret_cast<float *>(soff + 33);                                     // [33][W]

    const int r0 = (t / ntc) * tile_r, c0 = (t % ntc) * TC, gc = c0 + lane;
    pk S[NC][NP];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < NP; ++i) S[c][i] = 0ull;
    int cur = 0;
    auto next_row = [&]() {
        const int gr = r0 + cur;
        float v[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) v[c] = pk_get(S[c][0]).x;
        bool any = v[0] != 0.f;
        if (SPIN) any = any || v[NC - 1] != 0.f;
        if (any && gr < R && gc < pitch) {
            const int64_t o = (int64_t)gr * pitch + gc;
            if constexpr (SPIN) atomicAdd(reinterpret_cast<float2 *>(grid) + o, make_float2(v[0], v[NC - 1]));
            else atomicAdd(grid + o, v[0]);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int i = 0; i < NP; ++i)
                S[c][i] = pk_make(pk_get(S[c][i]).y, i + 1 < NP ? pk_get(S[c][i + 1 < NP ? i + 1 : i]).x : 0.f);
        ++cur;
    };
    if (lane == 0) {  // the look-ahead slot: no column
        sval[32] = make_float4(0.f, 0.f, 0.f, 0.f);
        soff[32] = make_int2(0, 64);
    }

    for (uint32_t pb = p0; pb < p1; pb += 32) {
        const int cnt = (int)min(32u, p1 - pb);
        if (lane < cnt) {
            const uint32_t p = pb + lane, c = cell[p];
            const float2 f = frac[p];
            const int lr = (int)(c / (uint32_t)pitch) - r0, lc = (int)(c % (uint32_t)pitch) - c0;
            const bool mine = (unsigned)lr < (unsigned)tile_r && (unsigned)lc < (unsigned)TC;
            const int32_t src = perm[p];
            float2 z = make_float2(map[src], 0.f);
            if constexpr (SPIN) {  // e^{-i s chi} (Q + i U)
                const float2 ph = phase[p];
                const float u = map[n + src];
                z = make_float2(ph.x * z.x + ph.y * u, ph.x * u - ph.y * z.x);
            }
            soff[lane] = mine ? make_int2(lr, lc) : make_int2(0, 64);  // column 64: no lane's
            const float tx = fmaf(2.f, f.x, -(float)(W - 1)), ty = fmaf(2.f, f.y, -(float)(W - 1));
            float wa[WA];
#pragma unroll
            for (int a = 0; a < WA; ++a) wa[a] = a < W ? ker_poly<W>(kp, a < W ? a : 0, tx) : 0.f;
#pragma unroll
            for (int a = 0; a < WA; a += 4)
                *reinterpret_cast<float4 *>(swa + lane * WA + a) = make_float4(wa[a], wa[a + 1], wa[a + 2], wa[a + 3]);
            sval[lane] = make_float4(z.x, z.x, z.y, z.y);
#pragma unroll
            for (int b = 0; b < W; ++b) swb[lane * W + b] = ker_poly<W>(kp, b, ty) * (SPIN ? 1.f : z.x);
        }
        __syncwarp();
        // each point's row and column are loaded two points ahead, its column weight and value one ahead
        int2 so = soff[0], sn = soff[1];
        float wb = (unsigned)(lane - so.y) < (unsigned)W ? swb[lane - so.y] : 0.f;
        ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(sval);
        const float *wap = swa, *wbp = swb + lane;
#pragma unroll 1
        for (int q = 0; q < cnt; ++q) {
            const pk w2 = pk_make(wb, wb);
            pk v[NC];
            if constexpr (SPIN) {
                v[0] = pk_mul(w2, z.x);
                v[NC - 1] = pk_mul(w2, z.y);
                z = *reinterpret_cast<const ulonglong2 *>(sval + q + 1);
            } else {
                v[0] = w2;
            }
            pk wa[2 * ((NP + 1) / 2)];
#pragma unroll
            for (int i = 0; i < NP; i += 2) {
                const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(wap + 2 * i);
                wa[i] = w.x;
                wa[i + 1] = w.y;
            }
            wap += WA;
            wbp += W;
            wb = (unsigned)(lane - sn.y) < (unsigned)W ? wbp[-sn.y] : 0.f;
            while (cur < so.x) next_row();
            so = sn;
            sn = soff[min(q + 2, 32)];
#pragma unroll
            for (int i = 0; i < NP; ++i)
#pragma unroll
                for (int c = 0; c < NC; ++c) S[c][i] = pk_fma(wa[i], v[c], S[c][i]);
        }
        __syncwarp();  // the staged points are rewritten by the next batch
    }
    const int last = min(tile_r + W - 1, cur + W);
    while (cur < last) next_row();
}

inline dim3 strip_grid(const Plan &p)
{
    return dim3((unsigned)((p.ntiles + kStripWarps - 1) / kStripWarps), (unsigned)p.parts);
}

template <int W, bool SPIN> cudaError_t spread_strip(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    const auto kern = k_spread_strip<W, SPIN>;
    const size_t sm = kStripWarps * strip_warp_smem<W>();
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<strip_grid(p), 32 * kStripWarps, sm, st>>>(
        (double *)grid, p.cell, p.perm, (const double2 *)p.phase, p.wts, (const double *)map, p.npts, p.pitch, p.R,
        p.ntile_c, p.ntiles, p.tile_start, p.tile_r, p.strip_part, p.flags + 1);
    return cudaGetLastError();
}

template <int W, bool SPIN> cudaError_t spread_strip32(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    const size_t sm = kStripWarps * strip32_warp_smem<W>();
    const cudaError_t e =
        cudaFuncSetAttribute(k_spread_strip32<W, SPIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_spread_strip32<W, SPIN><<<strip_grid(p), 32 * kStripWarps, sm, st>>>(
        (float *)grid, p.cell, (const float2 *)p.frac, p.perm, (const float2 *)p.phase, (const float *)map, p.npts,
        p.pitch, p.R, p.ntile_c, p.ntiles, p.tile_start, p.tile_r, p.strip_part, p.kpoly);
    return cudaGetLastError();
}

}  // namespace
}  // namespace gsl
