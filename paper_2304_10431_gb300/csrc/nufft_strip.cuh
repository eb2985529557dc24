// Spreading of FP64 plans with double-float weights (epsilon >= 5e-11): tiles swept row by row in registers.
//
// One warp owns a tile of tile_r rows x (33 - W) columns, so the W-wide windows of its points cover 32
// columns: lane c holds column c of the W rows that the points of one cell row touch, as sums of row pairs
// (f32x2 instructions).  The points are sorted by cell row (plan creation); after the points of a
// row, its grid row receives nothing more from this tile: the lane adds it into the grid with one atomic and
// the window moves down a row.  No shared-memory accumulation: the tiles of 64-bit integers that this replaces
// were bound by shared-memory atomics (1.1 taps per clock and SM; 24.2 ms for spin 0 and 42 ms for spin 2
// at lmax 4096, 50M points, W = 13).  A point costs the whole warp W/2 multiply-adds of a pair, whatever part
// of the 32 columns it covers (W = 13: 41%).
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
constexpr int kStripBatch = 16;  // points per weight copy

template <int W> __host__ __device__ constexpr size_t strip_warp_smem()
{
    // two weight buffers, values (float4), offsets (int), two mbarriers
    return 2 * kStripBatch * dd_words(W) * sizeof(float) + kStripBatch * (sizeof(float4) + sizeof(int)) + 16;
}

template <int W, bool SPIN>
__global__ void __launch_bounds__(32 * kStripWarps)
k_spread_strip(double *__restrict__ grid, const uint32_t *__restrict__ cell, const int32_t *__restrict__ perm,
               const double2 *__restrict__ phase, const double *__restrict__ wts, const double *__restrict__ map,
               int64_t n, int pitch, int R, int ntc, int ntiles, const uint32_t *__restrict__ tile_start, int tile_r,
               unsigned *__restrict__ status)
{
    constexpr int NP = dd_pairs(W), NC = SPIN ? 2 : 1, TC = 33 - W;
    constexpr uint32_t WBYTES = dd_words(W) * sizeof(float);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int t = blockIdx.x * kStripWarps + wid;
    if (t >= ntiles) return;
    const uint32_t p0 = tile_start[t], p1 = tile_start[t + 1];
    if (p0 == p1) return;
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

    // the tile's largest |value| (spin s: Q^2 + U^2) as the bits of a non-negative double
    unsigned long long mx = 0;
    for (uint32_t p = p0 + lane; p < p1; p += 32) {
        const int32_t src = perm[p];
        const double q = map[src], v = SPIN ? fma(q, q, map[n + src] * map[n + src]) : fabs(q);
        const unsigned long long b = (unsigned long long)__double_as_longlong(v);
        mx = b > mx ? b : mx;  // infinities and NaNs order above the finite values
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        mx = o > mx ? o : mx;
    }
    double top = __longlong_as_double((long long)mx);
    if (SPIN) top = sqrt(top);
    const bool bad = !(top < 1e300);  // infinity or NaN: the tile becomes NaN
    int ex = bad || top == 0.0 ? 0 : -ilogb(top);
    ex = min(max(ex, -1000), 1000);
    const double sc = ldexp(1.0, ex), inv = bad ? NAN : ldexp(1.0, -ex);

    const int r0 = (t / ntc) * tile_r, c0 = (t % ntc) * TC;
    D2 S[NC][NP];
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int i = 0; i < NP; ++i) S[c][i] = {0ull, 0ull};
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
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                S[c][i].h = pk_make(pk_get(S[c][i].h).y, i + 1 < NP ? pk_get(S[c][i + 1 < NP ? i + 1 : i].h).x : 0.f);
                S[c][i].l = pk_make(pk_get(S[c][i].l).y, i + 1 < NP ? pk_get(S[c][i + 1 < NP ? i + 1 : i].l).x : 0.f);
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
                       ? *reinterpret_cast<const float2 *>(wbuf + q * dd_words(W) + 4 * NP + 2 * b)
                       : make_float2(0.f, 0.f);
        };
        float2 wb = column(0, so);
#pragma unroll 1
        for (int q = 0; q < cnt; ++q) {
            const float *w = wbuf + q * dd_words(W);
            const int row = so >> 8;  // (-1 for a point of no tile: no row to move to, weights zero)
            D2 v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const df32 t = df_mul(df32{wb.x, wb.y}, c == 0 ? df32{xv.x, xv.y} : df32{xv.z, xv.w});
                v[c] = {pk_make(t.h, t.h), pk_make(t.l, t.l)};
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
        }
        // keep the low words below an ulp of the sums (2,000 points in one cell, unnormalised: 2e-12 of the a_lm)
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int i = 0; i < NP; ++i) S[c][i] = d2_norm(S[c][i]);
        __syncwarp();  // the buffers are rewritten by the next batch
    }
    if (!ok && lane == 0) atomicOr(status, FLAG_TIMEOUT);
    const int last = min(tile_r + W - 1, bad ? 1 << 20 : cur + W);  // rows the last points reach
    while (cur < last) next_row();
}

template <int W, bool SPIN> cudaError_t spread_strip(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    const auto kern = k_spread_strip<W, SPIN>;
    const size_t sm = kStripWarps * strip_warp_smem<W>();
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((p.ntiles + kStripWarps - 1) / kStripWarps), 32 * kStripWarps, sm, st>>>(
        (double *)grid, p.cell, p.perm, (const double2 *)p.phase, p.wts, (const double *)map, p.npts, p.pitch, p.R,
        p.ntile_c, p.ntiles, p.tile_start, p.tile_r, p.flags + 1);
    return cudaGetLastError();
}

}  // namespace
}  // namespace gsl
