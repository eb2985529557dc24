// Point preparation of the non-uniform FFT steps, the fixed-point scalars of a call and the entry points of
// interpolation and spreading; the kernels themselves are in nufft.cuh, compiled per precision in
// nufft_f32.cu, nufft_interp64.cu and nufft_spread64.cu.
#include <cuda_runtime.h>
#include <math.h>

#include <cub/cub.cuh>

#include "nufft.cuh"

namespace gsl {
namespace {

constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr double kPi = 3.141592653589793238462643383280;

// Grid coordinate u = t c with c = N / (2 pi) held as a double-double (c.x +
// c.y): the product's rounding error, ~1e-16 of u (up to N/2 ~ 10^4 cells),
// would otherwise move the point by about one ulp of theta, i.e. a relative
// error of ~lmax * 1e-16 in the interpolated field.  Returns the cell index
// ceil(u - W/2) and the offset u - index to full double precision.
__device__ __forceinline__ int grid_coord(double t, double2 c, double hw, double &frac)
{
    const double p = t * c.x;
    const double e = fma(t, c.x, -p) + t * c.y;
    const int i0 = (int)ceil((p + e) - hw);
    frac = (p - (double)i0) + e;  // p - i0 is exact: both lie within W of each other
    return i0;
}

__global__ void k_prep(const double *__restrict__ theta, const double *__restrict__ phi,
                       const double *__restrict__ chi, int64_t n, int N1, int N2, int W, int r_lo, int R, int pitch,
                       int spin, double2 c1, double2 c2, int tile_r, int tile_c, int rows, uint32_t *__restrict__ key,
                       int32_t *__restrict__ idx, uint32_t *__restrict__ cell_u, double2 *__restrict__ frac_u,
                       double2 *__restrict__ phase_u, unsigned *__restrict__ flags)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double th = theta[i], ph = phi[i];
    bool bad = !(isfinite(th) && isfinite(ph)) || th < 0.0 || th > kPi;
    if (bad) {
        atomicOr(flags, FLAG_DOMAIN);
        th = 0.0;
        ph = 0.0;
    }
    ph = fmod(ph, kTwoPi);
    if (ph < 0.0) ph += kTwoPi;
    if (ph >= kTwoPi) ph = 0.0;
    const double hw = 0.5 * W;
    double fu, fv;
    const int i0 = grid_coord(th, c1, hw, fu);
    int j0 = grid_coord(ph, c2, hw, fv);
    if (j0 < 0) j0 += N2;
    if (j0 >= N2) j0 -= N2;
    int row = i0 - r_lo;
    if (row < 0 || row > R - W) {  // cannot happen for theta in [0, pi]; guard the table
        atomicOr(flags, FLAG_OOB);
        row = row < 0 ? 0 : R - W;
    }
    cell_u[i] = (uint32_t)row * (uint32_t)pitch + (uint32_t)j0;
    frac_u[i] = make_double2(fu, fv);
    const int ntc = (N2 + tile_c - 1) / tile_c;
    const uint32_t tile = (uint32_t)(row / tile_r) * (uint32_t)ntc + (uint32_t)(j0 / tile_c);
    uint32_t k = tile;  // rows: by cell row within the tile, 2: then by column
    if (rows) k = k * (uint32_t)tile_r + (uint32_t)(row % tile_r);
    if (rows == 2) k = k * (uint32_t)tile_c + (uint32_t)(j0 % tile_c);
    key[i] = k;
    idx[i] = (int32_t)i;
    if (spin) {
        const double c = chi ? chi[i] : 0.0;
        double sn, cs;
        sincos(spin * c, &sn, &cs);
        phase_u[i] = make_double2(cs, sn);
    }
}

__global__ void k_gather_points(const int32_t *__restrict__ perm, int64_t n, const uint32_t *__restrict__ cell_u,
                                const double2 *__restrict__ frac_u, const double2 *__restrict__ phase_u, int prec,
                                int spin, uint32_t *__restrict__ cell, void *__restrict__ frac,
                                void *__restrict__ phase)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int32_t i = perm[p];
    cell[p] = cell_u[i];
    const double2 f = frac_u[i];
    if (prec == LENS_FP32) ((float2 *)frac)[p] = make_float2((float)f.x, (float)f.y);
    else ((double2 *)frac)[p] = f;
    if (spin) {
        const double2 ph = phase_u[i];
        if (prec == LENS_FP32) ((float2 *)phase)[p] = make_float2((float)ph.x, (float)ph.y);
        else ((double2 *)phase)[p] = ph;
    }
}

// start[t] = first sorted point whose tile (key / per) is >= t, t = 0..ntiles (the
// ranges (key[p-1], key[p]] partition 0..ntiles, so each entry is written once)
__global__ void k_tile_bounds(const uint32_t *__restrict__ skey, int64_t n, int ntiles, int per, uint32_t *__restrict__ start)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p > n) return;
    const int64_t lo = p == 0 ? -1 : (int64_t)(skey[p - 1] / per);
    const int64_t hi = p == n ? (int64_t)ntiles : (int64_t)(skey[p] / per);
    for (int64_t t = lo + 1; t <= hi; ++t) start[t] = (uint32_t)p;
}

// most[0]: points of the fullest tile; most[1]: the largest kmax (integer tiles)
__global__ void k_tile_most(const uint32_t *__restrict__ start, const unsigned short *__restrict__ kmax, int ntiles,
                            unsigned *__restrict__ most)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned c = __reduce_max_sync(0xffffffffu, t < ntiles ? start[t + 1] - start[t] : 0u);
    const unsigned k = __reduce_max_sync(0xffffffffu, t < ntiles && kmax ? (unsigned)kmax[t] : 0u);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(most, c);
        atomicMax(most + 1, k);
    }
}

// FP64 plans' 2W kernel weights of every (sorted) point, computed once, evaluated in FP64 and kept as
// doubles or (dd, plans with epsilon >= 5e-11) as double-float pairs (8 bytes
// each either way): the latter plans compute the interpolation and spreading
// taps in double-float arithmetic on the FP32 pipe, GB300's FP64 pipe running
// at 1/60 of it.
__global__ void k_weights(const double2 *__restrict__ frac, int64_t n, int W, double beta, double *__restrict__ wts,
                          int dd)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const double2 f = frac[p];
    const double twoW = 2.0 / W;
    if (dd) {  // layout: dd_words
        float *w = reinterpret_cast<float *>(wts) + p * dd_words(W);
        for (int a = 0; a < W; ++a) {
            const df32 x = df_split(es_kernel<double>(f.x - a, twoW, beta));
            const df32 y = df_split(es_kernel<double>(f.y - a, twoW, beta));
            const bool lone = (W & 1) && a == W - 1;
            const int i = lone ? 2 * a : 4 * (a >> 1) + (a & 1);
            w[i] = x.h;
            w[i + (lone ? 1 : 2)] = x.l;
            reinterpret_cast<float2 *>(w + 2 * W)[a] = make_float2(y.h, y.l);
        }
        return;
    }
    double *wd = wts + p * 2 * W;
    for (int a = 0; a < W; ++a) {
        wd[a] = es_kernel<double>(f.x - a, twoW, beta);
        wd[W + a] = es_kernel<double>(f.y - a, twoW, beta);
    }
}

// Plan time (integer-tile plans): kmax_t of every tile, the most of the tile's points
// whose W x W windows (from their first-tap cell) cover a single cell: counts
// h per first-tap cell of the tile, then window sums over W rows and W columns
// for every cell of the tile and its halo.
template <int W>
__global__ void __launch_bounds__(256) k_tile_window_kmax(const uint32_t *__restrict__ cell, int pitch, int ntc,
                                                         int tile_r,
                                                         const uint32_t *__restrict__ tile_start,
                                                         unsigned short *__restrict__ out)
{
    constexpr int TC = kTileC + W - 1;
    const int TR = tile_r + W - 1;
    extern __shared__ int kmax_smem[];
    int *h = kmax_smem;                    // [tile_r][32] points per first-tap cell (lr, lc)
    int *v = kmax_smem + tile_r * kTileC;  // [TR][32]: v[r][c] = sum over a < W of h[r - a][c]
    __shared__ int best;
    const int t = blockIdx.x;
    const uint32_t p0 = tile_start[t], p1 = tile_start[t + 1];
    for (int i = threadIdx.x; i < tile_r * kTileC; i += blockDim.x) h[i] = 0;
    if (threadIdx.x == 0) best = 0;
    __syncthreads();
    const int r0 = (t / ntc) * tile_r, c0 = (t % ntc) * kTileC;
    for (uint32_t p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const uint32_t c = cell[p];
        const int lr = (int)(c / (uint32_t)pitch) - r0, lc = (int)(c % (uint32_t)pitch) - c0;
        if ((unsigned)lr < (unsigned)tile_r && (unsigned)lc < (unsigned)kTileC) atomicAdd(&h[lr * kTileC + lc], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TR * kTileC; i += blockDim.x) {
        const int r = i / kTileC, c = i % kTileC;
        int sum = 0;
        for (int a = 0; a < W; ++a)
            if (r - a >= 0 && r - a < tile_r) sum += h[(r - a) * kTileC + c];
        v[i] = sum;
    }
    __syncthreads();
    int mx = 0;
    for (int i = threadIdx.x; i < TR * TC; i += blockDim.x) {
        const int r = i / TC, c = i % TC;
        int sum = 0;
        for (int b = 0; b < W; ++b)
            if (c - b >= 0 && c - b < kTileC) sum += v[r * kTileC + c - b];
        mx = max(mx, sum);
    }
    atomicMax(&best, mx);
    __syncthreads();
    if (threadIdx.x == 0) out[t] = (unsigned short)min(best, 65535);
}

// ---------------------------------------------- fixed point (deterministic plans)
// Largest |x| (spin 0) or |Q| + |U| (spin s) of a map, as the bits of a
// non-negative double, which order like unsigned integers (a NaN input gives
// NaN bits, above those of infinity).
template <typename T, bool SPIN>
__global__ void k_fx_maxabs(const T *__restrict__ map, int64_t n, unsigned long long *__restrict__ out)
{
    double a = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = SPIN ? fabs((double)map[i]) + fabs((double)map[n + i]) : fabs((double)map[i]);
        a = (v > a || v != v) ? v : a;
    }
    unsigned long long b = (unsigned long long)__double_as_longlong(a);
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, b, off);
        b = o > b ? o : b;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(out, b);
}

// unit[0] = 2^k with k the largest integer (up to 122) such that
// Kmax max|x| 2^k <= 2^62; NaN when the bound is not finite
__global__ void k_fx_grid_unit(const unsigned long long *__restrict__ maxbits, const uint32_t *__restrict__ kmax,
                               double *__restrict__ unit)
{
    unit[0] = fx_unit((double)*kmax * __longlong_as_double((long long)*maxbits));
}

// grid[i] = fx[i] / unit in the plan's precision (fx and grid may coincide)
template <typename T>
__global__ void k_fx_to_grid(const unsigned long long *fx, T *grid, int64_t n, const double *__restrict__ unit)
{
    const double inv = 1.0 / unit[0];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        grid[i] = fx_value<T>((long long)fx[i], inv);
}

// Kmax: the most points any cell can receive (a tile's count plus those of
// its left, upper and upper-left neighbours); start as k_tile_bounds writes it
__global__ void k_tile_kmax(const uint32_t *__restrict__ start, int ntr, int ntc, uint32_t *__restrict__ kmax)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ntr * ntc) return;
    const int tr = t / ntc, tc = t % ntc;
    auto cnt = [&](int r, int c) -> uint32_t {
        if (r < 0 || c < 0) return 0u;
        const int u = r * ntc + c;
        return start[u + 1] - start[u];
    };
    atomicMax(kmax, cnt(tr, tc) + cnt(tr, tc - 1) + cnt(tr - 1, tc) + cnt(tr - 1, tc - 1));
}

}  // namespace

// per precision (nufft_f32.cu, nufft_interp64.cu, nufft_spread64.cu)
cudaError_t interp_f32(const Plan &p, const void *grid, void *map, cudaStream_t st);
cudaError_t interp_f64(const Plan &p, const void *grid, void *map, cudaStream_t st);
cudaError_t spread_f32(const Plan &p, const void *map, void *grid, cudaStream_t st);
cudaError_t spread_f64(const Plan &p, const void *map, void *grid, cudaStream_t st);

cudaError_t launch_interp(const Plan &p, const void *grid, void *map, cudaStream_t st)
{
    return p.prec == LENS_FP32 ? interp_f32(p, grid, map, st) : interp_f64(p, grid, map, st);
}

cudaError_t launch_spread(const Plan &p, const void *map, void *grid, cudaStream_t st)
{
    const size_t eb = (p.prec == LENS_FP32 ? 4 : 8) * (p.spin ? 2 : 1);
    const size_t ncell = (size_t)p.R * p.pitch * (p.spin ? 2 : 1);
    cudaError_t e = cudaMemsetAsync(grid, 0, eb * (size_t)p.R * p.pitch, st);
    if (e != cudaSuccess) return e;
    const bool f32 = p.prec == LENS_FP32;
    if (!p.det) {
        if (p.tile_kmax) {  // fixed-point tiles: the map's largest |value| first
            if ((e = cudaMemsetAsync(p.maxbits, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
            if (p.npts > 0) {
                const unsigned mb = (unsigned)std::min<int64_t>((p.npts + 255) / 256, 152 * 8);
                if (f32) {
                    if (p.spin) k_fx_maxabs<float, true><<<mb, 256, 0, st>>>((const float *)map, p.npts, p.maxbits);
                    else k_fx_maxabs<float, false><<<mb, 256, 0, st>>>((const float *)map, p.npts, p.maxbits);
                } else {
                    if (p.spin) k_fx_maxabs<double, true><<<mb, 256, 0, st>>>((const double *)map, p.npts, p.maxbits);
                    else k_fx_maxabs<double, false><<<mb, 256, 0, st>>>((const double *)map, p.npts, p.maxbits);
                }
                if ((e = cudaGetLastError()) != cudaSuccess) return e;
            }
        }
        return f32 ? spread_f32(p, map, grid, st) : spread_f64(p, map, grid, st);
    }
    // fixed point: FP32 plans accumulate in their own int64 grid, FP64 plans in place
    void *fxg = f32 ? p.fx_grid : grid;
    if (f32 && (e = cudaMemsetAsync(fxg, 0, 8 * ncell, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(p.fx_maxbits, 0, sizeof(unsigned long long), st)) != cudaSuccess) return e;
    const unsigned mb = (unsigned)std::min<int64_t>((p.npts + 255) / 256, 152 * 8);
    if (p.npts > 0) {
        if (f32) {
            if (p.spin) k_fx_maxabs<float, true><<<mb, 256, 0, st>>>((const float *)map, p.npts, p.fx_maxbits);
            else k_fx_maxabs<float, false><<<mb, 256, 0, st>>>((const float *)map, p.npts, p.fx_maxbits);
        } else {
            if (p.spin) k_fx_maxabs<double, true><<<mb, 256, 0, st>>>((const double *)map, p.npts, p.fx_maxbits);
            else k_fx_maxabs<double, false><<<mb, 256, 0, st>>>((const double *)map, p.npts, p.fx_maxbits);
        }
    }
    k_fx_grid_unit<<<1, 1, 0, st>>>(p.fx_maxbits, p.fx_kmax, p.fx_scale);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = f32 ? spread_f32(p, map, fxg, st) : spread_f64(p, map, fxg, st);
    if (e != cudaSuccess) return e;
    const unsigned cb = (unsigned)std::min<size_t>((ncell + 255) / 256, 152 * 16);
    if (f32) k_fx_to_grid<float><<<cb, 256, 0, st>>>((const unsigned long long *)fxg, (float *)grid, ncell, p.fx_scale);
    else k_fx_to_grid<double><<<cb, 256, 0, st>>>((const unsigned long long *)fxg, (double *)grid, ncell, p.fx_scale);
    return cudaGetLastError();
}

// Point preparation: validate, compute cells/offsets/phases in user order,
// radix-sort by tile key, gather into sorted order.  Temporary buffers are
// released before returning; the stream is synchronised once.
cudaError_t launch_prep_points(Plan &p, const double *theta, const double *phi, const double *chi,
                               cudaStream_t st, std::string &err)
{
    const int64_t n = p.npts;
    if (n == 0) return cudaSuccess;
    if (n > (int64_t)0x7fffffff) { err = "npoints above 2^31 - 1"; return cudaErrorInvalidValue; }
    uint32_t *key = nullptr, *key2 = nullptr, *cell_u = nullptr;
    int32_t *idx = nullptr;
    double2 *frac_u = nullptr, *phase_u = nullptr;
    void *tmp = nullptr;
    size_t tmp_bytes = 0;
    cudaError_t e = cudaSuccess;
    auto cleanup = [&]() {
        cudaFree(key); cudaFree(key2); cudaFree(cell_u); cudaFree(idx);
        cudaFree(frac_u); cudaFree(phase_u); cudaFree(tmp);
    };
#define GSL_TRY(x) do { e = (x); if (e != cudaSuccess) { cleanup(); return e; } } while (0)
    GSL_TRY(cudaMalloc(&key, n * sizeof(uint32_t)));
    GSL_TRY(cudaMalloc(&key2, n * sizeof(uint32_t)));
    GSL_TRY(cudaMalloc(&idx, n * sizeof(int32_t)));
    GSL_TRY(cudaMalloc(&cell_u, n * sizeof(uint32_t)));
    GSL_TRY(cudaMalloc(&frac_u, n * sizeof(double2)));
    if (p.spin) GSL_TRY(cudaMalloc(&phase_u, n * sizeof(double2)));
    GSL_TRY(cudaMemsetAsync(p.flags, 0, sizeof(unsigned), st));
    const int thr = 256;
    const unsigned blocks = (unsigned)((n + thr - 1) / thr);
    // N / (2 pi) as double-doubles: quotient of N by 2 pi = T_HI + T_LO, refined once
    auto scale_of = [](int N) {
        const double th = 6.283185307179586232, tl = 2.4492935982947064e-16;
        const double q1 = N / th;
        const double p = q1 * th, pe = fma(q1, th, -p);
        const double r = (((double)N - p) - pe) - q1 * tl;
        const double q2 = r / th;
        const double hi = q1 + q2;
        return make_double2(hi, q2 - (hi - q1));
    };
    const int ntc = p.ntile_c;
    const uint64_t nkeys = (uint64_t)((p.R + p.tile_r - 1) / p.tile_r) * ntc;
    // Order within a tile, where the keys fit 32 bits.  Strips need rows.  The interpolation gains from rows and columns from 2^17
    // points on (fewer: within 1 us, and the longer keys cost plan creation, lmax 128 1.28 -> 1.44 ms).  Integer tiles pay for
    // columns with conflicts of their shared atomics, the more the more points share a cell, so from 3/4 points per cell on
    // they take rows alone.  us of spreading and interpolation, rows and columns / rows, FP32, spin 2:
    //   0.5 points per cell (lmax 2048, Nside 1024, W 7)    687 + 314 / 656 + 367
    //   0.8 (lmax 2048, Nside 1280, W 7)                   1036 + 451 / 963 + 529
    //   1.1 (lmax 2048, Nside 2048, W 6)                   2210 + 1022 / 1961 + 1170
    //   4.6 (lmax 1024, Nside 2048, W 6)                   3554 + 952 / 1792 + 995
    //   18 (lmax 512, Nside 2048, W 6)                     8035 + 927 / 2273 + 917
    const bool fit = nkeys * p.tile_r * p.tile_c <= 0xffffffffull;
    const bool dense = 4.0 * (double)n >= 3.0 * (0.5 * p.N1) * p.N2;
    const bool tiles64 = p.prec == LENS_FP64 && p.tile_kmax;  // FP64 interpolation without strips: nothing to gain
    const int rows = p.strip ? (fit ? 2 : 1) : n >= (1 << 17) && fit && !tiles64 ? (dense ? 1 : 2) : 0;
    p.sorted = rows > 0;
    const int per = rows == 2 ? p.tile_r * p.tile_c : rows ? p.tile_r : 1;
    k_prep<<<blocks, thr, 0, st>>>(theta, phi, chi, n, p.N1, p.N2, p.W, p.r_lo, p.R, p.pitch, p.spin, scale_of(p.N1),
                                   scale_of(p.N2), p.tile_r, p.tile_c, rows, key, idx, cell_u, frac_u, phase_u, p.flags);
    GSL_TRY(cudaGetLastError());
    int bits = 1;
    while (bits < 32 && (1ull << bits) < nkeys * per) ++bits;
    GSL_TRY(cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, key, key2, idx, p.perm, (int)n, 0, bits, st));
    GSL_TRY(cudaMalloc(&tmp, tmp_bytes));
    GSL_TRY(cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, key, key2, idx, p.perm, (int)n, 0, bits, st));
    k_gather_points<<<blocks, thr, 0, st>>>(p.perm, n, cell_u, frac_u, phase_u, p.prec, p.spin, p.cell, p.frac,
                                            p.phase);
    GSL_TRY(cudaGetLastError());
    if (nkeys != (uint64_t)p.ntiles) { cleanup(); err = "internal: tile count mismatch"; return cudaErrorInvalidValue; }
    k_tile_bounds<<<(unsigned)((n + 1 + thr - 1) / thr), thr, 0, st>>>(key2, n, p.ntiles, per, p.tile_start);
    GSL_TRY(cudaGetLastError());
    if (p.det) {
        GSL_TRY(cudaMemsetAsync(p.fx_kmax, 0, sizeof(uint32_t), st));
        k_tile_kmax<<<(unsigned)((p.ntiles + thr - 1) / thr), thr, 0, st>>>(p.tile_start, p.ntiles / ntc, ntc, p.fx_kmax);
        GSL_TRY(cudaGetLastError());
    }
    if (p.tile_kmax) {  // fixed-point spreading tiles: kmax_t per tile
        const size_t sm = sizeof(int) * (size_t)kTileC * (2 * p.tile_r + p.W - 1);
        const auto run = [&](auto kern) {
            kern<<<(unsigned)p.ntiles, 256, sm, st>>>(p.cell, p.pitch, ntc, p.tile_r, p.tile_start, p.tile_kmax);
        };
        switch (p.W) {
        case 4: run(k_tile_window_kmax<4>); break;
        case 5: run(k_tile_window_kmax<5>); break;
        case 6: run(k_tile_window_kmax<6>); break;
        case 7: run(k_tile_window_kmax<7>); break;
        case 8: run(k_tile_window_kmax<8>); break;
        case 9: run(k_tile_window_kmax<9>); break;
        case 10: run(k_tile_window_kmax<10>); break;
        case 11: run(k_tile_window_kmax<11>); break;
        case 12: run(k_tile_window_kmax<12>); break;
        case 13: run(k_tile_window_kmax<13>); break;
        case 14: run(k_tile_window_kmax<14>); break;
        case 15: run(k_tile_window_kmax<15>); break;
        default: run(k_tile_window_kmax<16>); break;
        }
        GSL_TRY(cudaGetLastError());
    }
    if (p.wts) {
        k_weights<<<blocks, thr, 0, st>>>((const double2 *)p.frac, n, p.W, p.beta, p.wts, p.wts_dd ? 1 : 0);
        GSL_TRY(cudaGetLastError());
    }
    if (!p.det) {
        GSL_TRY(cudaMemsetAsync(p.flags + 2, 0, 2 * sizeof(unsigned), st));
        k_tile_most<<<(unsigned)((p.ntiles + thr - 1) / thr), thr, 0, st>>>(p.tile_start, p.tile_kmax, p.ntiles, p.flags + 2);
        GSL_TRY(cudaGetLastError());
    }
    unsigned hf[4] = {0, 0, 0, 0};
    GSL_TRY(cudaMemcpyAsync(hf, p.flags, sizeof(hf), cudaMemcpyDeviceToHost, st));
    GSL_TRY(cudaStreamSynchronize(st));
    const unsigned hflags = hf[0], most = p.det ? 0 : hf[2];
    // Tiles with many points are shared by up to 64 warps or CTAs, more where the grid has few tiles
    const unsigned share = (unsigned)std::min(std::max((1 << 16) / p.ntiles, 64), 1024);
    p.parts = 1;
    if (p.strip && most > 0) {
        // A warp sweeps at most 4096 points (uniform skies have ~1000 per tile; a survey patch may pile its points into one
        // tile); fewer, down to one batch of 32, where the points lie in so few tiles that their warps would not fill the chip:
        // us with parts of 4096 / as now, FP64 W 13 at lmax 128, 49,152 points, spin 0 56 / 36, spin 2 72 / 51; FP32 W 12,
        // lmax 82, 13,584 points, spin 0 26 / 13
        p.strip_part = 4096;
        if ((uint64_t)most * 152 * 8 > (uint64_t)n)
            while (p.strip_part > 32 && (uint64_t)p.strip_part * 152 * 16 > 2 * (uint64_t)n) p.strip_part /= 2;
        while ((uint64_t)p.strip_part * share < most) p.strip_part *= 2;
        p.parts = (int)((most - 1) / p.strip_part + 1);
    } else if (p.tile_kmax && hf[3] >= (p.prec == LENS_FP32 ? kPassFrom<float> : kPassFrom<double>)) {
        const unsigned pass = p.prec == LENS_FP32 ? kPassPoints<float> : kPassPoints<double>;
        p.piles = true;
        p.parts = (int)std::min((most - 1) / pass + 1, share);
    }
#undef GSL_TRY
    cleanup();
    if (hflags & FLAG_DOMAIN) { err = "a coordinate is not finite or theta is outside [0, pi]"; return cudaErrorInvalidValue; }
    if (hflags & FLAG_OOB) { err = "internal: a point fell outside the kept rows"; return cudaErrorInvalidValue; }
    return cudaSuccess;
}

}  // namespace gsl
