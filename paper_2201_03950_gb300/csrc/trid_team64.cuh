// trid_team64.cuh -- FP64 systems of 256 < N <= 4096 rows in one pass (the
// tiled hybrid of Section 3.1, one block per SG neighbouring systems).
//
// Every thread keeps a tile of 16 rows in registers through the whole solve:
// tile_reduce, the block's reduced systems folded to one unknown per tile and
// solved by PCR in shared memory (stopping once the couplings are below 1/16
// ulp), tile_substitute.  FP64 arithmetic bounds these solves: reducing,
// solving and substituting once takes about 17 operations per row, where the
// passes through scratch reduce every row twice (9 + 3 operations, then 8
// between the known ends) and once more for the rows of the reduced systems,
// about 25.  Measured, passes -> this: 3000 x 1400 along x 217 -> 148 us, along
// y 212 -> 154; 4096 x 4096 along x 702 -> 593; 500 x 8000 along x 182 -> 131; 60
// systems of 600 rows 32 -> 15.
#pragma once
#include "trid_device.cuh"
#include "trid_twist.cuh"

namespace trid {

constexpr int TM_M = 16;             // rows per thread
constexpr int TM_MAX_TILES = 256;
constexpr int TM_THREADS = 384;     // at most: 140 registers a thread

// Shared memory: two buffers of the folded rows (ra, rc, rd), the S rows'
// values (as, cs, ds) of every tile, and x_e.
__host__ inline size_t team64_smem(int tiles, int sg) {
    return size_t(tiles) * sg * 9 * sizeof(double);
}

// MODE 0: strided systems (or any); 1: contiguous systems in whole 32-byte
// vectors.  Thread t: system t % SG of the block's, tile t / SG.
template <int SG, int MODE>
__global__ void __launch_bounds__(TM_THREADS)
k_team64(const double *__restrict__ a, const double *__restrict__ b, const double *__restrict__ c,
         const double *d, double *out, int accumulate, Lines L, int tiles) {
    constexpr int M = TM_M;
    extern __shared__ __align__(16) double sm_tm[];
    const int nt = tiles * SG;       // values per table
    double *ra0 = sm_tm, *rc0 = sm_tm + nt, *rd0 = sm_tm + 2 * nt;
    double *ra1 = sm_tm + 3 * nt, *rc1 = sm_tm + 4 * nt, *rd1 = sm_tm + 5 * nt;
    double *s_as = sm_tm + 6 * nt, *s_cs = sm_tm + 7 * nt, *s_ds = sm_tm + 8 * nt;
    const int t = threadIdx.x;
    const int sl = t % SG, tile = t / SG;
    const bool on = tile < tiles;    // threads beyond the tiles only meet the barriers
    const int n = int(L.n), stride = int(L.stride);
    const int64_t sys = int64_t(blockIdx.x) * SG + sl;
    const int i0 = tile * M;
    const int64_t base = sys < L.nsys ? L.base(sys) : 0;
    const bool active = on && sys < L.nsys &&
                        TRID_BOUNDS(base + int64_t(n - 1) * stride < L.nsys * L.n);

    double ra[M], rb[M], rc[M], rd[M];
    if (MODE == 1 && active && i0 + M <= n) {
#pragma unroll
        for (int q = 0; q < M; q += 4) {
            double v[4];
            ld_f64x4(a + base + i0 + q, v);
#pragma unroll
            for (int j = 0; j < 4; ++j) ra[q + j] = v[j];
            ld_f64x4(b + base + i0 + q, v);
#pragma unroll
            for (int j = 0; j < 4; ++j) rb[q + j] = v[j];
            ld_f64x4(c + base + i0 + q, v);
#pragma unroll
            for (int j = 0; j < 4; ++j) rc[q + j] = v[j];
            ld_f64x4(d + base + i0 + q, v);
#pragma unroll
            for (int j = 0; j < 4; ++j) rd[q + j] = v[j];
        }
    } else {
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const int i = i0 + j;
            if (active && i < n) {
                const int64_t p = base + int64_t(i) * stride;
                ra[j] = a[p]; rb[j] = b[p]; rc[j] = c[p]; rd[j] = d[p];
            } else {
                ra[j] = 0.0; rb[j] = 1.0; rc[j] = 0.0; rd[j] = 0.0;
            }
        }
    }
    if (i0 == 0) ra[0] = 0.0;
#pragma unroll
    for (int j = 0; j < M; ++j)
        if (i0 + j == n - 1) rc[j] = 0.0;
    double as, cs, ds, ae, ce, de;
    tile_reduce<double, M>(ra, rb, rc, rd, as, cs, ds, ae, ce, de);
    if (on) { s_as[t] = as; s_cs[t] = cs; s_ds[t] = ds; }
    __syncthreads();
    // fold the next tile's S row into the E row (as group_solve), then PCR over
    // the tiles of each system: neighbours at distance s are s * SG values away
    double fa = 0.0, fc = 0.0, fd = 0.0;
    if (on) {
        const bool nx = tile + 1 < tiles;
        const double nas = nx ? s_as[t + SG] : 0.0, ncs = nx ? s_cs[t + SG] : 0.0;
        const double nds = nx ? s_ds[t + SG] : 0.0;
        const double r = rcp(1.0 - ae * cs - ce * nas);
        fa = -(ae * as) * r;
        fc = -(ce * ncs) * r;
        fd = (de - ae * ds - ce * nds) * r;
    }
    for (int s = 1; s < tiles; s <<= 1) {
        if (on) { ra0[t] = fa; rc0[t] = fc; rd0[t] = fd; }
        const bool big = fmax(fabs(fa), fabs(fc)) >= 6.9388939039072284e-18;   // 2^-57
        if (!__syncthreads_or(big)) break;
        if (on) {
            const bool lo = tile >= s, hi = tile + s < tiles;
            const int m = t - s * SG, q = t + s * SG;
            const double am = lo ? ra0[m] : 0.0, cm = lo ? rc0[m] : 0.0, dm = lo ? rd0[m] : 0.0;
            const double ap = hi ? ra0[q] : 0.0, cp = hi ? rc0[q] : 0.0, dp = hi ? rd0[q] : 0.0;
            const double r = rcp(1.0 - fa * cm - fc * ap);
            fd = r * (fd - fa * dm - fc * dp);
            fa = -r * (fa * am);
            fc = -r * (fc * cp);
        }
        double *w = ra0; ra0 = ra1; ra1 = w;   // the next round writes the other buffer
        w = rc0; rc0 = rc1; rc1 = w;
        w = rd0; rd0 = rd1; rd1 = w;
    }
    __syncthreads();
    if (on) rd0[t] = fd;
    __syncthreads();
    const double xp = on && tile > 0 ? rd0[t - SG] : 0.0;
    const double xs = ds - as * xp - cs * fd;
    tile_substitute<double, M>(ra, rc, rd, xs, fd);
    if (!active) return;
    double *ob = out + base;
    if (MODE == 1 && i0 + M <= n) {
#pragma unroll
        for (int q = 0; q < M; q += 4) {
            double v[4];
            if (accumulate) ld_f64x4(ob + i0 + q, v);
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = accumulate ? v[j] + rd[q + j] : rd[q + j];
            st_f64x4(ob + i0 + q, v);
        }
    } else {
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const int i = i0 + j;
            if (i < n) {
                double *p = ob + int64_t(i) * stride;
                *p = accumulate ? *p + rd[j] : rd[j];
            }
        }
    }
}

}  // namespace trid
