// trid_team.cuh -- long systems in one pass (the tiled hybrid of Section 3.1, one
// block per SG neighbouring systems): FP64 of 256 < N <= 4096 rows, and the FP32
// systems of up to 8192 rows that neither the bulk-copy teams nor the clusters
// take.
//
// Every thread keeps a tile of 16 rows in registers through the whole solve:
// tile_reduce, the block's reduced systems folded to one unknown per tile and
// solved by PCR in shared memory (stopping once the couplings are below 1/16
// ulp), tile_substitute.  In FP64, arithmetic bounds these solves: reducing,
// solving and substituting once takes about 17 operations per row, where the
// passes through scratch reduce every row (12), run over it again between the
// known ends (8) and solve the reduced systems recursively, about 25.  Measured,
// passes -> this: 3000 x 1400 along x 217 -> 148 us, along y 212 -> 154; 4096 x 4096
// along x 702 -> 593; 500 x 8000 along x 182 -> 131; 60 systems of 600 rows 32 -> 15.
// In FP32 it saves the second reading of every array and four launches: see the
// launcher.
#pragma once
#include "trid_device.cuh"

namespace trid {

constexpr int TM_M = 16;             // rows per thread
template <typename T>
__host__ __device__ constexpr int tm_threads() { return sizeof(T) == 8 ? 384 : 512; }  // at most

// Shared memory: two buffers of the folded rows (ra, rc, rd), the S rows'
// values (as, cs, ds) of every tile.
template <typename T>
__host__ inline size_t team_smem(int tiles, int sg) {
    return size_t(tiles) * sg * 9 * sizeof(T);
}

// MODE 0: strided systems (or any); 1: contiguous systems in whole 16-byte
// vectors (out: also unaligned).  Thread t: system t % SG of the block's, tile t / SG.
template <typename T, int SG, int MODE>
__global__ void __launch_bounds__(tm_threads<T>())
k_team(const T *__restrict__ a, const T *__restrict__ b, const T *__restrict__ c, const T *d,
       T *out, int accumulate, Lines L, int tiles) {
    constexpr int M = TM_M;
    constexpr T negligible = sizeof(T) == 4 ? T(3.7252903e-09) : T(6.9388939039072284e-18);  // 2^-(p + 4)
    extern __shared__ __align__(16) unsigned char smem_tm[];
    T *sm_tm = reinterpret_cast<T *>(smem_tm);
    const int nt = tiles * SG;       // values per table
    T *ra0 = sm_tm, *rc0 = sm_tm + nt, *rd0 = sm_tm + 2 * nt;
    T *ra1 = sm_tm + 3 * nt, *rc1 = sm_tm + 4 * nt, *rd1 = sm_tm + 5 * nt;
    T *s_as = sm_tm + 6 * nt, *s_cs = sm_tm + 7 * nt, *s_ds = sm_tm + 8 * nt;
    const int t = threadIdx.x;
    const int sl = t % SG, tile = t / SG;
    const bool on = tile < tiles;    // threads beyond the tiles only meet the barriers
    const int n = int(L.n), stride = int(L.stride);
    const int64_t sys = int64_t(blockIdx.x) * SG + sl;
    const int i0 = tile * M;
    const int64_t base = sys < L.nsys ? L.base(sys) : 0;
    const bool active = on && sys < L.nsys &&
                        TRID_BOUNDS(base + int64_t(n - 1) * stride < L.nsys * L.n);

    T ra[M], rb[M], rc[M], rd[M];
    if (MODE == 1 && active && i0 + M <= n) {
        load_contig_vec<T, M>(a + base + i0, ra);
        load_contig_vec<T, M>(b + base + i0, rb);
        load_contig_vec<T, M>(c + base + i0, rc);
        load_contig_vec<T, M>(d + base + i0, rd);
    } else {
#pragma unroll
        for (int j = 0; j < M; ++j) {
            const int i = i0 + j;
            if (active && i < n) {
                const int64_t p = base + int64_t(i) * stride;
                ra[j] = a[p]; rb[j] = b[p]; rc[j] = c[p]; rd[j] = d[p];
            } else {
                ra[j] = T(0); rb[j] = T(1); rc[j] = T(0); rd[j] = T(0);
            }
        }
    }
    if (i0 == 0) ra[0] = T(0);
#pragma unroll
    for (int j = 0; j < M; ++j)
        if (i0 + j == n - 1) rc[j] = T(0);
    T as, cs, ds, ae, ce, de;
    tile_reduce<T, M>(ra, rb, rc, rd, as, cs, ds, ae, ce, de);
    if (on) { s_as[t] = as; s_cs[t] = cs; s_ds[t] = ds; }
    __syncthreads();
    // fold the next tile's S row into the E row (as group_solve), then PCR over
    // the tiles of each system: neighbours at distance s are s * SG values away
    T fa = T(0), fc = T(0), fd = T(0);
    if (on) {
        const bool nx = tile + 1 < tiles;
        const T nas = nx ? s_as[t + SG] : T(0), ncs = nx ? s_cs[t + SG] : T(0);
        const T nds = nx ? s_ds[t + SG] : T(0);
        const T r = rcp(T(1) - ae * cs - ce * nas);
        fa = -(ae * as) * r;
        fc = -(ce * ncs) * r;
        fd = (de - ae * ds - ce * nds) * r;
    }
    for (int s = 1; s < tiles; s <<= 1) {
        if (on) { ra0[t] = fa; rc0[t] = fc; rd0[t] = fd; }
        // (a coupling that is no number counts: it goes on to the whole system)
        const bool big = !(fmax(fabs(fa), fabs(fc)) < negligible);
        if (!__syncthreads_or(big)) break;
        if (on) {
            const bool lo = tile >= s, hi = tile + s < tiles;
            const int m = t - s * SG, q = t + s * SG;
            const T am = lo ? ra0[m] : T(0), cm = lo ? rc0[m] : T(0), dm = lo ? rd0[m] : T(0);
            const T ap = hi ? ra0[q] : T(0), cp = hi ? rc0[q] : T(0), dp = hi ? rd0[q] : T(0);
            const T r = rcp(T(1) - fa * cm - fc * ap);
            fd = r * (fd - fa * dm - fc * dp);
            fa = -r * (fa * am);
            fc = -r * (fc * cp);
        }
        T *w = ra0; ra0 = ra1; ra1 = w;   // the next round writes the other buffer
        w = rc0; rc0 = rc1; rc1 = w;
        w = rd0; rd0 = rd1; rd1 = w;
    }
    __syncthreads();
    if (on) rd0[t] = fd;
    __syncthreads();
    const T xp = on && tile > 0 ? rd0[t - SG] : T(0);
    const T xs = ds - as * xp - cs * fd;
    tile_substitute<T, M>(ra, rc, rd, xs, fd);
    if (!active) return;
    T *ob = out + base;
    if (MODE == 1 && (reinterpret_cast<uintptr_t>(ob) & 15) == 0 && i0 + M <= n) {
        if (accumulate) {
            T ru[M];
            load_contig_vec<T, M>(ob + i0, ru);
#pragma unroll
            for (int j = 0; j < M; ++j) rd[j] += ru[j];
        }
        store_contig_vec<T, M>(ob + i0, rd);
    } else {
        if (accumulate) {                // every load before the first store
            T ru[M];
#pragma unroll
            for (int j = 0; j < M; ++j)
                ru[j] = i0 + j < n ? ob[int64_t(i0 + j) * stride] : T(0);
#pragma unroll
            for (int j = 0; j < M; ++j) rd[j] += ru[j];
        }
#pragma unroll
        for (int j = 0; j < M; ++j)
            if (i0 + j < n) ob[int64_t(i0 + j) * stride] = rd[j];
    }
}

}  // namespace trid
