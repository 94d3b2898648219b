// trid_twist.cuh -- FP64 systems of up to 256 rows, solved from both ends
// (Algorithm "thomas" of Section 2 run downwards on the first half of a
// system's rows and upwards on the second half, the two meeting in a 2 x 2
// system: a twisted factorisation).
//
// FP64 arithmetic bounds these solves, not HBM: the FP64 pipe does 527 G
// operations/s, so 256^3 unknowns take 32 us per operation and row, against
// 99 us for all the bytes.  One warp per scheduler already fills the pipe
// (measured: 4 warps per SM with one dependent chain each reach 521 G/s), so
// nothing is won by cutting a system into many tiles, which costs three fill-in
// terms per row and a reduced solve (about 22 operations per row with the
// tiles of 8 rows).  Thomas needs 8 with the reciprocal below; the two ends
// give two threads per system at no extra operation.
//
// Lanes 0..15 of a warp own the upper halves of 16 systems, lanes 16..31 the
// lower halves of the same systems; the code is the same for both with the
// roles of a and c swapped and the row step negated.  Rows are loaded R ahead
// of their use.  The normalised super-diagonals c' stay in shared memory
// (256 bytes per row pair and warp), the eliminated right-hand sides d' are
// kept in the output array, each overwritten by its unknown on the way back
// (mostly from the L2); when the solution is added to `out` instead of
// stored, d' stays in shared memory too.
//
// Measured, 65536 systems of 256 rows: strided 305 us (749 us with the tiles
// of 8 rows and IEEE quotients, 655 us with this file's reciprocal there too),
// contiguous 381 us (690, 596).  8 operations for 16.8 M unknowns are 255 us
// of the pipe; contiguous systems lose the rest to 32-byte accesses of 32
// different lines.
#pragma once
#include "trid_device.cuh"

namespace trid {

constexpr int TW_R = 4;      // rows loaded ahead on the way to the middle
constexpr int TW_RB = 8;     // and on the way back
constexpr int TW_SYS = 16;   // systems per warp

// Four consecutive doubles (32-byte aligned) in one access.
__device__ __forceinline__ void ld_f64x4(const double *p, double (&v)[4]) {
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_f64x4(double *p, const double (&v)[4]) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};"
                 :: "l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
}

// Rows of the upper half: the middle, or with vector access (systems
// contiguous, n a multiple of 4) the next multiple of 4, so that both halves
// are whole vectors.  Never less than the lower half.
__host__ __device__ inline int twist_rows(int n, bool vec) {
    const int h = (n + 1) / 2;
    return vec ? (h + 3) / 4 * 4 : h;
}
__host__ inline size_t twist_smem(int n, bool vec, bool acc, int warps) {
    return size_t(warps) * twist_rows(n, vec) * 32 * sizeof(double) * (acc ? 2 : 1);
}

template <bool ACC, bool VEC, int WARPS>
__global__ void __launch_bounds__(32 * WARPS)
k_twist(const double *__restrict__ a, const double *__restrict__ b, const double *__restrict__ c,
        const double *d, double *out, Lines L) {
    constexpr int R = TW_R, RB = TW_RB;
    extern __shared__ __align__(16) double sm_tw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = int(L.n);
    const int h = twist_rows(n, VEC);
    const bool low = lane >= TW_SYS;
    const int64_t s = (int64_t(blockIdx.x) * WARPS + warp) * TW_SYS + (lane & (TW_SYS - 1));
    int64_t base = s < L.nsys ? L.base(s) : 0;
    const bool active =
        s < L.nsys && TRID_BOUNDS(base + int64_t(n - 1) * L.stride < L.nsys * L.n);
    const int cnt = !active ? 0 : low ? n - h : h;
    // (n - 1) * stride < 2^31 (host)
    const int step = low ? -int(L.stride) : int(L.stride);
    if (low) base += int64_t(n - 1) * L.stride;
    const double *lo = (low ? c : a) + base;   // towards the row before (in walking order)
    const double *hi = (low ? a : c) + base;   // towards the row after
    const double *bb = b + base, *dd = d + base;
    double *xx = out + base;
    double *sc = sm_tw + size_t(warp) * h * 32 * (ACC ? 2 : 1) + lane;
    double *sd = sc + size_t(h) * 32;          // ACC only

    double A[R], B[R], C[R], D[R];
    auto load = [&](int k0) {
        if constexpr (VEC) {
            if (k0 < cnt) {
                const int off = low ? -(k0 + 3) : k0;
                double va[4], vb[4], vc[4], vd[4];
                ld_f64x4(lo + off, va);
                ld_f64x4(bb + off, vb);
                ld_f64x4(hi + off, vc);
                ld_f64x4(dd + off, vd);
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    A[j] = low ? va[3 - j] : va[j];
                    B[j] = low ? vb[3 - j] : vb[j];
                    C[j] = low ? vc[3 - j] : vc[j];
                    D[j] = low ? vd[3 - j] : vd[j];
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (k0 + j < cnt) {
                    const int off = (k0 + j) * step;
                    A[j] = lo[off];
                    B[j] = bb[off];
                    C[j] = hi[off];
                    D[j] = dd[off];
                }
        }
    };

    // to the middle: x_k + cp x_{k+1} = dp
    double cp = 0.0, dp = 0.0;
    load(0);
    A[0] = 0.0;   // not part of the system
    for (int k0 = 0; k0 < h; k0 += R) {
        double pa[R], pb[R], pc[R], pd[R];
#pragma unroll
        for (int j = 0; j < R; ++j) { pa[j] = A[j]; pb[j] = B[j]; pc[j] = C[j]; pd[j] = D[j]; }
        if (k0 + R < h) load(k0 + R);
        double dv[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int k = k0 + j;
            if (k < cnt) {
                const double r = rcp(fma(-pa[j], cp, pb[j]));
                cp = pc[j] * r;
                dp = fma(-pa[j], dp, pd[j]) * r;
                sc[k * 32] = cp;
                dv[j] = dp;
                if constexpr (ACC) sd[k * 32] = dp;
                else if constexpr (!VEC) xx[k * step] = dp;
            }
        }
        if constexpr (VEC && !ACC) {
            if (k0 < cnt) {
                double v[4];
#pragma unroll
                for (int j = 0; j < R; ++j) v[j] = low ? dv[3 - j] : dv[j];
                st_f64x4(xx + (low ? -(k0 + 3) : k0), v);
            }
        }
    }
    if (cnt == n) cp = 0.0;   // no lower half: c of the last row is not part of the system
    // the two middle rows: x + cp y = dp, y + oc x = od
    constexpr unsigned FULL = 0xffffffffu;
    const double oc = __shfl_xor_sync(FULL, cp, TW_SYS);
    const double od = __shfl_xor_sync(FULL, dp, TW_SYS);
    double x = (dp - cp * od) * rcp(1.0 - cp * oc);

    // and back: row cnt - 1 is x, the others follow
    double V[RB];
    auto load_back = [&](int k0) {
        if constexpr (VEC) {
#pragma unroll
            for (int q = 0; q < RB; q += 4)
                if (k0 + q < cnt) {
                    double v[4];
                    ld_f64x4(xx + (low ? -(k0 + q + 3) : k0 + q), v);
#pragma unroll
                    for (int j = 0; j < 4; ++j) V[q + j] = low ? v[3 - j] : v[j];
                }
        } else {
#pragma unroll
            for (int j = 0; j < RB; ++j)
                if (k0 + j < cnt) V[j] = xx[(k0 + j) * step];
        }
    };
    const int klast = (h - 1) / RB * RB;
    load_back(klast);
    for (int k0 = klast; k0 >= 0; k0 -= RB) {
        double w[RB], cs[RB], ds[RB];
#pragma unroll
        for (int j = 0; j < RB; ++j) {
            w[j] = V[j];
            if (k0 + j < cnt) {
                cs[j] = sc[(k0 + j) * 32];
                if constexpr (ACC) ds[j] = sd[(k0 + j) * 32];
            }
        }
        if (k0 > 0) load_back(k0 - RB);
#pragma unroll
        for (int j = RB - 1; j >= 0; --j) {
            const int k = k0 + j;
            if (k < cnt) {
                if (k < cnt - 1) x = fma(-cs[j], x, ACC ? ds[j] : w[j]);
                w[j] = ACC ? w[j] + x : x;
                if constexpr (!VEC) xx[k * step] = w[j];
            }
        }
        if constexpr (VEC) {
#pragma unroll
            for (int q = 0; q < RB; q += 4)
                if (k0 + q < cnt) {
                    double v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] = low ? w[q + 3 - j] : w[q + j];
                    st_f64x4(xx + (low ? -(k0 + q + 3) : k0 + q), v);
                }
        }
    }
}

}  // namespace trid
