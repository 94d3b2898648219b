// trid_adi_planes.cuh -- 3D ADI step in two passes over whole planes and whole
// z lines (Section 4.1, Algorithm "adi"), odd and even extents and any lambda:
// x and y up to 160 nodes (FP64 128), the plane three times within a block's
// shared memory (about 128 x 128 in FP32, 90 x 90 in FP64), z up to 256 (FP64 128).  The
// launcher leaves what other schedules step faster (adi3_planes_run).
//
//   pass A (k_adi_planes): one block per interior z plane.  The plane and its
//     two z neighbours are brought to shared memory; the explicit part, the x
//     solve and the y solve run there with two threads per line (see
//     trid_adi_plane.cuh), and w = Y^{-1} X^{-1} d is written.
//   pass B (k_adi_zlines): two threads per z line, its values in registers:
//     u += Z^{-1} w.
// Per point A reads u (its z neighbours from the L2) and writes w, B reads w
// and u and writes u: 5 mesh words, and the intermediate stays in the delta
// form, so a step's rounding is that of the update, not of the field (100 steps
// of 48^3 in FP32: 3.5e-6 -> 6e-8 off the 64-bit result).  Meshes stacked along
// z are independent (each keeps its own boundary planes).
//
// What bounds pass A is the number of instructions and the shared-memory
// accesses of its three phases (48^3 x 72: 30 us, 46% of the issue slots and 45%
// of the shared-memory pipe busy, 21 warps per SM); loading the planes a few rows
// at a time instead of all at once took 56 us (latency of the loads), computing
// every copy's address anew 43, and handling the boundary columns' lanes apart
// from the others 34 (every warp has one).  Measured per step, FP32: 72 meshes of
// 48^3 108.8 -> 35.1 us, 24 of 64^3 at lambda 0.3 65.9 -> 31.4, one of 100^3 23.5
// -> 12.8; FP64 72 of 48^3 805 -> 251, one of 100^3 203 -> 82.
#pragma once
#include "trid_adi_plane.cuh"
#include "trid_tma.cuh"

namespace trid {

// Asynchronous copy of one element to shared memory.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst, const T *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
                 ::"r"(smem_u32(dst)), "l"(src), "n"(int(sizeof(T))) : "memory");
}

// Shared memory of pass A in elements: the plane and its two z neighbours.
template <typename T>
__host__ __device__ inline int planes_total(const PlaneLayout &l) {
    return l.total + (l.total - l.d0);
}

template <typename T, int HX, int HY>
__global__ void __launch_bounds__(32 * plane_max_warps(HX, HY),
                                  plane_min_blocks(HX, HY, sizeof(T)))
k_adi_planes(const T *u, T *w, int nx, int ny, int nz,
             const __grid_constant__ PlaneTabs<T, HX, HY> t) {
    static_assert(HX % 4 == 0 && HY % 4 == 0, "whole groups of four");
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int CX = HX / 4, CG = PL_STEP / 4;
    constexpr int p = plane_pitch<T>(HX);
    extern __shared__ __align__(16) unsigned char smem_pl[];
    T *sm = reinterpret_cast<T *>(smem_pl);
    const int hx = (nx + 1) / 2, hy = (ny + 1) / 2;
    const PlaneLayout l = plane_layout<T>(p, hy);
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    const int half = lane >> 4;
    const bool oddx = nx & 1, oddy = ny & 1;
    const int offx = HX - hx, offy = HY - hy;   // register of an end's boundary node
    auto pos = [&](int x) { return x < hx ? offx + x : HX + offx + (nx - 1 - x); };
    auto urow = [&](int y) { return y < hy ? y * p : l.u1 + (ny - 1 - y) * p; };
    auto drow = [&](int y) { return y < hy ? l.d0 + (y - 1) * p : l.d1 + (ny - 2 - y) * p; };
    const int edge = (half ? -HX : HX) + HX - 1 - oddx;   // across the middle, from the own half
    const bool dupx = oddx && half, dupy = oddy && half;  // the middle belongs to the first half

    const int eoff = l.total - l.d0;                      // from a row of z - 1 to that of z + 1
    const int mesh = int(blockIdx.x) / (nz - 2);
    const int z = 1 + int(blockIdx.x) - mesh * (nz - 2);
    const int plane = nx * ny;
    const size_t base = (size_t(mesh) * nz + z) * size_t(plane);
    // The group of four that the line begins in is read whole: what lies before
    // the boundary node is 0 (its factors are 0 too).  The boundary columns' z
    // neighbours and the plane's corners enter no explicit part: 0 as well.
    for (int r = tid; r < ny; r += blockDim.x) {
        const bool inner = r > 0 && r < ny - 1;
        T *du = sm + urow(r), *dd = sm + drow(r);
        for (int q = offx & ~3; q <= offx; ++q) {
            if (q < offx || !inner) du[q] = du[HX + q] = T(0);
            if (inner) dd[q] = dd[HX + q] = dd[eoff + q] = dd[eoff + HX + q] = T(0);
        }
    }
    pdl_trigger();
    pdl_wait();   // u is written by the previous kernel on the stream
    const T *up = u + base;
    char *wp = reinterpret_cast<char *>(w + base);
    // all three planes by asynchronous copies, every one in flight at once,
    // rows by warp (constant address steps): 32 columns of one half's rows at a
    // time, or where that leaves 16 lanes or more without a column, 16 columns
    // of both halves' rows
    auto fetch = [&](int hh, int x0, int dx) {
        const int rows = hh ? ny - hy : hy, gs = (hh ? -nx : nx) * nwarp;
        for (int x = x0; x < nx; x += dx) {
            const bool inner = x > 0 && x < nx - 1;
            const int px = pos(x);
            const T *q = up + (hh ? (ny - 1 - warp) * nx : warp * nx) + x;
            T *du = sm + (hh ? l.u1 : 0) + px + warp * p;
            T *dd = sm + (hh ? l.d1 : l.d0) + px + (warp - 1) * p;
            int k = warp;
            if (k == 0) {   // the boundary row
                if (inner) cp_async_elem(du, q);
                k += nwarp; q += gs; du += nwarp * p; dd += nwarp * p;
            }
#pragma unroll 4
            for (; k < rows; k += nwarp, q += gs, du += nwarp * p, dd += nwarp * p) {
                cp_async_elem(du, q);
                if (inner) {
                    cp_async_elem(dd, q - plane);
                    cp_async_elem(dd + eoff, q + plane);
                }
            }
        }
    };
    if ((nx + 31) / 32 * 32 - nx < 16) {
        fetch(0, lane, 32);
        fetch(1, lane, 32);
    } else {
        fetch(half, lane & 15, 16);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int first = 1 + 16 * warp; first <= ny - 2; first += 16 * nwarp) {
        // a lane without a row of its own repeats the last one
        const int line = first + (lane & 15);
        const int y = line <= ny - 2 ? line : ny - 2;
        const T *r0 = sm + urow(y) + half * HX;
        const T *rm = sm + urow(y - 1) + half * HX;
        const T *rp = sm + urow(y + 1) + half * HX;
        T *rd = sm + drow(y) + half * HX;   // the plane below, then X^{-1} d
        T v[HX];
        T cur[4], nxt[4], below[4], above[4], zs[4], ze[4];
        T before = T(0), prev = T(0);
        plane_ld4<T>(r0, nxt);
#pragma unroll
        for (int c = 0; c < CX; ++c) {
#pragma unroll
            for (int j = 0; j < 4; ++j) cur[j] = nxt[j];
            if (c < CX - 1) {
                plane_ld4<T>(r0 + 4 * c + 4, nxt);
            } else {
                nxt[0] = r0[edge];
            }
            if (c < CG && 4 * c + 3 < offx) {
#pragma unroll
                for (int j = 0; j < 4; ++j) v[4 * c + j] = T(0);
            } else {
                plane_ld4<T>(rm + 4 * c, below);
                plane_ld4<T>(rp + 4 * c, above);
                plane_ld4<T>(rd + 4 * c, zs);
                plane_ld4<T>(rd + eoff + 4 * c, ze);
                if (c == CX - 1 && dupx) {   // the middle element, from the left half
                    cur[3] = r0[-1];
                    below[3] = rm[-1];
                    above[3] = rp[-1];
                    zs[3] = rd[-1];
                    ze[3] = rd[eoff - 1];
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const T after = j < 3 ? cur[j < 3 ? j + 1 : 3] : nxt[0];
                    const T sum = ((before + after) + (below[j] + above[j])) + (zs[j] + ze[j]);
                    const T e = fma(T(-6), cur[j], sum);
                    prev = fma(t.gx[4 * c + j], prev, t.fx[4 * c + j] * e);
                    v[4 * c + j] = prev;
                    before = cur[j];
                }
            }
        }
        const T other = __shfl_xor_sync(FULL, oddx ? v[HX - 2] : v[HX - 1], 16);
        T x = fma(t.gx[HX - 1], other, v[HX - 1]) * t.kx;
        v[HX - 1] = x;
#pragma unroll
        for (int c = CX - 1; c >= 0; --c) {
            if (c >= CG || 4 * c + 3 >= offx) {
#pragma unroll
                for (int j = 3; j >= 0; --j) {
                    const int k = 4 * c + j;
                    if (k < HX - 1) v[k] = x = fma(t.gx[k], x, v[k]);
                }
                plane_st4<T>(rd + 4 * c, v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
            }
        }
    }
    __syncthreads();
    for (int first = 1 + 16 * warp; first <= nx - 2; first += 16 * nwarp) {
        const int line = first + (lane & 15);
        const bool act = line <= nx - 2;
        const int xc = act ? line : nx - 2;
        const int col = pos(xc);
        const T *pd = sm + (half ? l.d1 : l.d0) + col - (offy + 1) * p;
        // bytes from the plane's first element: 32 bits
        const unsigned step = unsigned(half ? -nx : nx) * unsigned(sizeof(T));
        unsigned o = unsigned(xc + (half ? (ny - 1) * nx : 0)) * unsigned(sizeof(T));
        T v[HY];
#pragma unroll
        for (int k = 0; k < HY - 1; ++k) {
            v[k] = T(0);
            if (k >= PL_STEP || k > offy) v[k] = pd[k * p];
        }
        {   // an odd column's middle row lies with the upper rows
            const T *last = dupy ? sm + l.d0 + col + (hy - 2) * p : pd + (HY - 1) * p;
            v[HY - 1] = *last;
        }
        T prev = T(0);
#pragma unroll
        for (int k = 0; k < HY; ++k) v[k] = prev = fma(t.gy[k], prev, t.fy[k] * v[k]);
        const T other = __shfl_xor_sync(FULL, oddy ? v[HY - 2] : v[HY - 1], 16);
        T x = fma(t.gy[HY - 1], other, v[HY - 1]) * t.ky;
        o += unsigned(hy - 1) * step;
        if (act && !dupy) *reinterpret_cast<T *>(wp + o) = x;
#pragma unroll
        for (int k = HY - 2; k >= 0; --k) {
            o -= step;
            if (k >= PL_STEP || k > offy) {
                x = fma(t.gy[k], x, v[k]);
                if (act) *reinterpret_cast<T *>(wp + o) = x;
            }
        }
    }
}

// Factors of a z line's half, aligned to the middle (see plane_axis).
template <typename T, int HZ>
struct ZLineTabs {
    T f[HZ], g[HZ];
    T k;
};

constexpr int ZL_WARPS = 4;   // 64 z lines per block

template <typename T, int HZ>
__global__ void __launch_bounds__(32 * ZL_WARPS, 16384 / (32 * (HZ * int(sizeof(T)) / 4 + 48)))
k_adi_zlines(const T *w, T *u, int nx, int ny, int nz,
             const __grid_constant__ ZLineTabs<T, HZ> t) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int R = 8;   // rows of u loaded ahead on the way back
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int half = lane >> 4;
    const int plane = nx * ny, hz = (nz + 1) / 2, offz = HZ - hz;
    const bool oddz = nz & 1, dupz = oddz && half;
    const int c = (int(blockIdx.x) * ZL_WARPS + warp) * 16 + (lane & 15);
    const int y = c / nx, x = c - y * nx;
    const bool act = c < plane && x > 0 && x < nx - 1 && y > 0 && y < ny - 1;
    // bytes from the mesh's first element: 32 bits (extents up to 256)
    const unsigned step = unsigned(half ? -plane : plane) * unsigned(sizeof(T));
    const unsigned end = unsigned((act ? c : 0) + (half ? (nz - 1) * plane : 0)) *
                         unsigned(sizeof(T));
    const size_t base = size_t(blockIdx.y) * nz * size_t(plane);
    const char *pw = reinterpret_cast<const char *>(w + base);
    char *pu = reinterpret_cast<char *>(u + base);
    pdl_trigger();
    pdl_wait();   // w is written, and u read, by the previous kernel on the stream
    // register k holds the half line's element k - offz, at `end` + its steps
    const unsigned o0 = end - unsigned(offz) * step;
    T v[HZ];
#pragma unroll
    for (int k = 0; k < HZ; ++k) {
        v[k] = T(0);
        if (act && (k >= PL_STEP || k > offz)) v[k] = *reinterpret_cast<const T *>(pw + (o0 + unsigned(k) * step));
    }
    T ahead[R];
    auto load_u = [&](int k0) {
#pragma unroll
        for (int j = 0; j < R; ++j)
            if (act && (k0 + j >= PL_STEP || k0 + j > offz))
                ahead[j] = *reinterpret_cast<const T *>(pu + (o0 + unsigned(k0 + j) * step));
    };
    load_u(HZ - R);
    T prev = T(0);
#pragma unroll
    for (int k = 0; k < HZ; ++k) v[k] = prev = fma(t.g[k], prev, t.f[k] * v[k]);
    const T other = __shfl_xor_sync(FULL, oddz ? v[HZ - 2] : v[HZ - 1], 16);
    T xv = fma(t.g[HZ - 1], other, v[HZ - 1]) * t.k;
#pragma unroll
    for (int k0 = HZ - R; k0 >= 0; k0 -= R) {
        T uv[R];
#pragma unroll
        for (int j = 0; j < R; ++j) uv[j] = ahead[j];
        if (k0 > 0) load_u(k0 - R);
#pragma unroll
        for (int j = R - 1; j >= 0; --j) {
            const int k = k0 + j;
            if (k < HZ - 1) xv = fma(t.g[k], xv, v[k]);
            if (act && (k >= PL_STEP || k > offz) && (k < HZ - 1 || !dupz))
                *reinterpret_cast<T *>(pu + (o0 + unsigned(k) * step)) = uv[j] + xv;
        }
    }
}

}  // namespace trid
