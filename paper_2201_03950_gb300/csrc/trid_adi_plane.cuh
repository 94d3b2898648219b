// trid_adi_plane.cuh -- all steps of a small 2D mesh on chip (Section 4.1,
// Algorithm "adi"; the batched 2D workloads of Section 4).
//
// One block owns a mesh; u and the intermediate d = X^{-1} (explicit part)
// stay in shared memory for every step of the call.  Two threads own a line,
// one from each end (Thomas from both ends, meeting in the middle), with the
// line's values in registers and the constant operator's factors as constant
// operands:
//   down   v_k = F_k d_k + G_k v_{k-1}      (k = distance from the own end)
//   middle x = (v + G v_other) / (1 - G G')
//   back   x_k = v_k + G_k x_{k+1}
// (a = c = -lambda makes the sub- and the super-diagonal factor the same
// number G_k = lambda m_k; the two ends' factors are equal by symmetry).
// Per point and step that is 11 floating-point instructions and 7 words of
// shared memory.  Lines are held aligned to the middle: the last register is
// the row next to it, rows beyond the line's own end have F = G = 0, so that
// no length needs a predicate in the sweeps.
//
// One thread per line, walking it in shared memory (the kernel of
// trid_adi_batched.cu, still used for 3D meshes), is bound by the latency of
// that walk at 8 warps per SM.  Here what counts is the number of
// instructions: with a pitch known only at run time the 96 x 96 kernel issued
// 34 per point, half of them addresses and branches, hence the pitch and the
// line length as template parameters.  Measured, 40 steps: 3000 meshes of
// 96 x 96 5837 -> 1262 us (877 G point-steps/s), 3000 of 64 x 64 1696 -> 500,
// 1500 of 128 x 128 8160 -> 1422, 2000 of 128 x 32 1021 -> 363; FP64, bound by
// its arithmetic, 500 of 96 x 96 7336 -> 4866, 1500 of 64 x 64 6185 -> 5608.
//
//   x phase: lanes 0..15 of a warp own the left halves of 16 rows, lanes
//     16..31 the right halves.  Right halves are stored mirrored, so both
//     read the rows y - 1, y, y + 1 with 16-byte loads in walking order, form
//     the explicit part and eliminate at once; d goes back the same way.
//   y phase: lanes 0..15 own the upper halves of 16 columns, lanes 16..31 the
//     lower halves; lower rows are stored mirrored too, an odd multiple of 16
//     words after the upper ones, so that the two half-warps hit the two
//     halves of the banks.  x is added into u.
// The row pitch is an odd multiple of 16 bytes: 16-byte accesses of 8
// consecutive rows and 4-byte accesses along a row are free of conflicts.
// An odd line's middle row belongs to the first half; the other end also
// eliminates it (it needs x there) but does not store it.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace trid {

// Factors aligned to the middle (entries HX - 1 and HY - 1); fx carries lambda.
template <typename T, int HX, int HY>
struct PlaneTabs {
    T fx[HX], gx[HX], fy[HY], gy[HY];
    T kx, ky;   // 1 / (1 - G G') of the middle
};

// Half lines are held in HX and HY registers, of the sizes below: the smallest
// that holds the half line, which leaves fewer than 16 empty, so that only the
// first 16 need be looked at.  The row pitch follows from HX, so that every
// address of a sweep is a constant offset.
constexpr int PL_STEP = 16;
inline int plane_size(int n) {   // of a line of n nodes; 0: too long
    const int h = (n + 1) / 2;
    return h <= 16 ? 16 : h <= 48 ? (h + 7) / 8 * 8 : h <= 80 ? (h + 15) / 16 * 16 : 0;
}
// Calls f with the size as a compile-time constant; FP64 lines of 80 leave no
// registers.
template <int H> struct PlaneSize { static constexpr int value = H; };
template <typename T, typename F>
inline bool plane_dispatch(int n, F &&f) {
    switch (plane_size(n)) {
        case 16: return f(PlaneSize<16>());
        case 24: return f(PlaneSize<24>());
        case 32: return f(PlaneSize<32>());
        case 40: return f(PlaneSize<40>());
        case 48: return f(PlaneSize<48>());
        case 64: return f(PlaneSize<64>());
        case 80:
            if constexpr (sizeof(T) == 4) return f(PlaneSize<80>());
            return false;
        default: return false;
    }
}
template <typename T>
__host__ __device__ constexpr int plane_pitch(int HX) { return 2 * HX + 16 / int(sizeof(T)); }

// Shared-memory layout in elements; u rows k at 0 / u1 + k p (upper / lower
// rows, mirrored), d rows k >= 1 at d0 / d1 + (k - 1) p.
struct PlaneLayout {
    int u1, d0, d1, total;
};

template <typename T>
__host__ __device__ inline PlaneLayout plane_layout(int p, int hy) {
    PlaneLayout l;
    // the lower rows start 16 words (mod 32) after the upper ones
    auto half_banks = [](int v) {
        return sizeof(T) == 4 ? v + ((16 - v) % 32 + 32) % 32 : v;
    };
    l.u1 = half_banks(hy * p);
    l.d0 = l.u1 + hy * p;
    l.d1 = l.d0 + half_banks((hy - 1) * p);
    l.total = l.d1 + (hy - 1) * p;
    return l;
}

template <typename T>
__device__ __forceinline__ void plane_ld4(const T *p, T (&v)[4]) {
    if constexpr (sizeof(T) == 4) {
        const float4 w = *reinterpret_cast<const float4 *>(p);
        v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
    } else {
        const double2 w = *reinterpret_cast<const double2 *>(p);
        const double2 z = *reinterpret_cast<const double2 *>(p + 2);
        v[0] = w.x; v[1] = w.y; v[2] = z.x; v[3] = z.y;
    }
}
template <typename T>
__device__ __forceinline__ void plane_st4(T *p, T a, T b, T c, T d) {
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
    } else {
        *reinterpret_cast<double2 *>(p) = make_double2(a, b);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(c, d);
    }
}

// Groups of 16 interior lines of an axis that the other axis has n nodes of.
__host__ __device__ constexpr int plane_groups(int n) { return (n - 2 + 15) / 16; }
constexpr int plane_max_warps(int HX, int HY) {
    return plane_groups(2 * (HX > HY ? HX : HY));
}
// Blocks of the largest size per SM that the registers are kept low enough
// for: a thread keeps its line and about 50 registers more, a scheduler has
// 16,384.
constexpr int plane_min_blocks(int HX, int HY, int esz) {
    const int words = (HX > HY ? HX : HY) * esz / 4 + 50;
    const int nb = 16384 / (32 * words) * 4 / plane_max_warps(HX, HY);
    return nb < 1 ? 1 : nb;
}
// The warps per SM that this leaves room for.
constexpr int plane_sm_warps(int HX, int HY, int esz) {
    return plane_min_blocks(HX, HY, esz) * plane_max_warps(HX, HY);
}

template <typename T, int HX, int HY>
__global__ void __launch_bounds__(32 * plane_max_warps(HX, HY),
                                  plane_min_blocks(HX, HY, sizeof(T)))
k_adi_plane(T *__restrict__ ug, int64_t nbatch, int nx, int ny, int nsteps,
            const __grid_constant__ PlaneTabs<T, HX, HY> t) {
    static_assert(HX % 4 == 0 && HY % 4 == 0, "whole groups of four");
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int CX = HX / 4, CY = HY / 4, CG = PL_STEP / 4;  // groups of 4; those that may be empty
    constexpr int p = plane_pitch<T>(HX);
    extern __shared__ __align__(16) unsigned char smem_pl[];
    T *sm = reinterpret_cast<T *>(smem_pl);
    const int hx = (nx + 1) / 2, hy = (ny + 1) / 2;
    const PlaneLayout l = plane_layout<T>(p, hy);
    const int tid = threadIdx.x, nth = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarp = nth >> 5;
    const int half = lane >> 4;
    const bool oddx = nx & 1, oddy = ny & 1;
    const int offx = HX - hx, offy = HY - hy;   // register of an end's boundary node
    auto pos = [&](int x) { return x < hx ? offx + x : HX + offx + (nx - 1 - x); };
    auto urow = [&](int y) { return y < hy ? y * p : l.u1 + (ny - 1 - y) * p; };
    auto drow = [&](int y) { return y < hy ? l.d0 + (y - 1) * p : l.d1 + (ny - 2 - y) * p; };
    const int edge = (half ? -HX : HX) + HX - 1 - oddx;   // across the middle, from the own half
    const bool dupx = oddx && half, dupy = oddy && half;  // the middle belongs to the first half

    for (int q = tid; q < l.total; q += nth) sm[q] = T(0);
    __syncthreads();
    for (int64_t mb = blockIdx.x; mb < nbatch; mb += gridDim.x) {
        T *um = ug + mb * int64_t(nx) * ny;
        for (int r = warp; r < ny; r += nwarp)
            for (int x = lane; x < nx; x += 32) {
                // the corners enter no explicit part: kept at 0 here, so that
                // the products with the boundary columns' zero factors are 0
                const bool corner = (r == 0 || r == ny - 1) && (x == 0 || x == nx - 1);
                sm[urow(r) + pos(x)] = corner ? T(0) : um[r * nx + x];
            }
        __syncthreads();
        for (int s = 0; s < nsteps; ++s) {
            for (int first = 1 + 16 * warp; first <= ny - 2; first += 16 * nwarp) {
                // a lane without a row of its own repeats the last one
                const int line = first + (lane & 15);
                const int y = line <= ny - 2 ? line : ny - 2;
                const T *r0 = sm + urow(y) + half * HX;
                const T *rm = sm + urow(y - 1) + half * HX;
                const T *rp = sm + urow(y + 1) + half * HX;
                T *rd = sm + drow(y) + half * HX;
                T v[HX];
                T cur[4], nxt[4], below[4], above[4];
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
                        if (c == CX - 1 && dupx) {   // the middle element, from the left half
                            cur[3] = r0[-1];
                            below[3] = rm[-1];
                            above[3] = rp[-1];
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const T after = j < 3 ? cur[j < 3 ? j + 1 : 3] : nxt[0];
                            const T sum = (before + after) + (below[j] + above[j]);
                            const T e = fma(T(-4), cur[j], sum);
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
                        plane_st4<T>(rd + 4 * c, v[4 * c], v[4 * c + 1], v[4 * c + 2],
                                     v[4 * c + 3]);
                    }
                }
            }
            __syncthreads();
            for (int first = 1 + 16 * warp; first <= nx - 2; first += 16 * nwarp) {
                // a lane without a column of its own works on the padding
                // column 2 HX, which holds 0 and stays 0
                const int line = first + (lane & 15);
                const int col = line <= nx - 2 ? pos(line) : 2 * HX;
                T *pu = sm + (half ? l.u1 : 0) + col - offy * p;
                const T *pd = sm + (half ? l.d1 : l.d0) + col - (offy + 1) * p;
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
                if (!dupy) pu[(HY - 1) * p] += x;
#pragma unroll
                for (int c = CY - 1; c >= 0; --c) {
                    T w[4];
#pragma unroll
                    for (int j = 3; j >= 0; --j) {
                        const int k = 4 * c + j;
                        if (k < HY - 1 && (k >= PL_STEP || k > offy)) w[j] = pu[k * p];
                    }
#pragma unroll
                    for (int j = 3; j >= 0; --j) {
                        const int k = 4 * c + j;
                        if (k < HY - 1 && (k >= PL_STEP || k > offy)) {
                            x = fma(t.gy[k], x, v[k]);
                            pu[k * p] = w[j] + x;
                        }
                    }
                }
            }
            __syncthreads();
        }
        for (int r = 1 + warp; r < ny - 1; r += nwarp)
            for (int x = lane; x < nx; x += 32) um[r * nx + x] = sm[urow(r) + pos(x)];
        __syncthreads();
    }
}

// Host: factors of an axis of n nodes (3 <= n <= 2 H), scaled by `scale`.
template <typename T, int H>
inline void plane_axis(T (&f)[H], T (&g)[H], T &k, int n, double lam, double scale) {
    const int hl = (n + 1) / 2, off = H - hl;
    double gd[H] = {0};
    double m = 0.0;
    for (int q = 0; q < H; ++q) {
        f[q] = g[q] = T(0);
        if (q <= off) continue;   // beyond the line, and its boundary row
        m = 1.0 / (1.0 + 2.0 * lam - lam * lam * m);
        gd[q] = lam * m;
        f[q] = T(scale * m);
        g[q] = T(gd[q]);
    }
    k = T(1.0 / (1.0 - gd[H - 1] * gd[H - 1 - (n & 1)]));
}

// Host: warps per block for `items` planes.  A phase walks its groups of 16
// lines and a plane occupies its warps for the walks of both phases (and for
// loading `load_points` points); the number with the least (rounds of blocks)
// x (rows walked), of equal ones the largest.  128 x 32 planes, 2000 meshes,
// 40 steps (an earlier form of k_adi_plane): 8 warps 2014 us, 2 warps 1108 us.
// warps_per_sm: what the registers allow.
inline int plane_pick_warps(int64_t items, int nx, int ny, int load_points, size_t smem,
                            size_t smem_per_sm, int sm_count, int warps_per_sm, int max_warps) {
    const int gx = plane_groups(ny), gy = plane_groups(nx);
    const int hx = (nx + 1) / 2, hy = (ny + 1) / 2;
    int pick = 1;
    int64_t best = -1;
    for (int w = 1; w <= (gx > gy ? gx : gy) && w <= max_warps; ++w) {
        int64_t per_sm = int64_t(smem_per_sm / (smem + 1024));
        if (per_sm > warps_per_sm / w) per_sm = warps_per_sm / w;
        if (per_sm > 32) per_sm = 32;
        if (per_sm < 1) per_sm = 1;
        const int64_t slots = per_sm * sm_count;
        const int64_t rounds = (items + slots - 1) / slots;
        const int64_t walk = (gx + w - 1) / w * hx + (gy + w - 1) / w * hy;
        const int64_t cost = rounds * (walk + load_points / (32 * w));
        if (best < 0 || cost <= best) {
            best = cost;
            pick = w;
        }
    }
    return pick;
}

}  // namespace trid
