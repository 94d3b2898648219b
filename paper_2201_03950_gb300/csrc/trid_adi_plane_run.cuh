// trid_adi_plane_run.cuh -- launch of the on-chip steps of small 2D meshes
// (trid_adi_plane.cuh) for one element type; each type is instantiated in a
// translation unit of its own.
#pragma once
#include "trid_adi_plane.cuh"
#include "trid_internal.h"

namespace trid {

template <typename T, int HX, int HY>
static bool plane_run_h(T *u, int64_t nbatch, int nx, int ny, double lam, int nsteps,
                        cudaStream_t st, trid_status &status) {
    const size_t smem =
        size_t(plane_layout<T>(plane_pitch<T>(HX), (ny + 1) / 2).total) * sizeof(T);
    const DeviceInfo *di = device_info();
    auto kern = k_adi_plane<T, HX, HY>;
    if (!di || smem > size_t(di->max_smem_optin)) return false;
    const int warps = plane_pick_warps(nbatch, nx, ny, 0, smem, size_t(di->smem_per_sm),
                                       di->sm_count, plane_sm_warps(HX, HY, int(sizeof(T))),
                                       plane_max_warps(HX, HY));
    const int per_sm =
        kernel_blocks_per_sm(reinterpret_cast<const void *>(kern), 32 * warps, smem);
    if (per_sm < 1) return false;
    const int64_t slots = int64_t(di->sm_count) * per_sm;
    const int64_t grid = nbatch < slots ? nbatch : slots;
    PlaneTabs<T, HX, HY> t;
    plane_axis<T, HX>(t.fx, t.gx, t.kx, nx, lam, lam);
    plane_axis<T, HY>(t.fy, t.gy, t.ky, ny, lam, 1.0);
    kern<<<dim3(unsigned(grid)), 32 * warps, smem, st>>>(u, nbatch, nx, ny, nsteps, t);
    status = launch_ok() ? TRID_OK : TRID_ERR_CUDA;
    return true;
}

// FP64 meshes that k_adi_fused steps faster.  Both kernels are bound by their FP64
// instructions: this one issues HX (HY) rows for every group of 16 lines, used or
// not, k_adi_fused one per line's row for every 32 lines (the explicit part along
// x among them).  It keeps the meshes whose padding costs more than two threads
// per line gain: with few meshes (latency) or one group of lines a ratio of issued
// rows below 0.87, else, once every SM has six meshes, below 1.55.  10 steps,
// this kernel against k_adi_fused: 3000 meshes of 5 x 5 179 against 140 us, of 40 x
// 3 620 / 349, of 20 x 20 599 / 477; 100 of 20 x 20 65 / 99, 3000 of 18 x 18 289 /
// 463.  (Over 36 square and 21 other extents with 1 to 20000 meshes the choice is
// 0.6% slower than the better one on the mean.)  k_adi_fused starts more slowly, so
// from 8 steps on (1000 of 20 x 20: 1 step 1.36 times as slow, 4 0.95, 8 0.87; 6 x
// 6: 2.2, 1.33, 1.04).
inline bool plane_padded64(int nx, int ny, int64_t nbatch, int nsteps, int sm_count) {
    if (nsteps < 8) return false;
    const int gx = plane_groups(ny), gy = plane_groups(nx);
    const int here = gx * plane_size(nx) + gy * plane_size(ny);
    const int fused = (ny + 31) / 32 * nx + 3 * ((nx + 31) / 32) * ny;
    const bool many = nbatch >= 6 * int64_t(sm_count) && gx * gy > 1;
    return 100 * fused < (many ? 155 : 87) * here;
}

template <typename T>
static trid_status plane_run(T *u, int64_t nbatch, int nx, int ny, double lam, int nsteps,
                             cudaStream_t st, bool &taken) {
    trid_status status = TRID_OK;
    const DeviceInfo *di = device_info();
    taken = false;
    if (!di || (sizeof(T) == 8 && plane_padded64(nx, ny, nbatch, nsteps, di->sm_count))) return status;
    taken = plane_dispatch<T>(nx, [&](auto sx) {
        return plane_dispatch<T>(ny, [&](auto sy) {
            return plane_run_h<T, decltype(sx)::value, decltype(sy)::value>(
                u, nbatch, nx, ny, lam, nsteps, st, status);
        });
    });
    return status;
}

}  // namespace trid
