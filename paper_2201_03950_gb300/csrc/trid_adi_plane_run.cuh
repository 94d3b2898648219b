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

template <typename T>
static trid_status plane_run(T *u, int64_t nbatch, int nx, int ny, double lam, int nsteps,
                             cudaStream_t st, bool &taken) {
    trid_status status = TRID_OK;
    taken = plane_dispatch<T>(nx, [&](auto sx) {
        return plane_dispatch<T>(ny, [&](auto sy) {
            return plane_run_h<T, decltype(sx)::value, decltype(sy)::value>(
                u, nbatch, nx, ny, lam, nsteps, st, status);
        });
    });
    return status;
}

}  // namespace trid
