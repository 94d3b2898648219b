// trid_adi_planes_run.cuh -- launch of the whole-plane 3D ADI step
// (trid_adi_planes.cuh) for one element type; each type is instantiated in a
// translation unit of its own.
#pragma once
#include "trid_adi_planes.cuh"
#include "trid_internal.h"

namespace trid {

// A launch that may start while the previous kernel of the stream drains.
template <typename... KA, typename... A>
static bool planes_launch(void (*kern)(KA...), dim3 grid, int threads, size_t smem,
                          cudaStream_t st, bool pdl, A... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    if (e != cudaSuccess) {
        note_cuda_error(e);
        cudaGetLastError();
    }
    return e == cudaSuccess;
}

// Pass A of one step (or, check_only, whether it can be launched).
template <typename T, int HX, int HY>
static bool planes_a(const T *u, T *w, const int64_t *n3, int64_t nb, double lam, cudaStream_t st,
                     bool pdl, bool check_only) {
    const int nx = int(n3[0]), ny = int(n3[1]), nz = int(n3[2]);
    const PlaneLayout l = plane_layout<T>(plane_pitch<T>(HX), (ny + 1) / 2);
    const size_t smem = size_t(planes_total<T>(l)) * sizeof(T);
    const DeviceInfo *di = device_info();
    if (!di || smem > size_t(di->max_smem_optin)) return false;
    auto kern = k_adi_planes<T, HX, HY>;
    const int64_t items = nb * (nz - 2);
    const int warps = plane_pick_warps(items, nx, ny, nx * ny, smem, size_t(di->smem_per_sm),
                                       di->sm_count, plane_sm_warps(HX, HY, int(sizeof(T))),
                                       plane_max_warps(HX, HY));
    if (check_only)
        return items < (int64_t(1) << 31) &&
               kernel_blocks_per_sm(reinterpret_cast<const void *>(kern), 32 * warps, smem) >= 1;
    PlaneTabs<T, HX, HY> t;
    plane_axis<T, HX>(t.fx, t.gx, t.kx, nx, lam, lam);
    plane_axis<T, HY>(t.fy, t.gy, t.ky, ny, lam, 1.0);
    return planes_launch(kern, dim3(unsigned(items)), 32 * warps, smem, st, pdl, u, w, nx, ny, nz,
                         t);
}

template <typename T>
static bool planes_a_xy(const T *u, T *w, const int64_t *n3, int64_t nb, double lam,
                        cudaStream_t st, bool pdl, bool check_only) {
    return plane_dispatch<T>(int(n3[0]), [&](auto sx) {
        return plane_dispatch<T>(int(n3[1]), [&](auto sy) {
            return planes_a<T, decltype(sx)::value, decltype(sy)::value>(u, w, n3, nb, lam, st,
                                                                         pdl, check_only);
        });
    });
}

template <typename T, int HZ>
static bool planes_b_h(const T *w, T *u, const int64_t *n3, int64_t nb, double lam,
                       cudaStream_t st, bool pdl) {
    ZLineTabs<T, HZ> t;
    plane_axis<T, HZ>(t.f, t.g, t.k, int(n3[2]), lam, 1.0);
    const int64_t lines = 16 * ZL_WARPS;
    const dim3 grid(unsigned((n3[0] * n3[1] + lines - 1) / lines), unsigned(nb));
    return planes_launch(k_adi_zlines<T, HZ>, grid, 32 * ZL_WARPS, 0, st, pdl, w, u, int(n3[0]),
                         int(n3[1]), int(n3[2]), t);
}

// Longest z line of pass B: two halves in registers.
template <typename T>
constexpr int planes_max_nz() { return sizeof(T) == 4 ? 256 : 128; }

template <typename T>
static bool planes_b(const T *w, T *u, const int64_t *n3, int64_t nb, double lam, cudaStream_t st,
                     bool pdl) {
    const int nz = int(n3[2]);
    if constexpr (sizeof(T) == 4) {
        if (nz > 224) return planes_b_h<T, 128>(w, u, n3, nb, lam, st, pdl);
        if (nz > 192) return planes_b_h<T, 112>(w, u, n3, nb, lam, st, pdl);
        if (nz > 160) return planes_b_h<T, 96>(w, u, n3, nb, lam, st, pdl);
    }
    return plane_dispatch<T>(nz, [&](auto sz) {
        return planes_b_h<T, decltype(sz)::value>(w, u, n3, nb, lam, st, pdl);
    });
}

template <typename T>
static trid_status planes_run(T *u, T *w, const int64_t *n3, int64_t nb, double lam, int nsteps,
                              cudaStream_t st, bool &taken) {
    taken = false;
    if (n3[2] > planes_max_nz<T>() || nb > 65535) return TRID_OK;
    const bool pdl = pdl_launch_allowed(st);
    if (!planes_a_xy<T>(u, w, n3, nb, lam, st, pdl, true)) return TRID_OK;
    taken = true;
    for (int s = 0; s < nsteps; ++s)
        if (!planes_a_xy<T>(u, w, n3, nb, lam, st, pdl, false) ||
            !planes_b<T>(w, u, n3, nb, lam, st, pdl))
            return TRID_ERR_CUDA;
    return TRID_OK;
}

}  // namespace trid
