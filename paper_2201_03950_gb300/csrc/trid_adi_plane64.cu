// trid_adi_plane64.cu -- all steps of small 2D meshes on chip
// (trid_adi_plane.cuh) in FP64.
#include "trid_adi_plane_run.cuh"

namespace trid {
trid_status adi_plane_run(double *u, int64_t nbatch, int nx, int ny, double lam, int nsteps,
                          cudaStream_t st, bool &taken) {
    return plane_run<double>(u, nbatch, nx, ny, lam, nsteps, st, taken);
}
}  // namespace trid
