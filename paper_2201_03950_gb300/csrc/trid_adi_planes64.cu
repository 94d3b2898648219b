// trid_adi_planes64.cu -- the whole-plane 3D ADI step (trid_adi_planes.cuh) in
// FP64.
#include "trid_adi_planes_run.cuh"

namespace trid {
trid_status adi_planes_run(double *u, double *w, const int64_t *n3, int64_t nb, double lam,
                           int nsteps, cudaStream_t st, bool &taken) {
    return planes_run<double>(u, w, n3, nb, lam, nsteps, st, taken);
}
}  // namespace trid
