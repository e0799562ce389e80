// The warp sweep's kernel with BF16 population storage.
#include "lbm_sweep_launch.cuh"

namespace lbm {

cudaError_t sweep_bf16_occupancy(const DevParams &p, int *occ) {
  return sweep_occupancy_t<StoreBF16>(p, occ);
}

cudaError_t sweep_bf16_launch(const DevParams &p, const void *gs, void *gout, const float *Tin,
                             float *Tout, unsigned *status, const StepScalars *sc,
                             const StepScalars &val, const SweepTiling &tl, cudaStream_t s) {
  return sweep_launch_t<StoreBF16>(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
}

}  // namespace lbm
