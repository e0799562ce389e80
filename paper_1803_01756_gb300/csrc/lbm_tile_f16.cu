// The tile kernel with FP16 population storage.
#include "lbm_tile_launch.cuh"

namespace lbm {

cudaError_t tile_f16_occupancy(const DevParams &p, int rows, int *occ) {
  return tile_occupancy_t<StoreF16>(p, rows, occ);
}

cudaError_t tile_f16_launch(const DevParams &p, const void *gs, void *gout, const float *Tin,
                            float *Tout, unsigned *status, const StepScalars *sc,
                            const StepScalars &val, const TileTiling &tl, cudaStream_t s) {
  return tile_launch_t<StoreF16>(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
}

}  // namespace lbm
