// The batched warp sweep with BF16 population storage.
#include "lbm_sweep_batch.cuh"

namespace lbm {

int sweep_batch_bf16_slots(const DevParams &mode, int device) {
  return sweep_batch_slots_t<StoreBF16>(mode, device);
}

cudaError_t sweep_batch_bf16_launch(const SweepBatchItem *items, int n, const BatchChannel *ch,
                      const StepScalars *sc, cudaStream_t s) {
  return sweep_batch_launch_t<StoreBF16>(items, n, ch, sc, s);
}

}  // namespace lbm
