// The batched warp sweep with FP32 population storage, and the dispatch on the storage.
#include "lbm_sweep_batch.cuh"

namespace lbm {

int sweep_batch_slots(const DevParams &mode, int storage, int device) {
  return storage == STORAGE_BF16  ? sweep_batch_bf16_slots(mode, device)
         : storage == STORAGE_F16 ? sweep_batch_f16_slots(mode, device)
                                  : sweep_batch_slots_t<StoreF32>(mode, device);
}

cudaError_t launch_sweep_batch(int storage, const SweepBatchItem *items, int n,
                               const BatchChannel *ch, const StepScalars *sc, cudaStream_t s) {
  switch (storage) {
    case STORAGE_BF16: return sweep_batch_bf16_launch(items, n, ch, sc, s);
    case STORAGE_F16: return sweep_batch_f16_launch(items, n, ch, sc, s);
    default: return sweep_batch_launch_t<StoreF32>(items, n, ch, sc, s);
  }
}

int sweep_batch_strips(const DevParams &p) { return sweep_strips(p.nx, p.thermal != 0); }
long long sweep_batch_ctas(const DevParams &p, int chunks) {
  return sweep_ctas(sweep_batch_strips(p), chunks);
}
int sweep_batch_width(bool thermal) { return sweep_width(thermal); }
int sweep_batch_fill(bool thermal) { return 2 * sweep_rows(thermal); }
int sweep_batch_warps() { return SW; }

}  // namespace lbm
