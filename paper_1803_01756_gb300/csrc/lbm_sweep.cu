// The warp sweep's FP32 kernel, the tiling of a lattice and the dispatch on the storage.
#include "lbm_sweep_launch.cuh"

namespace lbm {

SweepTiling sweep_tiling(const DevParams &p, int storage, int device) {
  SweepTiling tl{0, 0, 0, 0};
  int sms = 0, occ = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return tl;
  const cudaError_t e = storage == STORAGE_BF16  ? sweep_bf16_occupancy(p, &occ)
                        : storage == STORAGE_F16 ? sweep_f16_occupancy(p, &occ)
                                                 : sweep_occupancy_t<StoreF32>(p, &occ);
  if (e != cudaSuccess || occ < 1) return tl;
  const bool th = p.thermal != 0;
  tl.strips = sweep_strips(p.nx, th);
  tl.width = sweep_width(th);
  // The fewest row steps: a wave of resident CTAs with chunks of H rows takes H + 10 of them
  // (H + 2 without the energy equation).  That is one wave with the shortest chunks, unless
  // the strips alone nearly fill it: beside a full SM the fewer, taller chunks of a partly filled one gain less
  // from the shorter row step than they lose (GB300, FP32, us per update by row chunks:
  // 4096 x 512 47.9 at 24, 69 at 14; 2048 x 512 30.5 at 45, 37.2 at 32, 46.3 at 23;
  // 1237 x 531 23.3 at 76, 25.0 at 48, 27.9 at 38; 777 x 333 17.4 at 114 and at 66).
  const long long slots = (long long)sms * occ;
  const int fill = 2 * sweep_rows(th);
  long long best = -1;
  for (int c = 1; c <= p.ny && sweep_ctas(tl.strips, c - 1) <= 3 * slots; c++) {
    const long long waves = (sweep_ctas(tl.strips, c) + slots - 1) / slots;
    const long long cost = waves * ((p.ny + c - 1) / c + fill);
    if (best < 0 || cost < best) {
      best = cost;
      tl.chunks = c;
    }
  }
  // Programmatic dependent launch when the grid fills at least 90 % of the wave, as for the
  // CTA sweep: below that the waiting CTAs of the next update take issue slots (2048 x 512 at
  // 23 chunks: 46.3 against 39.4 us per update; at 45 chunks 30.5 either way).
  const long long ctas = sweep_ctas(tl.strips, tl.chunks);
  tl.pdl = ctas * 10 >= slots * 9 && ctas <= slots ? 1 : 0;
  return tl;
}

cudaError_t launch_sweep(const DevParams &p, int storage, const void *gs, void *gout,
                         const float *Tin, float *Tout, unsigned *status, const StepScalars *sc,
                         const StepScalars &val, const SweepTiling &tl, cudaStream_t s) {
  switch (storage) {
    case STORAGE_BF16:
      return sweep_bf16_launch(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
    case STORAGE_F16:
      return sweep_f16_launch(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
    default:
      return sweep_launch_t<StoreF32>(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
  }
}

}  // namespace lbm
