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
  // The shortest launch.  A warp with H rows sweeps H of them in full and the halo's row steps
  // (10; 2 without the energy equation) for about four fifths, since the pipeline fills there,
  // and a row step takes longer the more CTAs share the SM: with one, two and three of them
  // 0.71, 0.86 and 1 of the full SM's, with 16-bit storage (more instructions a row step) 0.79,
  // 0.89 and 1.  Several waves take a full SM's time each.  H counts half as the tallest chunk,
  // half as the mean one: the chunks of a row more are few where the division leaves little.
  // GB300, FP32, us per update at one, two and three CTAs per SM: 1000 x 300 19.7, 16.5, 18.7;
  // 520 x 510 20.5, 17.4, 18.7; 2048 x 256 28.4, 21.7, 21.7; 1237 x 531 32.8, 24.2, 23.2;
  // 2048 x 512 46.6, 32.5, 30.7; 1300 x 900 57.2, 39.7, 36.6, at two waves 49; FP16 storage
  // 1053 x 283 -, 20.1, 20.5; 1693 x 235 -, 23.2, 21.9; 1237 x 531 41.8, 29.2, 27.1; without the
  // energy equation 1000 x 300 9.6, 7.3, 7.1; 1237 x 531 17.3, 11.6, 9.9.  On 60 sizes of 0.26 to
  // 0.7 M nodes the choice is 0.6 % behind the fastest of five (1.5 % with the tallest chunk
  // alone, 2.8 % with the fewest row steps whatever the CTAs per SM).
  const long long slots = (long long)sms * occ;
  const double fill = 0.8 * 2 * sweep_rows(th), alone = storage == STORAGE_F32 ? 0.57 : 0.68;
  double best = -1.0;
  for (int c = 1; c <= p.ny && sweep_ctas(tl.strips, c - 1) <= 3 * slots; c++) {
    const long long ctas = sweep_ctas(tl.strips, c), waves = (ctas + slots - 1) / slots;
    const long long per_sm = (ctas + sms - 1) / sms;
    const double step = waves > 1 ? (double)waves : alone + (1.0 - alone) * (double)per_sm / occ;
    const double rows = 0.5 * ((p.ny + c - 1) / c + (double)p.ny / c);
    const double cost = step * (rows + fill);
    if (best < 0.0 || cost < best) {
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
