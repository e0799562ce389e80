// The tile kernel's FP32 instantiation, the tiling of a lattice and the dispatch on the storage.
#include "lbm_tile_launch.cuh"

namespace lbm {

int tile_max_rows(bool thermal) { return TW - 2 * sweep_rows(thermal); }

namespace {

// A CTA's rows in tiles of equal height, at most tile_max_rows
int rows_of(int h, int most) {
  const int tiles = ceil_div(h, most);
  return ceil_div(h, tiles);
}

cudaError_t occupancy(const DevParams &p, int storage, int rows, int *occ) {
  return storage == STORAGE_BF16  ? tile_bf16_occupancy(p, rows, occ)
         : storage == STORAGE_F16 ? tile_f16_occupancy(p, rows, occ)
                                  : tile_occupancy_t<StoreF32>(p, rows, occ);
}

}  // namespace

TileTiling tile_tiling(const DevParams &p, int storage, int device) {
  TileTiling best{0, 0, 0, 0, 0};
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return best;
  const bool th = p.thermal != 0;
  const int strips = sweep_strips(p.nx, th), most = tile_max_rows(th), fill = 2 * sweep_rows(th);
  // The height of a CTA's rows with the shortest launch: waves of CTAs (the registers leave
  // one of 20 warps on an SM, and one of 12), each of tiles one after another, and a tile
  // takes 0.70 us and 0.0875 us a warp (GB300, FP32: 200 x 50 with tiles of 2 rows, 12 warps,
  // 3.54 us per update, of which 1.8 are the launch and the first loads; 1600 x 48 with 10
  // rows, 20 warps, 4.49; 777 x 333 in several waves of tiles of 9 rows 13.9).
  double best_cost = -1.0;
  int occ_of[TW + 1] = {};  // resident CTAs per SM by rows of a tile, 0 until asked for
  for (int h = 1; h <= p.ny; h = h < 64 ? h + 1 : h + 16) {
    const int chunks = ceil_div(p.ny, h);
    if (chunks > 65535) continue;
    const int rows = rows_of(h, most), tiles = ceil_div(h, rows);
    int &occ = occ_of[rows];
    if (occ == 0 && (occupancy(p, storage, rows, &occ) != cudaSuccess || occ < 1)) return best;
    const long long slots = (long long)sms * occ;
    const long long waves = ((long long)strips * chunks + slots - 1) / slots;
    const double cost = (double)waves * tiles * (0.70 + 0.0875 * (rows + fill));
    if (best_cost < 0.0 || cost < best_cost) {
      best_cost = cost;
      best = TileTiling{strips, chunks, rows, sweep_width(th), h};
    }
  }
  return best;
}

cudaError_t launch_tile(const DevParams &p, int storage, const void *gs, void *gout,
                        const float *Tin, float *Tout, unsigned *status, const StepScalars *sc,
                        const StepScalars &val, const TileTiling &tl, cudaStream_t s) {
  switch (storage) {
    case STORAGE_BF16:
      return tile_bf16_launch(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
    case STORAGE_F16:
      return tile_f16_launch(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
    default:
      return tile_launch_t<StoreF32>(p, gs, gout, Tin, Tout, status, sc, val, tl, s);
  }
}

}  // namespace lbm
