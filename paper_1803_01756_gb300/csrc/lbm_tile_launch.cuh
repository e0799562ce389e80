// The single-lattice tile kernel (lbm_tile.cuh) and its launch, templated on the population
// storage: lbm_tile.cu (FP32, with the tiling), lbm_tile_f16.cu and lbm_tile_bf16.cu
// instantiate one each, so that the three compile in parallel.
#pragma once
#include <algorithm>

#include "lbm_tile.cuh"

namespace lbm {

namespace {

// Most warps of a CTA, for which the registers are sized (96 a thread, no spills): 10 output
// rows and their 10 halo rows a tile.  28 warps (18 rows, 72 registers, spills) are faster on
// lattices of many tiles (777 x 333: 11.5 against 13.9 us per update, 1024 x 128 6.5 against 7.4)
// and slower where there are few (200 x 50: 4.9 against 3.5 us, 1600 x 48: 5.1 against 4.5 us);
// 14 and 16 warps spend too much of a tile on the halo (777 x 333: 23.6 and 18.1 us).
constexpr int TW = 20;

template <bool YW, bool XO, bool TH, bool MP, class ST>
__global__ void __launch_bounds__(32 * TW, 1)
    k_tile(const __grid_constant__ DevParams p, const __grid_constant__ SweepConsts k,
           const typename ST::T *gs, typename ST::T *gout, const float *Tin, float *Tout,
           unsigned *status, const StepScalars *__restrict__ sc, const StepScalars val,
           int rows) {
  __shared__ TileSmem<TW> S;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const StepScalars ssc = sc ? *sc : val;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int Y0 = (int)(((long long)blockIdx.y * p.ny) / gridDim.y);
  const int ye = (int)(((long long)(blockIdx.y + 1) * p.ny) / gridDim.y);
  Tile<YW, XO, TH, MP, ST, TW> t(p, k, gs, gout, Tin, Tout, ssc,
                                 sweep_c0((int)blockIdx.x, TH));
  for (int y = Y0; y < ye; y += rows) {
    if (y > Y0) __syncthreads();
    t.run(y, min(y + rows, ye), S);
  }
  t.finish(status);
}

template <class ST>
using TileFn = void (*)(DevParams, SweepConsts, const typename ST::T *, typename ST::T *,
                        const float *, float *, unsigned *, const StepScalars *, StepScalars, int);

template <class ST>
TileFn<ST> tile_variant(const DevParams &p) {
#define KT(a, b, c, d) k_tile<a, b, c, d, ST>
  static const TileFn<ST> table[16] = {
      KT(false, false, false, false), KT(false, false, false, true), KT(false, false, true, false),
      KT(false, false, true, true),   KT(false, true, false, false), KT(false, true, false, true),
      KT(false, true, true, false),   KT(false, true, true, true),   KT(true, false, false, false),
      KT(true, false, false, true),   KT(true, false, true, false),  KT(true, false, true, true),
      KT(true, true, false, false),   KT(true, true, false, true),   KT(true, true, true, false),
      KT(true, true, true, true)};
#undef KT
  const int k = (p.y_walls ? 8 : 0) | (p.x_open ? 4 : 0) | (p.thermal ? 2 : 0) |
                (p.multiphase ? 1 : 0);
  return table[k];
}

template <class ST>
cudaError_t tile_launch_t(const DevParams &p, const void *gs, void *gout, const float *Tin,
                          float *Tout, unsigned *status, const StepScalars *sc,
                          const StepScalars &val, const TileTiling &tl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tl.strips, (unsigned)tl.chunks);
  cfg.blockDim = dim3((unsigned)(32 * (tl.rows + 2 * sweep_rows(p.thermal != 0))));
  cfg.stream = s;
  // dependent launch: the next update's CTAs take their places while this one drains, which
  // hides part of the launch on every size the kernel is used for
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, tile_variant<ST>(p), p, sweep_consts(p),
                            static_cast<const typename ST::T *>(gs),
                            static_cast<typename ST::T *>(gout), Tin, Tout, status, sc, val,
                            tl.rows);
}

template <class ST>
cudaError_t tile_occupancy_t(const DevParams &p, int rows, int *occ) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      occ, tile_variant<ST>(p), 32 * (rows + 2 * sweep_rows(p.thermal != 0)), 0);
}

}  // namespace

}  // namespace lbm
