// The single-lattice kernel of the warp sweep (lbm_sweep.cuh) and its launch, templated on the
// population storage: lbm_sweep.cu (FP32, with the tiling), lbm_sweep_f16.cu and
// lbm_sweep_bf16.cu instantiate one each, so that the three compile in parallel.
#pragma once
#include <algorithm>

#include "lbm_sweep.cuh"

namespace lbm {

namespace {

constexpr int SW = 4;  // warps of a CTA: four adjacent strips, which share their halo columns
                       // in L1 (one-warp CTAs: 48.4 against 47.9 us on 4096 x 512)
constexpr int SNT = 32 * SW;
// CTAs across a lattice: its strips four by four.  One or two strips leave no warp idle:
// the warps of a CTA then take four or two row chunks (5 x 65537: 75 us per update, 249 with a
// CTA per row chunk).
__host__ __device__ constexpr int sweep_cols(int strips) { return (strips + SW - 1) / SW; }
// row chunks of a CTA
__host__ __device__ constexpr int sweep_stack(int strips) {
  return strips == 1 ? SW : strips == 2 ? SW / 2 : 1;
}
// CTAs along it
__host__ __device__ constexpr int sweep_rows_of_ctas(int strips, int chunks) {
  return (chunks + sweep_stack(strips) - 1) / sweep_stack(strips);
}
// The strip and row chunk of a warp of the CTA in column bx and row by.  The two forms are the
// same numbers; with one or the other the compiler schedules the row steps differently (GB300,
// 4096 x 512, us per update, DIV / not: open ends FP32 47.7 / 48.2, FP16 53.5 / 54.0; doubly
// periodic FP32 54.5 / 66.1, FP16 60.0 / 54.2; walls with periodic x FP32 55.5 / 52.7, 1237 x 531
// FP16 30.4 / 26.6; open ends without the pseudopotential FP32 47.2 / 43.3).
struct SweepTile {
  int strip, chunk;
};
template <bool DIV>
__device__ __forceinline__ SweepTile sweep_tile(int strips, int bx, int by, int warp) {
  if (DIV) {
    if (strips > 2) return SweepTile{bx * SW + warp, by};
    const int tile = by * SW + warp;
    return SweepTile{tile % strips, tile / strips};
  }
  const int sh = strips == 1 ? 2 : strips == 2 ? 1 : 0;
  return SweepTile{bx * SW + (warp & ((SW - 1) >> sh)), (by << sh) + (warp >> (2 - sh))};
}
template <bool YW, bool XO, bool TH, bool MP, class ST>
__host__ __device__ constexpr bool sweep_div() {
  return (MP || !TH) && (XO || (!YW && sizeof(typename ST::T) == 4));
}
// Resident CTAs per SM the registers are sized for: 12 warps with 168 registers a thread.
// Eight warps with 214 registers let the compiler keep more constants but cover less of the
// latency of a row step (4096 x 512: 52.7 against 48.6 us per update, 16384 x 2048: 664
// against 575 us, 16-bit storage 987 against 720 us); 16 warps (128 registers) spill.
constexpr int SMIN = 3;

template <bool YW, bool XO, bool TH, bool MP, class ST>
__global__ void __launch_bounds__(SNT, SMIN)
    k_sweep(const __grid_constant__ DevParams p, const __grid_constant__ SweepConsts k,
            const typename ST::T *gs, typename ST::T *gout, const float *Tin, float *Tout,
            unsigned *status, const StepScalars *__restrict__ sc, const StepScalars val,
            int strips, int chunks) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const StepScalars ssc = sc ? *sc : val;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ float4 rings[SW][TH ? 4 * 3 * 32 : 32];
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const SweepTile t =
      sweep_tile<sweep_div<YW, XO, TH, MP, ST>()>(strips, (int)blockIdx.x, (int)blockIdx.y, warp);
  // (a warp beyond the last strip sweeps without a store: returning here is 3 % slower on
  // 1237 x 531)
  if (t.chunk >= chunks) return;
  const int Y0 = (int)(((long long)t.chunk * p.ny) / chunks);
  const int ye = (int)(((long long)(t.chunk + 1) * p.ny) / chunks);
  float4 *ring = rings[warp];
  Sweep<YW, XO, TH, MP, ST> s(p, k, gs, gout, Tin, Tout, ssc, sweep_c0(t.strip, TH), Y0, ye,
                              ring);
  s.run(status);
}

template <class ST>
using SweepFn = void (*)(DevParams, SweepConsts, const typename ST::T *, typename ST::T *,
                         const float *, float *, unsigned *, const StepScalars *, StepScalars, int,
                         int);

template <class ST>
SweepFn<ST> sweep_variant(const DevParams &p) {
#define KS(a, b, c, d) k_sweep<a, b, c, d, ST>
  static const SweepFn<ST> table[16] = {
      KS(false, false, false, false), KS(false, false, false, true), KS(false, false, true, false),
      KS(false, false, true, true),   KS(false, true, false, false), KS(false, true, false, true),
      KS(false, true, true, false),   KS(false, true, true, true),   KS(true, false, false, false),
      KS(true, false, false, true),   KS(true, false, true, false),  KS(true, false, true, true),
      KS(true, true, false, false),   KS(true, true, false, true),   KS(true, true, true, false),
      KS(true, true, true, true)};
#undef KS
  const int k = (p.y_walls ? 8 : 0) | (p.x_open ? 4 : 0) | (p.thermal ? 2 : 0) |
                (p.multiphase ? 1 : 0);
  return table[k];
}

long long sweep_ctas(int strips, int chunks) {
  return (long long)sweep_cols(strips) * sweep_rows_of_ctas(strips, chunks);
}

template <class ST>
cudaError_t sweep_launch_t(const DevParams &p, const void *gs, void *gout, const float *Tin,
                           float *Tout, unsigned *status, const StepScalars *sc,
                           const StepScalars &val, const SweepTiling &tl, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)sweep_cols(tl.strips),
                     (unsigned)sweep_rows_of_ctas(tl.strips, tl.chunks));
  cfg.blockDim = dim3(SNT);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = tl.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, sweep_variant<ST>(p), p, sweep_consts(p),
                            static_cast<const typename ST::T *>(gs),
                            static_cast<typename ST::T *>(gout), Tin, Tout, status, sc, val,
                            tl.strips, tl.chunks);
}

template <class ST>
cudaError_t sweep_occupancy_t(const DevParams &p, int *occ) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, sweep_variant<ST>(p), SNT, 0);
}

}  // namespace

}  // namespace lbm
