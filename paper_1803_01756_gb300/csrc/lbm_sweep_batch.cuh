// The warp sweep (lbm_sweep.cuh) over many lattices in one launch.
//
// The lattices' physics travel as kernel arguments, so that a CTA reads them through the
// constant bank like the single-lattice kernel (the CTA-sweep batch kernel copies them to
// shared memory, and its loop reads them from there); the buffers of the step come from the
// batch's device table.  A CTA finds its lattice by its index; its warps take the
// lattice's tiles as in the single-lattice kernel, and the hardware hands the CTAs out in order, largest
// lattices first.
// lbm_sweep_batch.cu, lbm_sweep_batch_f16.cu and lbm_sweep_batch_bf16.cu instantiate one
// storage each.
#pragma once

#include "lbm_sweep_launch.cuh"

namespace lbm {

namespace {

struct SweepBatchArgs {
  struct Entry {
    DevParams p;
    SweepConsts k;
    int begin;         // index of the lattice's first CTA
    int strips, chunks;
  };
  int n;
  Entry e[kSweepBatch];
};
static_assert(sizeof(SweepBatchArgs) <= 32764 - 64, "kernel arguments");

template <bool YW, bool XO, bool TH, bool MP, class ST>
__global__ void __launch_bounds__(SNT, SMIN)
    k_sweep_batch(const __grid_constant__ SweepBatchArgs a, const BatchChannel *__restrict__ ch,
                  const StepScalars *__restrict__ sc) {
  const int b = (int)blockIdx.x;
  int lo = 0, hi = a.n - 1;  // last lattice whose first CTA is b or before
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.e[mid].begin <= b) lo = mid;
    else hi = mid - 1;
  }
  const SweepBatchArgs::Entry &e = a.e[lo];
  const BatchChannel &c = ch[lo];
  const StepScalars ssc = sc[lo];
  __shared__ float4 rings[SW][TH ? 4 * 3 * 32 : 32];
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
  const int cols = sweep_cols(e.strips), local = b - e.begin;
  const SweepTile t =
      sweep_tile<sweep_div<YW, XO, TH, MP, ST>()>(e.strips, local % cols, local / cols, warp);
  if (t.chunk >= e.chunks) return;
  const int Y0 = (int)(((long long)t.chunk * e.p.ny) / e.chunks);
  const int ye = (int)(((long long)(t.chunk + 1) * e.p.ny) / e.chunks);
  Sweep<YW, XO, TH, MP, ST> s(e.p, e.k, static_cast<const typename ST::T *>(c.gs),
                              static_cast<typename ST::T *>(c.gout), c.Tin, c.Tout, ssc,
                              sweep_c0(t.strip, TH), Y0, ye, rings[warp]);
  s.run(c.status);
}

template <class ST>
using SweepBatchFn = void (*)(SweepBatchArgs, const BatchChannel *, const StepScalars *);

template <class ST>
SweepBatchFn<ST> sweep_batch_variant(const DevParams &p) {
#define KB(a, b, c, d) k_sweep_batch<a, b, c, d, ST>
  static const SweepBatchFn<ST> table[16] = {
      KB(false, false, false, false), KB(false, false, false, true), KB(false, false, true, false),
      KB(false, false, true, true),   KB(false, true, false, false), KB(false, true, false, true),
      KB(false, true, true, false),   KB(false, true, true, true),   KB(true, false, false, false),
      KB(true, false, false, true),   KB(true, false, true, false),  KB(true, false, true, true),
      KB(true, true, false, false),   KB(true, true, false, true),   KB(true, true, true, false),
      KB(true, true, true, true)};
#undef KB
  const int k = (p.y_walls ? 8 : 0) | (p.x_open ? 4 : 0) | (p.thermal ? 2 : 0) |
                (p.multiphase ? 1 : 0);
  return table[k];
}

template <class ST>
int sweep_batch_slots_t(const DevParams &p, int device) {
  int sms = 0, occ = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sweep_batch_variant<ST>(p), SNT, 0) !=
          cudaSuccess)
    return 0;
  return sms * occ;
}

template <class ST>
cudaError_t sweep_batch_launch_t(const SweepBatchItem *items, int n, const BatchChannel *ch,
                                 const StepScalars *sc, cudaStream_t s) {
  if (n < 1 || n > kSweepBatch) return cudaErrorInvalidValue;
  SweepBatchArgs a;
  a.n = n;
  long long ctas = 0;
  for (int i = 0; i < n; i++) {
    SweepBatchArgs::Entry &e = a.e[i];
    e.p = *items[i].p;
    e.k = sweep_consts(e.p);
    e.begin = (int)ctas;
    e.strips = sweep_strips(e.p.nx, e.p.thermal != 0);
    e.chunks = items[i].chunks;
    ctas += sweep_ctas(e.strips, e.chunks);
    if (ctas > 2147483647LL) return cudaErrorInvalidConfiguration;
  }
  sweep_batch_variant<ST>(*items[0].p)<<<(unsigned)ctas, SNT, 0, s>>>(a, ch, sc);
  return cudaGetLastError();
}

}  // namespace

}  // namespace lbm
