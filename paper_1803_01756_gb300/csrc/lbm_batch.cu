// Batched updates of many lattices, one launch per step for those of a kernel.
#include <algorithm>
#include <cstring>
#include <new>
#include <queue>
#include <vector>

#include "lbm_handle.h"

using lbm::BatchChannel;
using lbm::StepScalars;

struct lbm_batch {
  int device = 0;
  int storage = 0;
  lbm::DevParams mode{};  // boundary modes and physics switches shared by all lattices
  // A lattice runs in the batch with the arithmetic it has alone, and so has the same bits: the
  // first nsweep lattices (on the tile kernel or the warp sweep alone) in the batched warp
  // sweep, whose tiles are a warp's strip of a row chunk, the others (on the CTA sweep or the
  // two passes alone) in the work-list kernel.  In each part those with most tiles come first.
  std::vector<lbm_lattice *> lat;
  int nsweep = 0;
  int sweep_rows = 64;             // output rows per tile of the warp sweep
  int sweep_slots = 0;             // its resident CTAs
  std::vector<lbm::SweepBatchItem> items;
  int tile_rows = 64;              // output rows per tile (default_rows, or set / autotuned)
  int tile_cols = 0;               // output columns per tile (even with two columns per thread)
  int cpt = 1;                     // lattice columns per thread of the work-list kernel
  int grid_of[3] = {0, 0, 0};      // resident CTAs with 1 and 2 columns per thread (0: none)
  int ntiles = 0, grid = 0, sms = 1;  // of the work-list
  int sweep_tiles = 0;
  // The lattices of one launch, first .. first + n - 1 of lat: a launch of the warp sweep takes
  // kSweepBatch of them at most, and the work-list kernel takes its own.  The lattices of
  // different groups have nothing to do with one another, so each group runs its updates on a
  // stream of its own and the GPU fills with all of them (192 channels of 100 x 32 at 8 rows:
  // 34 us per update, 85 with the launches one after another).
  struct Group {
    bool sweep;
    int first, n;
    cudaStream_t stream;  // (the first group runs on the caller's)
    cudaEvent_t done;
  };
  std::vector<Group> groups;
  cudaEvent_t fork = nullptr;
  BatchChannel *d_ch[2] = {nullptr, nullptr};  // tables for even and odd steps of a call
  std::vector<BatchChannel> h_ch[2];
  StepScalars *d_sc = nullptr;                  // [chunk][n] scalars of the next chunk
  StepScalars *h_sc[2] = {nullptr, nullptr};    // pinned host staging, double buffered
  cudaEvent_t sc_ev[2] = {nullptr, nullptr};
  bool sc_used[2] = {false, false};
  int sc_buf = 0;
  int *d_counter = nullptr;
  int chunk = 16;  // steps per scalar upload; also the graph length (even)
  bool use_graph = false;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  cudaStream_t cap_stream = nullptr;
};

namespace {

using lbm_host::cuda_fail;

bool swept(const lbm_lattice *h) { return h->tile.strips > 0 || h->sweep.strips > 0; }

int tiles_of(const lbm_batch *b, const lbm_lattice *h, int rows) {
  const int H = std::min(rows, h->ny), chunks = (h->ny + H - 1) / H;
  return (swept(h) ? lbm::sweep_batch_strips(h->dp) : (h->nx + b->tile_cols - 1) / b->tile_cols) *
         chunks;
}

void drop_graph(lbm_batch *b) {
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  if (b->graph) cudaGraphDestroy(b->graph);
  b->gexec = nullptr;
  b->graph = nullptr;
}

// Layout for the current tile heights: lattices with the most work first
void layout(lbm_batch *b) {
  auto work = [&](const lbm_lattice *h) {
    return (long long)tiles_of(b, h, swept(h) ? b->sweep_rows : b->tile_rows) * h->nx;
  };
  std::stable_sort(b->lat.begin(), b->lat.end(), [&](const lbm_lattice *x, const lbm_lattice *y) {
    return swept(x) != swept(y) ? swept(x) : work(x) > work(y);
  });
  // each group of the sweep gets its share of the large lattices and of the small ones
  const std::vector<lbm_lattice *> sorted = b->lat;
  const int ng = (b->nsweep + lbm::kSweepBatch - 1) / lbm::kSweepBatch;
  int at = 0;
  for (int g = 0; g < ng; g++) {
    b->groups[g].first = at;
    for (int i = g; i < b->nsweep; i += ng) b->lat[at++] = sorted[i];
    b->groups[g].n = at - b->groups[g].first;
  }
  b->items.clear();
  b->sweep_tiles = b->ntiles = 0;
  for (auto *h : b->lat) {
    if (swept(h)) {
      b->sweep_tiles += tiles_of(b, h, b->sweep_rows);
      b->items.push_back({&h->dp, (h->ny + b->sweep_rows - 1) / b->sweep_rows});
    } else {
      b->ntiles += tiles_of(b, h, b->tile_rows);
    }
  }
  b->grid = b->grid_of[b->cpt];
  drop_graph(b);
}

// the groups, their streams and events
cudaError_t make_groups(lbm_batch *b) {
  const int n = (int)b->lat.size();
  for (int at = 0; at < b->nsweep; at += lbm::kSweepBatch)
    b->groups.push_back({true, 0, 0, nullptr, nullptr});
  if (b->nsweep < n) b->groups.push_back({false, b->nsweep, n - b->nsweep, nullptr, nullptr});
  cudaError_t e = cudaSuccess;
  for (size_t g = 1; g < b->groups.size() && e == cudaSuccess; g++) {
    e = cudaStreamCreateWithFlags(&b->groups[g].stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->groups[g].done, cudaEventDisableTiming);
  }
  if (b->groups.size() > 1 && e == cudaSuccess)
    e = cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
  return e;
}

// Greedy list schedule of lattices of one kernel at tile height H over the resident CTAs (CTAs in
// launch order, each taken by the first free slot, costing its row steps: H + 15, in the warp
// sweep H + 10, or H + 2 without the energy equation): returns the makespan in row steps and
// the number of tiles.
double schedule(const lbm_batch *b, const std::vector<const lbm_lattice *> &order, int H,
                long long &ntiles) {
  const int W = b->tile_cols;
  const bool sweep = swept(order[0]);
  std::priority_queue<double, std::vector<double>, std::greater<double>> slots;
  const int resident = sweep ? b->sweep_slots : b->grid_of[b->cpt];
  const double fill = sweep ? lbm::sweep_batch_fill(b->mode.thermal != 0) : 15.0;
  for (int k = 0; k < resident; k++) slots.push(0.0);
  double makespan = 0.0;
  ntiles = 0;
  for (const lbm_lattice *h : order) {
    const int rows = std::min(H, h->ny);
    const int chunks = (h->ny + rows - 1) / rows, strips = (h->nx + W - 1) / W;
    long long done = 0;  // CTAs of the row chunks so far
    for (int c = 0; c < chunks; c++) {
      const double len = std::min(rows, h->ny - c * rows) + fill;
      const long long upto = sweep ? lbm::sweep_batch_ctas(h->dp, c + 1) : done + strips;
      for (; done < upto; done++) {
        const double t = slots.top() + len;
        slots.pop();
        slots.push(t);
        makespan = std::max(makespan, t);
      }
    }
    ntiles += tiles_of(b, h, H);
  }
  return makespan;
}

// Time of a launch of the warp sweep at tile height H where every CTA is resident, in row steps
// of a full SM; 0 where they are not.  The tallest tile (a lattice's rows are divided evenly) is
// the launch, and a row step takes 0.71, 0.86 and 1 with one, two and three CTAs on the SM, as
// for the single lattice (lbm_sweep.cu).
double one_wave(const lbm_batch *b, const std::vector<const lbm_lattice *> &order, int H) {
  long long ctas = 0;
  int tallest = 0;
  for (const lbm_lattice *h : order) {
    const int rows = std::min(H, h->ny), chunks = (h->ny + rows - 1) / rows;
    ctas += lbm::sweep_batch_ctas(h->dp, chunks);
    tallest = std::max(tallest, (h->ny + chunks - 1) / chunks);
  }
  if (ctas > b->sweep_slots) return 0.0;
  const long long per_sm = (ctas + b->sms - 1) / b->sms, occ = b->sweep_slots / b->sms;
  return (0.57 + 0.43 * (double)per_sm / occ) *
         (tallest + lbm::sweep_batch_fill(b->mode.thermal != 0));
}

// Default tile height.  Each candidate of 128 .. 16 rows is scored by the makespan of its
// greedy schedule and the shortest wins, the taller on a tie.  Measured on GB300 against
// fixed heights, this picks the best or within 4 % of it on four shapes: 12 channels of
// 512 x 64 (16 rows, 2.8x the 64-row rate), 20 of 1024 x 256, one of 4096 x 512 and 96
// uneven channels.  When that leaves fewer tiles than SMs, most of the GPU would idle:
// then heights down to one row compete, each makespan weighted by the time of a row step
// with k tiles per SM (relative, as in the single-lattice tiling: 0.85, 1.0, 1.15 for
// k = 1 .. 3 with FP32 storage, three CTAs per SM; 0.85, 0.97, 1.42, 1.64 for k = 1 .. 4
// with 16-bit storage, four: one CTA alone is bound by the latency of its row step, a
// full SM shares the issue slots), so that a few small lattices spread over the SMs
// (200 x 50 alone: 1 row, 17.0 against 39.3 us per update with 16; 1024 x 128: 4 rows,
// 22.8 against 39.6 us).  The figures are the CTA kernel's.
//
// In the warp sweep the heights that make one wave compete by the time of that wave
// (one_wave): every height up to 24 rows, so that a few small lattices spread over the SMs,
// and the multiples of four up to 256.  GB300, FP32, us per update at the height chosen, at the
// fastest of twelve and at 16 rows: 1024 x 128 alone 16.1 (5 rows), 15.6 (3), 28.2; 8 of 200 x 50
// 14.2 (3), 14.0 (3), 24.8; 24 of them 19.1 (5), 20.2 (3), 25.5; 12 of 512 x 64 22.8 (9), 22.7 (8),
// 29.0; 48 of 100 x 32 17.0 (3), 16.9 (3), 30.3; 8 uneven ones of 64-464 x 16-80 15.2 (3),
// 14.3 (2), 28.9.  16 channels of 2.9 M nodes 76.8 at 36 (chosen), 91.9 at 48; 20 of 3.8 M 91.1 at
// 44 (chosen), 98.0 at 48; 30 of 4.1 M 108.9 at 56 (chosen), 121.4 at 64.  In several waves the
// schedule does not tell heights close apart (40 channels of 6.3 M nodes 170.4 at 96 rows and
// 163.5 at 92 in one wave, 178.7 at 40 in two), so those stay the seven.
int default_rows(const lbm_batch *b, bool sweep) {
  static const int tall[] = {128, 96, 64, 48, 32, 24, 16};
  static const int small[] = {16, 12, 8, 6, 4, 3, 2, 1};
  static const double kStep3[4] = {0.0, 0.85, 1.0, 1.15};
  static const double kStep4[5] = {0.0, 0.85, 0.97, 1.42, 1.64};
  std::vector<const lbm_lattice *> order;
  for (const lbm_lattice *h : b->lat)
    if (swept(h) == sweep) order.push_back(h);
  if (order.empty()) return 64;
  std::stable_sort(order.begin(), order.end(), [](const lbm_lattice *x, const lbm_lattice *y) {
    return (long long)x->nx * x->ny > (long long)y->nx * y->ny;
  });
  int best = 16;
  long long best_tiles = 0;
  double best_cost = 0.0;
  for (int H : tall) {
    long long n = 0;
    const double cost = schedule(b, order, H, n);
    if (best_cost == 0.0 || cost < best_cost) {
      best = H;
      best_cost = cost;
      best_tiles = n;
    }
  }
  if (sweep) {
    for (int H = 256; H >= 1; H -= H > 24 ? 4 : 1) {
      const double cost = one_wave(b, order, H);
      if (cost > 0.0 && cost < best_cost) {
        best = H;
        best_cost = cost;
      }
    }
    return best;
  }
  if (best_tiles >= b->sms) return best;
  const int occ = std::max(1, std::min(4, b->grid_of[b->cpt] / b->sms));
  const double *kStep = occ >= 4 ? kStep4 : kStep3;
  best_cost = 0.0;
  for (int H : small) {
    long long n = 0;
    const double span = schedule(b, order, H, n);
    const int k = (int)std::max(1LL, std::min<long long>(occ, (n + b->sms - 1) / b->sms));
    const double cost = span * kStep[k];
    if (best_cost == 0.0 || cost < best_cost) {
      best = H;
      best_cost = cost;
    }
  }
  return best;
}

// Channel tables for the lattices' current buffers: table 0 for steps at even
// offsets from now, table 1 for odd offsets.
int upload_tables(lbm_batch *b, cudaStream_t s) {
  const int W = b->tile_cols;
  int begin = 0;
  for (int par = 0; par < 2; par++) b->h_ch[par].resize(b->lat.size());
  for (size_t i = 0; i < b->lat.size(); i++) {
    lbm_lattice *h = b->lat[i];
    const int H = std::min(b->tile_rows, h->ny);
    for (int par = 0; par < 2; par++) {
      const int gc = h->cur ^ par;
      const int tc = h->dp.thermal ? (h->tcur ^ par) : h->tcur;
      BatchChannel &c = b->h_ch[par][i];
      c.p = h->dp;
      c.gs = h->g[gc];
      c.gout = h->g[1 - gc];
      c.Tin = h->T[tc];
      c.Tout = h->dp.thermal ? h->T[1 - tc] : h->T[tc];
      c.status = h->status;
      c.W = W;
      c.H = H;
      c.strips = (h->nx + W - 1) / W;
      c.tile_begin = begin;
    }
    if (!swept(h)) begin += tiles_of(b, h, b->tile_rows);
  }
  const size_t bytes = sizeof(BatchChannel) * b->lat.size();
  for (int par = 0; par < 2; par++)
    LBM_CUDA(cudaMemcpyAsync(b->d_ch[par], b->h_ch[par].data(), bytes, cudaMemcpyHostToDevice, s));
  return LBM_OK;
}

// CTAs of a launch of the work-list kernel: the resident grid, or one per tile when there are
// fewer tiles
int launch_grid(const lbm_batch *b) { return std::min(b->grid, b->ntiles); }

// step k of a chunk of group g with the buffers of table par
cudaError_t launch_one(lbm_batch *b, const lbm_batch::Group &g, int k, int par, cudaStream_t s) {
  const BatchChannel *ch = b->d_ch[par] + g.first;
  const StepScalars *sc = b->d_sc + (size_t)k * b->lat.size() + g.first;
  if (g.sweep) return lbm::launch_sweep_batch(b->storage, b->items.data() + g.first, g.n, ch, sc, s);
  return lbm::launch_fused_batch(b->mode, b->storage, b->cpt, ch, g.n, sc, b->ntiles, b->d_counter,
                                 launch_grid(b), s);
}

// The m steps of a chunk, the first with table phase: the groups beside one another, each on
// its stream, behind the work of stream s and before what follows on it.
int launch_chunk(lbm_batch *b, int m, int phase, cudaStream_t s) {
  const int ng = (int)b->groups.size();
  if (ng > 1) LBM_CUDA(cudaEventRecord(b->fork, s));
  int forked = 1;
  cudaError_t e = cudaSuccess;
  for (; forked < ng && e == cudaSuccess; forked++)
    e = cudaStreamWaitEvent(b->groups[forked].stream, b->fork, 0);
  for (int k = 0; k < m && e == cudaSuccess; k++)
    for (int g = 0; g < ng && e == cudaSuccess; g++)
      e = launch_one(b, b->groups[g], k, (phase + k) & 1, g ? b->groups[g].stream : s);
  for (int g = 1; g < forked; g++) {  // (joined also when a launch failed)
    cudaError_t j = cudaEventRecord(b->groups[g].done, b->groups[g].stream);
    if (j == cudaSuccess) j = cudaStreamWaitEvent(s, b->groups[g].done, 0);
    if (e == cudaSuccess) e = j;
  }
  return cuda_fail(e);
}

int build_graph(lbm_batch *b) {
  drop_graph(b);
  LBM_CUDA(cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
  const int rc = launch_chunk(b, b->chunk, 0, b->cap_stream);
  cudaError_t e = cudaStreamEndCapture(b->cap_stream, &b->graph);
  if (rc != LBM_OK) return rc;
  LBM_CUDA(e);
  LBM_CUDA(cudaGraphInstantiate(&b->gexec, b->graph, 0));
  return LBM_OK;
}

void free_batch(lbm_batch *b) {
  drop_graph(b);
  for (auto &g : b->groups) {
    if (g.done) cudaEventDestroy(g.done);
    if (g.stream) cudaStreamDestroy(g.stream);
  }
  if (b->fork) cudaEventDestroy(b->fork);
  cudaFree(b->d_ch[0]);
  cudaFree(b->d_ch[1]);
  cudaFree(b->d_sc);
  cudaFree(b->d_counter);
  for (int k = 0; k < 2; k++) {
    if (b->h_sc[k]) cudaFreeHost(b->h_sc[k]);
    if (b->sc_ev[k]) cudaEventDestroy(b->sc_ev[k]);
  }
  if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
}

}  // namespace

extern "C" {

int lbm_batch_create(lbm_h *lattices, int n, lbm_batch_h *out) {
  if (!lattices || n < 1 || !out) return LBM_ERR_ARG;
  *out = nullptr;
  lbm_lattice *first = lattices[0];
  if (!first) return LBM_ERR_ARG;
  for (int i = 0; i < n; i++) {
    lbm_lattice *h = lattices[i];
    // lattices on the fused or the two-pass path (both keep the fused kernel's 32-bit
    // element offsets, which the batched kernel uses)
    if (!h || h->device != first->device ||
        (h->kernel != LBM_KERNEL_FUSED && h->kernel != LBM_KERNEL_TWOPASS))
      return LBM_ERR_ARG;
    if (h->dp.y_walls != first->dp.y_walls || h->dp.x_open != first->dp.x_open ||
        h->dp.thermal != first->dp.thermal || h->dp.multiphase != first->dp.multiphase ||
        h->p.storage != first->p.storage)
      return LBM_ERR_ARG;
    for (int j = 0; j < i; j++)
      if (lattices[j] == h) return LBM_ERR_ARG;
  }
  lbm_batch *b = new (std::nothrow) lbm_batch();
  if (!b) return LBM_ERR_OOM;
  b->device = first->device;
  b->storage = first->p.storage;
  b->mode = first->dp;
  b->lat.assign(lattices, lattices + n);
  cudaError_t e = cudaSetDevice(b->device);
  for (int c = 1; c <= 2 && e == cudaSuccess; c++)
    b->grid_of[c] = lbm::fused_batch_grid(b->mode, b->storage, c, b->device);
  b->grid = b->grid_of[1];
  b->tile_cols = lbm::fused_batch_width(1);
  if (b->grid > 0 &&
      cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device) != cudaSuccess)
    b->grid = 0;
  if (b->grid < 1) {
    delete b;
    return LBM_ERR_CUDA;
  }
  for (int k = 0; k < 2 && e == cudaSuccess; k++) e = cudaMalloc(&b->d_ch[k], sizeof(BatchChannel) * n);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_sc, sizeof(StepScalars) * n * b->chunk);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_counter, 2 * sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(b->d_counter, 0, 2 * sizeof(int));
  for (int k = 0; k < 2 && e == cudaSuccess; k++)
    e = cudaMallocHost((void **)&b->h_sc[k], sizeof(StepScalars) * n * b->chunk);
  for (int k = 0; k < 2 && e == cudaSuccess; k++)
    e = cudaEventCreateWithFlags(&b->sc_ev[k], cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    free_batch(b);
    delete b;
    return cuda_fail(e);
  }
  b->sweep_slots = lbm::sweep_batch_slots(b->mode, b->storage, b->device);
  for (auto *h : b->lat) b->nsweep += swept(h) ? 1 : 0;
  e = b->nsweep > 0 && b->sweep_slots < 1 ? cudaErrorUnknown : make_groups(b);
  if (e != cudaSuccess) {
    free_batch(b);
    delete b;
    return cuda_fail(e);
  }
  b->sweep_rows = default_rows(b, true);
  b->tile_rows = default_rows(b, false);
  layout(b);
  *out = b;
  return LBM_OK;
}

int lbm_batch_step(lbm_batch_h b, long nsteps, void *stream) {
  if (!b || nsteps < 0) return LBM_ERR_ARG;
  LBM_CUDA(cudaSetDevice(b->device));
  cudaStream_t s = (cudaStream_t)stream;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  LBM_CUDA(cudaStreamIsCapturing(s, &cs));
  if (cs != cudaStreamCaptureStatusNone) return LBM_ERR_ARG;  // as lbm_step
  int rc = upload_tables(b, s);
  if (rc) return rc;
  const int n = (int)b->lat.size();
  long done = 0;
  int phase = 0;  // parity of the steps taken in this call
  while (done < nsteps) {
    const int m = (int)std::min<long>(b->chunk, nsteps - done);
    const int buf = b->sc_buf;
    if (b->sc_used[buf]) LBM_CUDA(cudaEventSynchronize(b->sc_ev[buf]));
    StepScalars *hs = b->h_sc[buf];
    for (int k = 0; k < m; k++)
      for (int i = 0; i < n; i++)
        hs[(size_t)k * n + i] = lbm_host::scalars_at(b->lat[i], b->lat[i]->t + done + k);
    LBM_CUDA(cudaMemcpyAsync(b->d_sc, hs, sizeof(StepScalars) * n * m, cudaMemcpyHostToDevice, s));
    LBM_CUDA(cudaEventRecord(b->sc_ev[buf], s));
    b->sc_used[buf] = true;
    b->sc_buf ^= 1;
    if (b->use_graph && m == b->chunk && phase == 0) {
      if (!b->gexec) {
        rc = build_graph(b);
        if (rc) return rc;
      }
      LBM_CUDA(cudaGraphLaunch(b->gexec, s));
    } else {
      // (phase: a step runs with the table of its parity in the call)
      rc = launch_chunk(b, m, phase, s);
      if (rc) return rc;
    }
    phase = (phase + m) & 1;
    done += m;
  }
  for (auto *h : b->lat) {
    h->t += nsteps;
    if (nsteps & 1) {
      h->cur ^= 1;
      if (h->dp.thermal) h->tcur ^= 1;
    }
  }
  return LBM_OK;
}

int lbm_batch_set_graph(lbm_batch_h b, int enable) {
  if (!b) return LBM_ERR_ARG;
  b->use_graph = enable != 0;
  if (!b->use_graph) drop_graph(b);
  return LBM_OK;
}

int lbm_batch_set_tile_rows(lbm_batch_h b, int rows) {
  if (!b || rows < 1) return LBM_ERR_ARG;
  b->sweep_rows = b->tile_rows = rows;
  layout(b);
  return LBM_OK;
}

int lbm_batch_set_tiling(lbm_batch_h b, int rows, int cols, int cols_per_thread) {
  if (!b || rows < 1 || cols < 1) return LBM_ERR_ARG;
  if (cols_per_thread != 1 && cols_per_thread != 2) return LBM_ERR_ARG;
  if (b->grid_of[cols_per_thread] < 1) return LBM_ERR_ARG;
  if (cols > lbm::fused_batch_width(cols_per_thread)) return LBM_ERR_ARG;
  if (cols_per_thread == 2 && (cols & 1)) return LBM_ERR_ARG;
  // (the warp sweep takes the rows: its strips have their own width and two columns per lane)
  b->sweep_rows = b->tile_rows = rows;
  b->tile_cols = cols;
  b->cpt = cols_per_thread;
  layout(b);
  return LBM_OK;
}

int lbm_batch_tiling(lbm_batch_h b, int *rows, int *cols, int *cols_per_thread) {
  if (!b) return LBM_ERR_ARG;
  const bool all = b->nsweep == (int)b->lat.size();
  if (rows) *rows = all ? b->sweep_rows : b->tile_rows;
  if (cols) *cols = all ? lbm::sweep_batch_width(b->mode.thermal != 0) : b->tile_cols;
  if (cols_per_thread) *cols_per_thread = all ? 2 : b->cpt;
  return LBM_OK;
}

int lbm_batch_autotune(lbm_batch_h b, int steps_per_candidate, int *best_rows, void *stream) {
  if (!b || steps_per_candidate < 2) return LBM_ERR_ARG;
  LBM_CUDA(cudaSetDevice(b->device));
  cudaStream_t s = (cudaStream_t)stream;
  struct Cand {
    int sweep_rows, rows, cols, cpt;
  };
  static const int heights[] = {16, 24, 32, 48, 64, 96, 128};
  cudaEvent_t e0, e1;
  LBM_CUDA(cudaEventCreate(&e0));
  LBM_CUDA(cudaEventCreate(&e1));
  const bool graph = b->use_graph;
  b->use_graph = false;
  float best = -1.0f;
  const Cand before{b->sweep_rows, b->tile_rows, b->tile_cols, b->cpt};
  Cand win = before;
  int rc = LBM_OK;
  auto use = [&](const Cand &c) {
    b->sweep_rows = c.sweep_rows;
    b->tile_rows = c.rows;
    b->tile_cols = c.cols;
    b->cpt = c.cpt;
    layout(b);
  };
  auto time_one = [&](const Cand &c) -> int {
    use(c);
    int r = lbm_batch_step(b, 2, stream);  // warm-up
    if (r) return r;
    LBM_CUDA(cudaEventRecord(e0, s));
    r = lbm_batch_step(b, steps_per_candidate, stream);
    if (r) return r;
    LBM_CUDA(cudaEventRecord(e1, s));
    LBM_CUDA(cudaEventSynchronize(e1));
    float ms = 0.0f;
    LBM_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    if (best < 0.0f || ms < best) {
      best = ms;
      win = c;
    }
    return LBM_OK;
  };
  const bool all = b->nsweep == (int)b->lat.size();
  if (all) {
    // the warp sweep: the same heights, the height in place (the default lies between them where
    // that makes one wave) and three quarters of the winner's
    auto rows_only = [&](int H) { return Cand{H, H, before.cols, before.cpt}; };
    for (int H : heights)
      if (rc == LBM_OK) rc = time_one(rows_only(H));
    if (rc == LBM_OK) rc = time_one(before);
    if (rc == LBM_OK) rc = time_one(rows_only(std::max(1, win.sweep_rows * 3 / 4)));
  } else {
    // tile heights at the widest tiles, for each column count the mode has a kernel for
    for (int cpt = 1; cpt <= 2 && rc == LBM_OK; cpt++) {
      if (b->grid_of[cpt] < 1) continue;
      for (int H : heights) {
        rc = time_one(Cand{H, H, lbm::fused_batch_width(cpt), cpt});
        if (rc) break;
      }
    }
    // then narrower tiles (three quarters and half the width) at the winner's height
    const Cand base = win;
    const int Wmax = lbm::fused_batch_width(base.cpt);
    for (int num : {3, 2}) {
      if (rc) break;
      int W = Wmax * num / 4;
      if (base.cpt == 2) W &= ~1;
      rc = time_one(Cand{base.sweep_rows, base.rows, W, base.cpt});
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  b->use_graph = graph;
  use(rc == LBM_OK ? win : before);
  if (best_rows) *best_rows = all ? b->sweep_rows : b->tile_rows;
  return rc;
}

int lbm_batch_info(lbm_batch_h b, int *ntiles, int *grid, int *tile_rows) {
  if (!b) return LBM_ERR_ARG;
  if (ntiles) *ntiles = b->sweep_tiles + b->ntiles;
  if (grid)
    *grid = (b->nsweep > 0 ? b->sweep_slots * lbm::sweep_batch_warps() : 0) +
            (b->nsweep < (int)b->lat.size() ? b->grid : 0);
  if (tile_rows) *tile_rows = b->nsweep == (int)b->lat.size() ? b->sweep_rows : b->tile_rows;
  return LBM_OK;
}

void lbm_batch_destroy(lbm_batch_h b) {
  if (!b) return;
  cudaSetDevice(b->device);
  cudaDeviceSynchronize();
  free_batch(b);
  delete b;
}

}  // extern "C"
