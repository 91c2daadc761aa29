// Autotuner of the particle layout: the tile shape of the particle sort and the
// sort cadence, timed on a window of steps of the run itself (by default its first
// steps) and cached per run shape and window. Every trial is an ordinary context
// built through the public ABI. pic_autotune's trials push every chunk: on the
// first steps nearly all plasma is at rest, where chunks only move their boxes, and
// a layout chosen there is one for a push that has next to nothing to do (the run's
// costs grow with the pulse's way through the plasma: on the 4096 x 256 stage tiles
// of 8 x 8 take 0.19 ms a step over steps 20 to 148 and 0.68 from step 2500 on,
// tiles of 8 x 16 take 0.22 and 0.61). pic_autotune_window's are the run's own steps
// of the window that the caller names.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <vector>

#include "../../include/pic.h"
#include "pic_batch.h"

namespace {

// trial sets: tiles of 8/16/32 cells on each axis, then cadences around the default
constexpr int kTiles[3] = {8, 16, 32};
constexpr int kCadences[5] = {8, 16, 32, 64, 128};

// nx, nz, ppc_x, ppc_z, order, precision, gamma*1e6, warm-up steps, timed steps; for a window of the run itself also what
// decides which plasma moves in it, and what a step costs besides the push
typedef std::vector<double> Key;

std::mutex g_mu;
std::map<Key, pic_tune_result> g_cache;

Key key_of(const pic_config* c, const pic_plasma* p, const pic_laser* l, int warm, int steps, bool all) {
  Key k{(double)c->nx, (double)c->nz, (double)p->ppc_x, (double)p->ppc_z, (double)c->shape_order, (double)c->precision,
        (double)(long long)(c->gamma_boost * 1e6), (double)warm, (double)steps, all ? 1.0 : 0.0};
  if (all) return k;
  const double more[] = {c->dz_lab, c->dx, c->courant, c->dt, c->theta, (double)c->pml_cells, (double)c->filter_passes,
                         (double)c->filter_stride, (double)c->filter_compensate, (double)c->gather_scheme,
                         (double)c->filter_J, (double)c->filter_gather, (double)c->particle_guard,
                         (double)c->moving_window, c->window_beta, p->n0, p->z_start_lab, p->ramp_lab, p->length_lab,
                         (double)p->ions};
  k.insert(k.end(), std::begin(more), std::end(more));
  for (int q = 0; q < 4; q++) k.push_back((double)c->filter_stride_set[q]);
  if (l) {
    const double pulse[] = {l->lambda0, l->a0, l->w0, l->tau_fwhm, l->t_peak, l->x_center, l->phase, l->z_antenna, l->beta_s};
    k.insert(k.end(), std::begin(pulse), std::end(pulse));
  }
  return k;
}

// one trial: a context with this layout, warm-up steps, then timed steps (ms per step; < 0 on failure)
double trial(const pic_config* cfg0, const pic_plasma* pl, const pic_laser* laser, int tx, int tz, int sort_every,
             int warm, int steps, bool all, pic_alloc_fn alloc, pic_free_fn free_fn, void* user, void* stream) {
  pic_config cfg = *cfg0;
  cfg.tile_x = tx;
  cfg.tile_z = tz;
  cfg.sort_every = sort_every;
  pic_ctx* ctx = nullptr;
  if (pic_init(&cfg, alloc, free_fn, user, stream, &ctx) != PIC_OK) return -1.0;
  if (all) picgb::push_every_chunk(ctx);
  double ms = -1.0;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (pic_load_plasma(ctx, pl) == PIC_OK && (!laser || pic_inject_laser(ctx, laser) == PIC_OK) &&
      pic_step(ctx, warm) == PIC_OK && pic_sync(ctx) == PIC_OK && cudaEventCreate(&e0) == cudaSuccess &&
      cudaEventCreate(&e1) == cudaSuccess) {
    cudaEventRecord(e0, (cudaStream_t)stream);
    const int r = pic_step(ctx, steps);
    cudaEventRecord(e1, (cudaStream_t)stream);
    float t = 0.0f;
    if (r == PIC_OK && pic_sync(ctx) == PIC_OK && cudaEventSynchronize(e1) == cudaSuccess &&
        cudaEventElapsedTime(&t, e0, e1) == cudaSuccess)
      ms = (double)t / steps;
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  pic_free(ctx);
  return ms;
}

void record(pic_tune_result* o, int tx, int tz, int se, double ms) {
  if (o->n_trials >= PIC_TUNE_MAX_TRIALS) return;
  const int i = o->n_trials++;
  o->trial_tile_x[i] = tx;
  o->trial_tile_z[i] = tz;
  o->trial_sort_every[i] = se;
  o->trial_ms[i] = ms;
}

// all: the trials push every chunk
int tune(const pic_config* cfg, const pic_plasma* plasma, const pic_laser* laser, int warm, int steps, bool all,
         pic_alloc_fn alloc, pic_free_fn free_fn, void* alloc_user, void* cuda_stream, pic_tune_result* out) {
  if (!cfg || !plasma || !out || out->struct_size != sizeof(pic_tune_result)) return PIC_EINVAL;
  if (steps < 1 || warm < 0 || cfg->dim != 2) return PIC_EINVAL;
  const Key key = key_of(cfg, plasma, laser, warm, steps, all);
  {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_cache.find(key);
    if (it != g_cache.end()) {
      *out = it->second;
      out->cached = 1;
      return PIC_OK;
    }
  }
  pic_tune_result r{};
  r.struct_size = sizeof(pic_tune_result);
  r.version = PIC_API_VERSION;
  // one untimed trial first: the GPU reaches its clocks before the candidates are compared
  trial(cfg, plasma, laser, kTiles[0], kTiles[2], 32, warm, steps, all, alloc, free_fn, alloc_user, cuda_stream);
  // 1. tile shape at the default cadence; each tile timed twice, the faster time counts
  double best = -1.0;
  int btx = 0, btz = 0;
  for (int tx : kTiles)
    for (int tz : kTiles) {
      double ms = -1.0;
      for (int rep = 0; rep < 2; rep++) {
        const double m = trial(cfg, plasma, laser, tx, tz, 32, warm, steps, all, alloc, free_fn, alloc_user, cuda_stream);
        if (m > 0.0 && (ms < 0.0 || m < ms)) ms = m;
      }
      record(&r, tx, tz, 32, ms);
      if (ms > 0.0 && (best < 0.0 || ms < best)) { best = ms; btx = tx; btz = tz; }
    }
  if (best < 0.0) return PIC_ECUDA;
  // 2. sort cadence for that tile, twice each (the faster counts), all over the same steps, at least two periods of the
  // longest: the cost of a step changes along a run
  int bse = 32;
  double bse_ms = -1.0;
  for (int se : kCadences) {
    const int n = std::max(steps, 2 * kCadences[4]);
    double ms = -1.0;
    for (int rep = 0; rep < 2; rep++) {
      const double m = trial(cfg, plasma, laser, btx, btz, se, warm, n, all, alloc, free_fn, alloc_user, cuda_stream);
      if (m > 0.0 && (ms < 0.0 || m < ms)) ms = m;
    }
    record(&r, btx, btz, se, ms);
    if (ms > 0.0 && (bse_ms < 0.0 || ms < bse_ms)) { bse_ms = ms; bse = se; }
  }
  r.tile_x = btx;
  r.tile_z = btz;
  r.sort_every = bse;
  r.ms_per_step = bse_ms > 0.0 ? bse_ms : best;
  r.cached = 0;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    g_cache[key] = r;
  }
  *out = r;
  return PIC_OK;
}

}  // namespace

extern "C" int pic_autotune_window(const pic_config* cfg, const pic_plasma* plasma, const pic_laser* laser,
                                   int warm, int steps, pic_alloc_fn alloc, pic_free_fn free_fn, void* alloc_user,
                                   void* cuda_stream, pic_tune_result* out) {
  return tune(cfg, plasma, laser, warm, steps, false, alloc, free_fn, alloc_user, cuda_stream, out);
}

extern "C" int pic_autotune(const pic_config* cfg, const pic_plasma* plasma, const pic_laser* laser, int steps,
                            pic_alloc_fn alloc, pic_free_fn free_fn, void* alloc_user, void* cuda_stream,
                            pic_tune_result* out) {
  return tune(cfg, plasma, laser, 4, steps, true, alloc, free_fn, alloc_user, cuda_stream, out);
}
