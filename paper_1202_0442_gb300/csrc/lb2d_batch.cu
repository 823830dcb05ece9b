// lb2d_batch.cu -- many independent lattices advanced by one persistent
// launch (lb_batch_*): the tile lists, the autotuner and its cache, and the
// captured graph of iterations.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "lb2d.h"
#include "lbapi.h"
#include "lbbatch.h"
#include "lbctx.h"
#include "lbint.h"

using namespace lbk;

// ======================================================================
// batched lattices
// ======================================================================

struct lb_batch {
  std::vector<lb_ctx *> ctxs;
  int device = 0;
  cudaStream_t stream = nullptr;
  int storage = ST_FP32;
  std::string err;
  uint64_t launches = 0;
  BatchLat *d_lat = nullptr;
  int4 *d_tiles = nullptr;
  unsigned int *d_counters = nullptr;
  unsigned int *d_tick = nullptr;
  bool odd = false;  // the last call ended with an odd number of launches
  std::vector<BatchLat> h_lat;
  // two iterations per launch (k_march_batch): the lattices' descriptors for
  // either parity and the tasks; mtasks 0: not used
  MarchBatchLat *d_mlat = nullptr;
  int4 *d_mtasks = nullptr;
  int mtasks = 0;
  int shape = 0, dynamic = 1, order = 1;
  int ntiles = 0, grid = 0;
  cudaGraphExec_t gexec = nullptr;
  int graph_steps = 0, graph_launches = 0;
  // graphs are captured and replayed on a private stream (the caller's may
  // be the legacy default stream, which cannot be captured), fenced to the
  // caller's stream by events
  cudaStream_t gstream = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  int fail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    err = buf;
    return code;
  }
};

namespace {

int batch_cuda(lb_batch *b, cudaError_t e, const char *what) {
  return b->fail(LB_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define BCK(call)                                            \
  do {                                                       \
    cudaError_t e_ = (call);                                 \
    if (e_ != cudaSuccess) return batch_cuda(b, e_, #call);  \
  } while (0)

void drop_graph(lb_batch *b) {
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  b->gexec = nullptr;
  b->graph_steps = 0;
}

// tile list for the current shape and order: 0 = lattice by lattice,
// 1 = round robin over lattices, 2 = largest lattices first
int build_tiles(lb_batch *b) {
  const int TX = batch_shape_tx(b->shape), TY = batch_shape_ty(b->shape);
  std::vector<std::vector<int4>> per(b->ctxs.size());
  for (size_t l = 0; l < b->ctxs.size(); l++) {
    const lb_ctx *c = b->ctxs[l];
    for (int y0 = 0; y0 < c->ny; y0 += TY)
      for (int x0 = 0; x0 < c->nx; x0 += TX) per[l].push_back(make_int4((int)l, x0, y0, 0));
  }
  std::vector<int> idx(b->ctxs.size());
  for (size_t l = 0; l < idx.size(); l++) idx[l] = (int)l;
  if (b->order == 2)
    std::stable_sort(idx.begin(), idx.end(), [&](int a, int c) { return per[a].size() > per[c].size(); });
  std::vector<int4> tiles;
  if (b->order == 1) {
    size_t maxn = 0;
    for (auto &v : per) maxn = std::max(maxn, v.size());
    for (size_t k = 0; k < maxn; k++)
      for (int l : idx)
        if (k < per[l].size()) tiles.push_back(per[l][k]);
  } else {
    for (int l : idx) tiles.insert(tiles.end(), per[l].begin(), per[l].end());
  }
  if (b->d_tiles) cudaFree(b->d_tiles);
  b->d_tiles = nullptr;
  BCK(cudaMalloc((void **)&b->d_tiles, tiles.size() * sizeof(int4)));
  BCK(cudaMemcpyAsync(b->d_tiles, tiles.data(), tiles.size() * sizeof(int4), cudaMemcpyHostToDevice, b->stream));
  b->ntiles = (int)tiles.size();
  int sms = 0;
  BCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device));
  int occ = batch_occupancy(b->storage, b->shape);
  b->grid = std::max(1, std::min(b->ntiles, sms * std::max(occ, 1)));
  drop_graph(b);
  return LB_OK;
}

// the tasks of k_march_batch, if the batch suits it: one rounding and
// momentum mode, and enough nodes in strips that fill their lanes (below, the few
// rows per warp are a serial chain, as in march_ok).  Time over that of one
// iteration per launch, FP32 | exact momentum | FP16.  Lanes filled to 0.75 or more:
// 2 lattices of 480^2 (460 K) 1.06 | 1.08 | 0.85, 720^2 0.91 | 0.94 | 0.73, 22 of
// 100 x 300 (660 K) 0.83 | 0.82 | 0.68, 24 uneven ones (2.2 M) 0.70 | 0.76 | 0.75.
// Less: 40 of 128^2 (655 K) 1.10 | 1.20 | 1.00, 66 of 122^2 (982 K) 1.15 | 1.20 | 1.08, 80 of 128^2
// (1.3 M) 0.99 | 1.12 | 0.95, 132 of 122^2 (2.0 M) 0.81 | 0.89 | 0.97; in 16 bits a
// little more than one wave of warps (66 of 122^2: 1.3) is the only loss.
int build_march(lb_batch *b) {
  int64_t nodes = 0, slots = 0;
  for (const lb_ctx *c : b->ctxs) {
    if (c->pm != b->ctxs[0]->pm || c->sr != b->ctxs[0]->sr) return LB_OK;
    nodes += (int64_t)c->nx * c->ny;
    slots += (int64_t)((c->nx + MARCH_COLS - 1) / MARCH_COLS) * 64 * c->ny;
  }
  const bool fp32 = b->storage == ST_FP32, full = nodes * 4 >= slots * 3;
  if (nodes < (!fp32 ? 320000 : full ? 500000 : 1900000) || nodes * 5 < slots * 3) return LB_OK;
  int sms = 0;
  BCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device));
  // rows per warp: two or more waves of 16 warps per SM, where that leaves 8
  // rows, and at most 24 (256 lattices: flat from 16 to 48, 8 rows 7 % slower)
  const int rows = (int)std::min<int64_t>(24, std::max<int64_t>(8, slots / 64 / (2 * 16 * sms)));
  std::vector<int4> tasks;
  for (size_t k = 0; k < b->ctxs.size(); k++) {
    const lb_ctx *c = b->ctxs[k];
    const int sw = march_strip_width(c->nx), n = (c->ny + rows - 1) / rows, seg = (c->ny + n - 1) / n;
    for (int y = 0; y < c->ny; y += seg)
      for (int x = 0; x < c->nx; x += sw) tasks.push_back(make_int4((int)k, x, y, seg));
  }
  if (!full && (int)tasks.size() > 16 * sms && (int)tasks.size() * 2 < 3 * 16 * sms) return LB_OK;
  BCK(cudaMalloc((void **)&b->d_mlat, 2 * b->ctxs.size() * sizeof(MarchBatchLat)));
  BCK(cudaMalloc((void **)&b->d_mtasks, tasks.size() * sizeof(int4)));
  BCK(cudaMemcpyAsync(b->d_mtasks, tasks.data(), tasks.size() * sizeof(int4), cudaMemcpyHostToDevice, b->stream));
  b->mtasks = (int)tasks.size();
  return LB_OK;
}

// refresh the per-lattice descriptors (a context may have been advanced on
// its own since the last batch call)
int sync_descs(lb_batch *b) {
  bool dirty = b->h_lat.empty();
  if (dirty) b->h_lat.resize(b->ctxs.size());
  for (size_t l = 0; l < b->ctxs.size(); l++) {
    lb_ctx *c = b->ctxs[l];
    BatchLat L{};
    L.nx = c->g.nx;
    L.ny = c->g.ny;
    L.pitch = c->g.pitch;
    L.mw = c->g.mw;
    L.plane = c->g.plane;
    L.buf[0] = c->fbuf[0];
    L.buf[1] = c->fbuf[1];
    L.cur = c->cur;
    L.mask = c->mask;
    L.nbc = c->nbc;
    L.rho_ref = (float)c->rho_ref[0];
    L.scale = c->scale;
    L.inv_scale = c->inv_scale;
    L.tau = (float)c->tau[0];
    L.omega = (float)(1.0 / c->tau[0]);
    L.pm = c->pm ? 1 : 0;
    L.sr = c->sr ? 1 : 0;
    L.fx = (float)c->fave[0][0];
    L.fy = (float)c->fave[0][1];
    L.ax = (float)c->acc[0][0];
    L.ay = (float)c->acc[0][1];
    if (memcmp(&L, &b->h_lat[l], sizeof L)) {
      b->h_lat[l] = L;
      dirty = true;
    }
  }
  if (!dirty) return LB_OK;
  BCK(cudaMemcpyAsync(b->d_lat, b->h_lat.data(), b->h_lat.size() * sizeof(BatchLat), cudaMemcpyHostToDevice,
                      b->stream));
  if (b->mtasks) {
    const size_t n = b->ctxs.size();
    std::vector<MarchBatchLat> m(2 * n);
    for (size_t k = 0; k < 2 * n; k++) {
      const int parity = k >= n;
      const BatchLat &L = b->h_lat[k - parity * n];
      MarchLat &l = m[k].l;
      const int in = (L.cur + parity) & 1;
      l.fin = L.buf[in];
      l.fout = L.buf[1 - in];
      l.nbc = L.nbc;
      l.nx = L.nx;
      l.ny = L.ny;
      l.pitch = L.pitch;
      l.plane = (unsigned)L.plane;
      l.rho_ref = L.rho_ref;
      l.scale = L.scale;
      l.inv_scale = L.inv_scale;
      l.tau = L.tau;
      l.omega = L.omega;
      l.keep = 1.0f - L.omega;
      l.wa = 1.0f / 9.0f;
      l.wd = 1.0f / 36.0f;
      l.fx = L.fx;
      l.fy = L.fy;
      l.ax = L.ax;
      l.ay = L.ay;
      m[k].sw = march_strip_width(L.nx);
    }
    BCK(cudaMemcpyAsync(b->d_mlat, m.data(), m.size() * sizeof(MarchBatchLat), cudaMemcpyHostToDevice, b->stream));
  }
  return LB_OK;
}

BatchLaunch launch_desc(lb_batch *b) {
  BatchLaunch L{};
  L.lat = b->d_lat;
  L.tiles = b->d_tiles;
  L.ntiles = b->ntiles;
  L.grid = b->grid;
  L.shape = b->shape;
  L.dynamic = b->dynamic;
  L.counters = b->d_counters;
  L.tick = b->d_tick;
  return L;
}

// LB_DEBUG_POISON on member contexts: NaN in the buffers the launch of
// this parity writes (every member's next population buffer)
int batch_poison(lb_batch *b, int parity) {
  for (lb_ctx *c : b->ctxs) {
    if (!(c->debug & LB_DEBUG_POISON)) continue;
    const int out = 1 - ((c->cur + parity) & 1);
    const cudaError_t e = cudaMemsetAsync(c->fbuf[out], 0xff, 9 * c->g.plane * storage_bytes(c->storage), b->stream);
    if (e != cudaSuccess) return batch_cuda(b, e, "poison");
  }
  return LB_OK;
}

bool batch_poisoned(const lb_batch *b) {
  for (const lb_ctx *c : b->ctxs)
    if (c->debug & LB_DEBUG_POISON) return true;
  return false;
}

// n iterations: by twos an even number of times where k_march_batch serves
// (a launch switches every lattice's buffers once), the others one by one
int batch_launch(lb_batch *b, int parity0, int n, bool march, bool poison, cudaStream_t s, int *launched) {
  const BatchLaunch L = launch_desc(b);
  MarchBatch M{};
  M.tasks = b->d_mtasks;
  M.ntasks = b->mtasks;
  M.pm = b->ctxs[0]->pm;
  M.sr = b->ctxs[0]->sr;
  M.counters = b->d_counters;
  M.tick = b->d_tick;
  const int pairs = march && b->mtasks ? n / 4 * 2 : 0, total = n - pairs;
  for (int k = 0; k < total; k++) {
    const int parity = (parity0 + k) & 1;
    if (poison) {
      const int rc = batch_poison(b, parity);
      if (rc != LB_OK) return rc;
    }
    M.lat = b->d_mlat + (parity ? b->ctxs.size() : 0);
    if ((k < pairs ? launch_march_batch(b->storage, M, parity, s) : launch_batch(b->storage, L, parity, s)) < 0)
      return batch_cuda(b, cudaGetLastError(), "batch launch");
  }
  *launched = total;
  return LB_OK;
}

int batch_direct(lb_batch *b, int parity0, int n, bool march = true) {
  int launched = 0;
  const int rc = batch_launch(b, parity0, n, march, batch_poisoned(b), b->stream, &launched);
  b->launches += (uint64_t)launched;
  return rc;
}

// before launches that start with parity 0: after an odd number of launches
// its work counter is cleared (the last launch, of parity 0 too, used it) and
// takes up the launch number
int batch_start(lb_batch *b) {
  if (!b->odd) return LB_OK;
  BCK(cudaMemsetAsync(b->d_counters, 0, sizeof(unsigned int), b->stream));
  BCK(cudaMemcpyAsync(b->d_tick, b->d_tick + 1, sizeof(unsigned int), cudaMemcpyDeviceToDevice, b->stream));
  b->odd = false;
  return LB_OK;
}

void batch_advance(lb_batch *b, int n) {
  for (lb_ctx *c : b->ctxs) {
    c->cur = (c->cur + n) & 1;
    c->t += n;
    c->fields_valid = false;
  }
  b->h_lat.clear();
}

constexpr int GRAPH_STEPS = 20;  // iterations per captured graph (a multiple of four)

int ensure_graph(lb_batch *b) {
  if (b->gexec) return LB_OK;
  if (!b->gstream) {
    BCK(cudaStreamCreateWithFlags(&b->gstream, cudaStreamNonBlocking));
    BCK(cudaEventCreateWithFlags(&b->ev_in, cudaEventDisableTiming));
    BCK(cudaEventCreateWithFlags(&b->ev_out, cudaEventDisableTiming));
  }
  cudaGraph_t graph = nullptr;
  BCK(cudaStreamBeginCapture(b->gstream, cudaStreamCaptureModeThreadLocal));
  const int bad = batch_launch(b, 0, GRAPH_STEPS, true, false, b->gstream, &b->graph_launches) != LB_OK;
  cudaError_t e = cudaStreamEndCapture(b->gstream, &graph);
  if (bad || e != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return batch_cuda(b, e != cudaSuccess ? e : cudaGetLastError(), "graph capture");
  }
  e = cudaGraphInstantiate(&b->gexec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) return batch_cuda(b, e, "cudaGraphInstantiate");
  b->graph_steps = GRAPH_STEPS;
  return LB_OK;
}

}  // namespace

extern "C" {

int lb_batch_create(lb_ctx *const *ctxs, int n, lb_batch **out) {
  if (!out || !ctxs || n < 1) return LB_E_ARG;
  *out = nullptr;
  lb_batch *b = new (std::nothrow) lb_batch();
  if (!b) return LB_E_NOMEM;
  for (int k = 0; k < n; k++) {
    lb_ctx *c = ctxs[k];
    int rc = LB_OK;
    if (!c) rc = LB_E_ARG;
    else if (c->nc != 1 || c->qs || !c->open.empty() || c->sc || c->ads[0] || c->bstyle != 0 || c->rank >= 0)
      rc = c->fail(LB_E_UNSUPPORTED, "batched lattices are periodic single-component noslip lattices with body forces");
    else {
      for (int s = 0; s < c->nc && rc == LB_OK; s++)
        if (!c->painted_f[s] && !c->state_set[s]) rc = c->fail(LB_E_ORDER, "lattice %d has no initial state", k);
      if (rc == LB_OK) rc = commit(c);
    }
    if (rc == LB_OK && k > 0 && (c->device != ctxs[0]->device || c->stream != ctxs[0]->stream ||
                                 c->storage != ctxs[0]->storage))
      rc = LB_E_ARG;
    if (rc != LB_OK) {
      delete b;
      return rc;
    }
    b->ctxs.push_back(c);
  }
  b->device = ctxs[0]->device;
  b->stream = ctxs[0]->stream;
  b->storage = ctxs[0]->storage;
  if (cudaSetDevice(b->device) != cudaSuccess || cudaMalloc((void **)&b->d_lat, n * sizeof(BatchLat)) != cudaSuccess ||
      cudaMalloc((void **)&b->d_counters, 2 * sizeof(unsigned int)) != cudaSuccess ||
      cudaMemsetAsync(b->d_counters, 0, 2 * sizeof(unsigned int), b->stream) != cudaSuccess ||
      cudaMalloc((void **)&b->d_tick, 2 * sizeof(unsigned int)) != cudaSuccess ||
      cudaMemsetAsync(b->d_tick, 0, 2 * sizeof(unsigned int), b->stream) != cudaSuccess) {
    lb_batch_destroy(b);
    return LB_E_CUDA;
  }
  if (build_tiles(b) != LB_OK || build_march(b) != LB_OK) {
    lb_batch_destroy(b);
    return LB_E_CUDA;
  }
  *out = b;
  return LB_OK;
}

int lb_batch_destroy(lb_batch *b) {
  if (!b) return LB_E_ARG;
  cudaSetDevice(b->device);
  cudaStreamSynchronize(b->stream);
  drop_graph(b);
  if (b->gstream) cudaStreamSynchronize(b->gstream);
  if (b->gstream) cudaStreamDestroy(b->gstream);
  if (b->ev_in) cudaEventDestroy(b->ev_in);
  if (b->ev_out) cudaEventDestroy(b->ev_out);
  if (b->d_lat) cudaFree(b->d_lat);
  if (b->d_tiles) cudaFree(b->d_tiles);
  if (b->d_counters) cudaFree(b->d_counters);
  if (b->d_tick) cudaFree(b->d_tick);
  if (b->d_mlat) cudaFree(b->d_mlat);
  if (b->d_mtasks) cudaFree(b->d_mtasks);
  delete b;
  return LB_OK;
}

const char *lb_batch_last_error(const lb_batch *b) { return b ? b->err.c_str() : "no batch"; }

int lb_batch_launch_count(const lb_batch *b, uint64_t *out) {
  if (!b || !out) return LB_E_ARG;
  *out = b->launches;
  return LB_OK;
}

int lb_batch_iteration(lb_batch *b, int Nt, int use_graph) {
  if (!b) return LB_E_ARG;
  NvtxRange range("lb_batch_iteration");
  if (Nt < 0) return b->fail(LB_E_ARG, "Nt must be >= 0");
  BCK(cudaSetDevice(b->device));
  int rc = sync_descs(b);
  if (rc != LB_OK) return rc;
  if (Nt > 0) {
    rc = batch_start(b);
    if (rc != LB_OK) return rc;
    b->odd = Nt & 1;
  }
  int done = 0;
  // poisoned members run without the graph (the poisoning is not captured)
  if (use_graph && !batch_poisoned(b)) {
    rc = ensure_graph(b);
    if (rc != LB_OK) return rc;
    if (Nt >= b->graph_steps) {
      BCK(cudaEventRecord(b->ev_in, b->stream));
      BCK(cudaStreamWaitEvent(b->gstream, b->ev_in, 0));
      while (Nt - done >= b->graph_steps) {
        BCK(cudaGraphLaunch(b->gexec, b->gstream));
        b->launches += (uint64_t)b->graph_launches;
        done += b->graph_steps;
      }
      BCK(cudaEventRecord(b->ev_out, b->gstream));
      BCK(cudaStreamWaitEvent(b->stream, b->ev_out, 0));
    }
  }
  rc = batch_direct(b, done & 1, Nt - done);
  if (rc != LB_OK) return rc;
  batch_advance(b, Nt);
  return LB_OK;
}

int lb_batch_autotune(lb_batch *b, const char *cache_json) {
  if (!b) return LB_E_ARG;
  BCK(cudaSetDevice(b->device));
  // cache key: device name, storage and the lattice shapes
  cudaDeviceProp prop;
  BCK(cudaGetDeviceProperties(&prop, b->device));
  uint64_t hsh = 1469598103934665603ULL;
  for (lb_ctx *c : b->ctxs) {
    hsh = (hsh ^ (uint64_t)c->nx) * 1099511628211ULL;
    hsh = (hsh ^ (uint64_t)c->ny) * 1099511628211ULL;
  }
  char key[512];
  snprintf(key, sizeof key, "%s|st%d|n%zu|%016llx", prop.name, b->storage, b->ctxs.size(), (unsigned long long)hsh);
  std::string cache;
  if (cache_json) {
    FILE *fp = fopen(cache_json, "rb");
    if (fp) {
      char buf[4096];
      size_t n;
      while ((n = fread(buf, 1, sizeof buf, fp)) > 0) cache.append(buf, n);
      fclose(fp);
    }
    size_t p = cache.find(std::string("\"") + key + "\"");
    if (p != std::string::npos) {
      int sh, dy, od;
      const char *q = strchr(cache.c_str() + p, '{');
      if (q && sscanf(q, "{\"shape\": %d, \"dynamic\": %d, \"order\": %d", &sh, &dy, &od) == 3 && sh >= 0 &&
          sh < BATCH_SHAPES) {
        b->shape = sh;
        b->dynamic = dy;
        b->order = od;
        return build_tiles(b);
      }
    }
  }
  // keep the lattices' states: time on them, then put the states back
  int rc = sync_descs(b);
  if (rc == LB_OK) rc = batch_start(b);
  if (rc != LB_OK) return rc;
  std::vector<void *> saved(b->ctxs.size(), nullptr);
  std::vector<size_t> sizes(b->ctxs.size());
  for (size_t l = 0; l < b->ctxs.size(); l++) {
    lb_ctx *c = b->ctxs[l];
    sizes[l] = (size_t)9 * c->g.plane * storage_bytes(c->storage);
    BCK(cudaMalloc(&saved[l], sizes[l]));
    BCK(cudaMemcpyAsync(saved[l], c->fbuf[c->cur], sizes[l], cudaMemcpyDeviceToDevice, b->stream));
  }
  cudaEvent_t e0, e1;
  BCK(cudaEventCreate(&e0));
  BCK(cudaEventCreate(&e1));
  float best = 1e30f;
  int bs = 0, bd = 1, bo = 1;
  const int reps = 6;
  for (int sh = 0; sh < BATCH_SHAPES; sh++)
    for (int dy = 0; dy < 2; dy++)
      for (int od = 0; od < 3; od++) {
        if (dy && od == 0) continue;  // dynamic hand-out makes lattice order moot
        b->shape = sh;
        b->dynamic = dy;
        b->order = od;
        rc = build_tiles(b);
        if (rc != LB_OK) return rc;
        rc = batch_direct(b, 0, 2, false);
        if (rc != LB_OK) return rc;
        BCK(cudaEventRecord(e0, b->stream));
        rc = batch_direct(b, 0, reps, false);
        if (rc != LB_OK) return rc;
        BCK(cudaEventRecord(e1, b->stream));
        BCK(cudaEventSynchronize(e1));
        float ms = 0;
        BCK(cudaEventElapsedTime(&ms, e0, e1));
        if (ms < best) {
          best = ms;
          bs = sh;
          bd = dy;
          bo = od;
        }
      }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  // an even number of launches per candidate leaves buf[cur] the input
  for (size_t l = 0; l < b->ctxs.size(); l++) {
    lb_ctx *c = b->ctxs[l];
    BCK(cudaMemcpyAsync(c->fbuf[c->cur], saved[l], sizes[l], cudaMemcpyDeviceToDevice, b->stream));
  }
  BCK(cudaStreamSynchronize(b->stream));
  for (void *p : saved) cudaFree(p);
  b->shape = bs;
  b->dynamic = bd;
  b->order = bo;
  rc = build_tiles(b);
  if (rc != LB_OK) return rc;
  if (cache_json) {
    std::string entry = std::string("\"") + key + "\": {\"shape\": " + std::to_string(bs) +
                        ", \"dynamic\": " + std::to_string(bd) + ", \"order\": " + std::to_string(bo) +
                        ", \"ms_per_iter\": " + std::to_string(best / reps) + "}";
    std::string body;
    size_t l = cache.find('{'), r = cache.rfind('}');
    if (l != std::string::npos && r != std::string::npos && r > l) body = cache.substr(l + 1, r - l - 1);
    while (!body.empty() && isspace((unsigned char)body.back())) body.pop_back();
    std::string outs = "{" + body + (body.empty() ? "\n  " : ",\n  ") + entry + "\n}\n";
    FILE *fp = fopen(cache_json, "wb");
    if (fp) {
      fwrite(outs.data(), 1, outs.size(), fp);
      fclose(fp);
    }
  }
  return LB_OK;
}

}  // extern "C"
