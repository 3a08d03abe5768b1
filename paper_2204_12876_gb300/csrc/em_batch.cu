// em_batch.cu -- the batched form: many maps updated by one kernel sequence.
//
// Every kernel of the update already works on a list of maps and clouds (the
// device descriptor), so a batch is the same launch sequence as one em_update
// with more maps in the descriptor: per-point kernels span all clouds of all
// maps, per-cell kernels walk the tiles of all maps' cells.  With EM_BATCH_GRAPH the
// sequence becomes a graph once per descriptor slot (grids sized from the batch
// capacities), replayed by one cudaGraphLaunch.
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "em.h"
#include "em_host.h"
#include "em_internal.cuh"

using namespace em;

namespace {

constexpr int kSlots = 3;

#define EB_TRY(expr, what)                                  \
  do {                                                      \
    cudaError_t _e = (expr);                                \
    if (_e != cudaSuccess) return map_record_error((what), _e); \
  } while (0)

bool tuning_ok(const em_tuning& t) {
  const int r = t.ray_group, f = t.fuse_chunk;
  return (r == 1 || r == 2 || r == 4 || r == 8 || r == 16 || r == 32) && f >= 64 && f <= 1024 && (f & (f - 1)) == 0 &&
         t.big_thresh >= 32 && t.big_thresh <= 1023;
}

}  // namespace

struct em_batch {
  int device = 0;
  int32_t max_maps = 0, max_clouds = 0, max_cells = 0;
  int64_t max_points = 0;
  uint32_t flags = 0;
  BatchCtl* bctl = nullptr;
  SumTable tab{};         // for maps beyond kFlatCells; no slots when max_cells allows none
  long long wait_budget = 0;  // SM clock cycles of EM_PERSIST_WAIT_MS
  size_t desc_bytes = 0;
  unsigned char* desc_host = nullptr;
  unsigned char* desc_dev = nullptr;
  cudaEvent_t ev[kSlots] = {};
  int slot = 0;
  bool dirty = false;  // a launch failed half way through an update: bctl must be cleared
  em_tuning tune{8, 512, 256};
  cudaGraphExec_t graph[kSlots] = {};
  UpdateKind graph_kind[kSlots] = {};
  // host scratch for grouping
  std::vector<int> first_of, order, map_of;
  std::vector<em_map*> uniq;
  // per-kernel profiling
  bool prof = false;
  bool prof_pending = false;
  cudaEvent_t pev[2 * EM_PROF_SLOTS] = {};
  bool pused[EM_PROF_SLOTS] = {};
  double pms[EM_PROF_SLOTS] = {};
  int64_t pn[EM_PROF_SLOTS] = {};
};

namespace {

int prof_collect(em_batch* b) {
  if (!b->prof_pending) return EM_OK;
  b->prof_pending = false;
  for (int k = 0; k < EM_PROF_SLOTS; ++k) {
    if (!b->pused[k]) continue;
    b->pused[k] = false;
    EB_TRY(cudaEventSynchronize(b->pev[2 * k + 1]), "cudaEventSynchronize");
    float ms = 0.f;
    EB_TRY(cudaEventElapsedTime(&ms, b->pev[2 * k], b->pev[2 * k + 1]), "cudaEventElapsedTime");
    b->pms[k] += ms;
    b->pn[k] += 1;
  }
  return EM_OK;
}

// The update's kernels on a stream, with events around each when the batch is profiling.
cudaError_t launch_sequence(em_batch* b, const Sequence& q, const BatchDev* bd, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < q.n && e == cudaSuccess; ++i) {
    const int slot = q.k[i].slot;
    if (b->prof && !b->pused[slot]) cudaEventRecord(b->pev[2 * slot], s);  // a slot spans its launches
    e = run(q.k[i], &bd, s);
    if (b->prof) {
      cudaEventRecord(b->pev[2 * slot + 1], s);
      b->pused[slot] = true;
      b->prof_pending = true;
    }
  }
  return e;
}

struct Prepared {
  const BatchDev* bd = nullptr;
  int slot = -1;
  int64_t points = 0;
  int32_t n_maps = 0;
  int64_t cells = 0;  // padded size of the cell space
  UpdateKind kind{};
};

// Check the pairs and group them by map (b->uniq, b->map_of; points per map).
int group(em_batch* b, em_map* const* maps, const em_cloud* clouds, int32_t count, std::vector<int64_t>* map_pts,
          int64_t* points) {
  if (!maps || !clouds || count < 1) return EM_ERR_INVALID_ARG;
  if (count > b->max_clouds) return EM_ERR_CAPACITY;
  b->uniq.clear();
  b->map_of.assign(count, -1);
  for (int i = 0; i < count; ++i) {
    const em_cloud& c = clouds[i];
    if (!maps[i] || c.n < 0 || (c.stride != 3 && c.stride != 4) || (c.n > 0 && !c.points) || !word_aligned(c.points))
      return EM_ERR_INVALID_ARG;
    for (int k = 0; k < 12; ++k)
      if (!std::isfinite(c.pose[k])) return EM_ERR_INVALID_ARG;
    if (map_device(maps[i]) != b->device) return EM_ERR_INVALID_ARG;
    int u = -1;
    for (size_t j = 0; j < b->uniq.size(); ++j)
      if (b->uniq[j] == maps[i]) { u = (int)j; break; }
    if (u < 0) {
      if ((int)b->uniq.size() >= b->max_maps) return EM_ERR_CAPACITY;
      if (map_cells(maps[i]) > b->max_cells) return EM_ERR_CAPACITY;
      u = (int)b->uniq.size();
      b->uniq.push_back(maps[i]);
    }
    b->map_of[i] = u;
  }
  map_pts->assign(b->uniq.size(), 0);
  int64_t total = 0;
  for (int i = 0; i < count; ++i) {
    (*map_pts)[b->map_of[i]] += clouds[i].n;
    total += clouds[i].n;
  }
  if (total > b->max_points) return EM_ERR_CAPACITY;
  *points = total;
  return EM_OK;
}

// Does an update of `count` clouds of the one map m run as em_update does?  With
// nothing to upload and grids of its own size instead of the capacity's; a served
// request at 2,000 updates/s (a lightly loaded server's batches are of one map)
// took 67 us through the graph, em_update 49.
bool runs_alone(const em_batch* b, const em_map* m, const em_tuning& tune, int32_t count, int64_t total) {
  return count <= kDescClouds && tune.ray_group == kValueGroup && !b->prof && !(b->flags & EM_BATCH_PERSISTENT) &&
         !(map_flags(m) & EM_F_TRACE) && map_has_room(m, total);
}

// A failed update may have stopped between its launches.
void mark_dirty(em_batch* b) {
  b->dirty = true;
  for (em_map* m : b->uniq) map_set_dirty(m);
}

// Build the descriptor of the grouped pairs in the next slot and upload it.
int prepare(em_batch* b, const em_cloud* clouds, int32_t count, const std::vector<int64_t>& map_pts, int64_t total,
            const em_tuning& tune, cudaStream_t s, Prepared* out) {
  const int nm = (int)b->uniq.size();
  if (b->dirty) EB_TRY(cudaMemsetAsync(b->bctl, 0, sizeof(BatchCtl), s), "clear scratch");
  if (b->dirty && b->tab.slots) EB_TRY(table_clear(b->tab, s), "clear scratch");
  b->dirty = false;
  for (em_map* m : b->uniq) {
    int rc = map_clean(m, s);
    if (rc) return rc;
  }
  const int slot = b->slot;
  b->slot = (b->slot + 1) % kSlots;
  EB_TRY(cudaEventSynchronize(b->ev[slot]), "cudaEventSynchronize");
  unsigned char* hb = b->desc_host + (size_t)slot * b->desc_bytes;
  unsigned char* db = b->desc_dev + (size_t)slot * b->desc_bytes;
  BatchDev* bd = reinterpret_cast<BatchDev*>(hb);
  MapDev* md = reinterpret_cast<MapDev*>(hb + sizeof(BatchDev));
  CloudDev* cd = reinterpret_cast<CloudDev*>(hb + sizeof(BatchDev) + (size_t)b->max_maps * sizeof(MapDev));
  memset(bd, 0, sizeof(BatchDev));
  UpdateKind kind{};
  kind.ray_group = tune.ray_group;
  kind.persistent = (b->flags & EM_BATCH_PERSISTENT) != 0;
  int64_t cells = 0, flat_cells = 0, items = 0;
  for (int u = 0; u < nm; ++u) {
    md[u] = map_begin_update(b->uniq[u], map_pts[u]);
    md[u].cell_begin = cells;
    cells += pad_tile(map_cells(b->uniq[u]));
    if (map_cells(b->uniq[u]) > kFlatCells) {
      md[u].acc = b->tab.acc;
      md[u].rej = b->tab.rej;
      md[u].cnt = md[u].wall > 0 ? b->tab.cnt : nullptr;
      md[u].keys = b->tab.keys;
      kind.slots = b->tab.slots;
      kind.ext = true;
    } else {
      flat_cells += pad_tile(map_cells(b->uniq[u]));
    }
    md[u].ibegin = items;
    items += (int64_t)md[u].IW * md[u].IH;
    const UpdateKind k = map_kind(b->uniq[u], tune.ray_group);
    kind.ray |= k.ray;
    kind.drift |= k.drift;
    kind.wall |= k.wall;
    kind.ext |= k.ext;
    kind.stencils |= k.stencils;
  }
  // clouds ordered by map (stable), so each map's points are contiguous
  int ci = 0;
  int64_t begin = 0;
  for (int u = 0; u < nm; ++u)
    for (int i = 0, first = 1; i < count; ++i) {
      if (b->map_of[i] != u) continue;
      if (first) {  // the map's first cloud's sensor origin, as in em_update_multi
        md[u].z_ref = clouds[i].pose[11];
        md[u].ref_x = clouds[i].pose[3];
        md[u].ref_y = clouds[i].pose[7];
      }
      first = 0;
      CloudDev& c = cd[ci++];
      memset(&c, 0, sizeof(c));
      c.pts = clouds[i].points;
      c.n = clouds[i].n;
      c.begin = begin;
      c.stride = clouds[i].stride;
      c.map = u;
      for (int r = 0; r < 3; ++r) {
        for (int k = 0; k < 3; ++k) c.R[r * 3 + k] = clouds[i].pose[r * 4 + k];
        c.t[r] = clouds[i].pose[r * 4 + 3];
      }
      begin += clouds[i].n;
    }
  bd->n_maps = nm;
  bd->n_clouds = count;
  bd->n_points = total;
  bd->maps = reinterpret_cast<const MapDev*>(db + sizeof(BatchDev));
  bd->clouds = reinterpret_cast<const CloudDev*>(db + sizeof(BatchDev) + (size_t)b->max_maps * sizeof(MapDev));
  bd->n_cells = cells;
  for (int u = 0; u < nm; ++u)
    if (md[u].keys || !use_flags(flat_cells, total)) md[u].touched = nullptr;
  bd->n_items = items;
  bd->ctl = b->bctl;
  if (kind.slots) bd->tab = b->tab;
  bd->passes = (kind.wall || kind.drift ? kPassPre : 0u) | (kind.ray || kind.drift ? kPassCells : 0u);
  bd->wait_budget = b->wait_budget;
  // upload header + maps, and the clouds at their fixed offset
  cudaError_t e = cudaMemcpyAsync(db, hb, sizeof(BatchDev) + (size_t)nm * sizeof(MapDev), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(db + sizeof(BatchDev) + (size_t)b->max_maps * sizeof(MapDev), cd,
                        (size_t)count * sizeof(CloudDev), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) {
    for (int u = 0; u < nm; ++u) map_undo_update(b->uniq[u], map_pts[u]);
    return map_record_error("upload batch descriptor", e);
  }
  out->bd = reinterpret_cast<const BatchDev*>(db);
  out->slot = slot;
  out->points = total;
  out->n_maps = nm;
  out->cells = cells;
  out->kind = kind;
  return EM_OK;
}

void finish(em_batch* b, const Prepared& p, cudaStream_t s) {
  for (size_t u = 0; u < b->uniq.size(); ++u) map_end_update(b->uniq[u], s, 0);
  cudaEventRecord(b->ev[p.slot], s);
}

int run_graph(em_batch* b, const Prepared& p, cudaStream_t s) {
  if (!b->graph[p.slot] || !(b->graph_kind[p.slot] == p.kind)) {
    if (b->graph[p.slot]) {
      cudaGraphExecDestroy(b->graph[p.slot]);
      b->graph[p.slot] = nullptr;
    }
    cudaGraph_t g = nullptr;
    const Sequence q = update_sequence(p.kind, b->max_points, (int64_t)b->max_maps * pad_tile(b->max_cells));
    EB_TRY(build_graph(q, p.bd, &g), "cudaGraphAddKernelNode");
    cudaGraphExec_t ex = nullptr;
    cudaError_t ie = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    EB_TRY(ie, "cudaGraphInstantiate");
    b->graph[p.slot] = ex;
    b->graph_kind[p.slot] = p.kind;
  }
  EB_TRY(cudaGraphLaunch(b->graph[p.slot], s), "cudaGraphLaunch");
  return EM_OK;
}

int set_dev(int dev) {
  int cur = -1;
  if (cudaGetDevice(&cur) != cudaSuccess || cur != dev) EB_TRY(cudaSetDevice(dev), "cudaSetDevice");
  return EM_OK;
}

void release(em_batch* b) {
  for (int i = 0; i < 2 * EM_PROF_SLOTS; ++i)
    if (b->pev[i]) cudaEventDestroy(b->pev[i]);
  for (int i = 0; i < kSlots; ++i) {
    if (b->graph[i]) cudaGraphExecDestroy(b->graph[i]);
    if (b->ev[i]) cudaEventDestroy(b->ev[i]);
  }
  cudaFree(b->bctl);
  table_free(&b->tab);
  cudaFree(b->desc_dev);
  cudaFreeHost(b->desc_host);
  delete b;
}

}  // namespace

extern "C" {

int em_wait_selftest(int device, int32_t wait_us) {
  if (wait_us < 1 || wait_us > 10 * 1000 * 1000) return EM_ERR_INVALID_ARG;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return EM_ERR_INVALID_ARG;
  int rc = set_dev(device);
  if (rc) return rc;
  unsigned long long* word = nullptr;  // nothing ever sets it
  int* flag = nullptr;
  cudaStream_t s = nullptr;
  cudaError_t e = cudaMalloc((void**)&word, sizeof(*word));
  if (e == cudaSuccess) e = cudaMalloc((void**)&flag, sizeof(*flag));
  if (e == cudaSuccess) e = cudaMemset(word, 0, sizeof(*word));
  if (e == cudaSuccess) e = cudaMemset(flag, 0, sizeof(*flag));
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = launch_wait_selftest(word, flag, wait_us, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  int timed_out = 0;
  if (e == cudaSuccess) e = cudaMemcpy(&timed_out, flag, sizeof(timed_out), cudaMemcpyDeviceToHost);
  if (s) cudaStreamDestroy(s);
  cudaFree(word);
  cudaFree(flag);
  if (e != cudaSuccess) return map_record_error("em_wait_selftest", e);
  return timed_out ? EM_ERR_TIMEOUT : EM_OK;
}

int em_batch_create(int device, int32_t max_maps, int32_t max_clouds, int64_t max_points, int32_t max_cells,
                    uint32_t flags, em_batch** out) {
  if (!out) return EM_ERR_INVALID_ARG;
  *out = nullptr;
  if (max_maps < 1 || max_maps > 65535 || max_clouds < 1 || max_points < 0 || max_points > (int64_t(1) << 31) - 1 ||
      max_cells < 1 || max_cells > (1 << 26) || (flags & ~(uint32_t)(EM_BATCH_GRAPH | EM_BATCH_PERSISTENT)))
    return EM_ERR_INVALID_ARG;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return EM_ERR_INVALID_ARG;
  int rc = set_dev(device);
  if (rc) return rc;
  em_batch* b = new (std::nothrow) em_batch();
  if (!b) return EM_ERR_OOM;
  b->device = device;
  b->max_maps = max_maps;
  b->max_clouds = max_clouds;
  b->max_points = max_points;
  b->max_cells = max_cells;
  b->flags = flags;
  b->desc_bytes = (sizeof(BatchDev) + (size_t)max_maps * sizeof(MapDev) + (size_t)max_clouds * sizeof(CloudDev) + 255) &
                  ~size_t(255);
  cudaError_t e = cudaMalloc((void**)&b->bctl, sizeof(BatchCtl));
  if (e == cudaSuccess) e = cudaMemset(b->bctl, 0, sizeof(BatchCtl));
  if (e == cudaSuccess && max_cells > kFlatCells)
    e = table_alloc(&b->tab, table_slots(std::min(max_points, (int64_t)max_maps * max_cells)), true, nullptr);
  if (e == cudaSuccess) e = cudaMalloc((void**)&b->desc_dev, b->desc_bytes * kSlots);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&b->desc_host, b->desc_bytes * kSlots);
  for (int i = 0; i < kSlots && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&b->ev[i], cudaEventDisableTiming);
  long long wait_us = EM_PERSIST_WAIT_MS * 1000ll;
  if (const char* v = getenv("EM_PERSIST_WAIT_US")) wait_us = std::max(0ll, std::min(wait_us, atoll(v)));
  b->wait_budget = clock_budget(wait_us);
  if (e != cudaSuccess) {
    release(b);
    return map_record_error("em_batch_create", e);
  }
  *out = b;
  return EM_OK;
}

int em_batch_destroy(em_batch* b) {
  if (!b) return EM_OK;
  set_dev(b->device);
  cudaDeviceSynchronize();
  release(b);
  return EM_OK;
}

int em_update_batch(em_batch* b, em_map* const* maps, const em_cloud* clouds, int32_t count, em_stream_t stream) {
  if (!b) return EM_ERR_INVALID_ARG;
  int rc = set_dev(b->device);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (b->prof) {
    rc = prof_collect(b);
    if (rc) return rc;
  }
  std::vector<int64_t> map_pts;
  int64_t total = 0;
  rc = group(b, maps, clouds, count, &map_pts, &total);
  if (rc) return rc;
  if (b->uniq.size() == 1 && runs_alone(b, b->uniq[0], b->tune, count, total))
    return map_update_one(b->uniq[0], clouds, count, total, s);
  Prepared p;
  rc = prepare(b, clouds, count, map_pts, total, b->tune, s, &p);
  if (rc) return rc;
  if ((b->flags & EM_BATCH_GRAPH) && !b->prof) {
    rc = run_graph(b, p, s);
  } else {
    cudaError_t e = launch_sequence(b, update_sequence(p.kind, p.points, p.cells), p.bd, s);
    rc = e == cudaSuccess ? EM_OK : map_record_error("batch launches", e);
  }
  if (rc) mark_dirty(b);
  finish(b, p, s);
  return rc;
}

int em_batch_profile(em_batch* b, int enable) {
  if (!b) return EM_ERR_INVALID_ARG;
  int rc = set_dev(b->device);
  if (rc) return rc;
  if (enable && !b->pev[0])
    for (int i = 0; i < 2 * EM_PROF_SLOTS; ++i) EB_TRY(cudaEventCreate(&b->pev[i]), "cudaEventCreate");
  if (!enable) {
    rc = prof_collect(b);
    if (rc) return rc;
  }
  if (enable && !b->prof)
    for (int k = 0; k < EM_PROF_SLOTS; ++k) { b->pms[k] = 0.0; b->pn[k] = 0; }
  b->prof = enable != 0;
  return EM_OK;
}

int em_batch_profile_read(em_batch* b, double* ms, int64_t* launches) {
  if (!b || !ms || !launches) return EM_ERR_INVALID_ARG;
  int rc = set_dev(b->device);
  if (rc) return rc;
  rc = prof_collect(b);
  if (rc) return rc;
  for (int k = 0; k < EM_PROF_SLOTS; ++k) {
    ms[k] = b->pms[k];
    launches[k] = b->pn[k];
  }
  return EM_OK;
}

int em_batch_set_tuning(em_batch* b, const em_tuning* t) {
  if (!b || !t || !tuning_ok(*t)) return EM_ERR_INVALID_ARG;
  b->tune = *t;
  return EM_OK;
}

int em_batch_get_tuning(const em_batch* b, em_tuning* t) {
  if (!b || !t) return EM_ERR_INVALID_ARG;
  *t = b->tune;
  return EM_OK;
}

int em_batch_autotune(em_batch* b, em_map* const* maps, const em_cloud* clouds, int32_t count, em_stream_t stream,
                      int32_t reps, em_tuning* out) {
  if (!b || !maps || !clouds || count < 1) return EM_ERR_INVALID_ARG;
  int rc = set_dev(b->device);
  if (rc) return rc;
  if (reps < 1) reps = 3;
  cudaStream_t s = (cudaStream_t)stream;
  // scratch copies of the distinct maps
  std::vector<em_map*> uniq, clones;
  std::vector<em_map*> cmaps(count);
  for (int i = 0; i < count; ++i) {
    if (!maps[i]) return EM_ERR_INVALID_ARG;
    size_t j = 0;
    while (j < uniq.size() && uniq[j] != maps[i]) ++j;
    if (j == uniq.size()) {
      em_params p = map_params(maps[i]);
      p.flags &= ~(uint32_t)EM_F_TRACE;
      em_map* c = nullptr;
      rc = em_create(&p, b->device, &c);
      if (rc) {
        for (em_map* x : clones) em_destroy(x);
        return rc;
      }
      uniq.push_back(maps[i]);
      clones.push_back(c);
    }
    cmaps[i] = clones[j];
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  auto time_one = [&](const em_tuning& t, float* ms_out) -> int {
    std::vector<float> ms;
    auto timed = [&]() -> int {
      cudaEventRecord(e1, s);
      if (cudaEventSynchronize(e1) != cudaSuccess) return EM_ERR_CUDA;
      float x = 0.f;
      cudaEventElapsedTime(&x, e0, e1);
      ms.push_back(x);
      return EM_OK;
    };
    for (int r = 0; r < reps + 1; ++r) {
      for (size_t j = 0; j < uniq.size(); ++j) {
        int c = map_copy_state(clones[j], uniq[j], s);
        if (c) return c;
      }
      Prepared p;
      std::vector<int64_t> map_pts;
      int64_t total = 0;
      int c = group(b, cmaps.data(), clouds, count, &map_pts, &total);
      // one map: each shape the way em_update_batch would run it
      const bool alone = uniq.size() == 1 && runs_alone(b, uniq[0], t, count, total);
      if (c == EM_OK && alone) c = em_reserve(clones[0], total);
      if (c == EM_OK && alone) {
        cudaEventRecord(e0, s);
        c = map_update_one(clones[0], clouds, count, total, s);
        if (c == EM_OK) c = timed();
        if (c) return c;
        continue;
      }
      if (c == EM_OK) c = prepare(b, clouds, count, map_pts, total, t, s, &p);
      if (c) return c;
      cudaEventRecord(e0, s);
      cudaError_t le = launch_sequence(b, update_sequence(p.kind, p.points, p.cells), p.bd, s);
      finish(b, p, s);
      if (le != cudaSuccess) {
        mark_dirty(b);
        return map_record_error("autotune launches", le);
      }
      c = timed();
      if (c) return c;
    }
    ms.erase(ms.begin());  // the first run warms up
    std::sort(ms.begin(), ms.end());
    *ms_out = ms[ms.size() / 2];
    return EM_OK;
  };
  em_tuning best = b->tune;
  float best_ms = 0.f;
  rc = time_one(best, &best_ms);
  const bool any_ray = [&] {
    for (em_map* m : uniq)
      if (map_params(m).ray_step > 0.f) return true;
    return false;
  }();
  for (int g : {1, 2, 4, 8, 16}) {
    if (!any_ray || rc != EM_OK) break;
    em_tuning t = best;
    t.ray_group = g;
    if (t.ray_group == best.ray_group) continue;
    float ms = 0.f;
    rc = time_one(t, &ms);
    if (rc == EM_OK && ms < best_ms) {
      best_ms = ms;
      best = t;
    }
  }
  cudaStreamSynchronize(s);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  for (em_map* x : clones) em_destroy(x);
  if (rc) return rc;
  b->tune = best;
  if (out) *out = best;
  return EM_OK;
}

}  // extern "C"
