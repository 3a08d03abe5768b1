// em_noalloc.cu -- em_update_noalloc: one map update that allocates no memory.
//
// Some callers cannot call cudaMalloc at update time: a real-time control loop
// that forbids allocation after start-up (an allocation can block on the
// driver for milliseconds), or a host framework whose own caching allocator
// has already claimed the device memory.  For them this entry point runs the
// same kernels as em_update (gate + sums + ray march, fusion, removal) on map
// layers the caller owns, and keeps every piece of scratch memory in one
// file-scope __device__ array of fixed size.  The call's
// descriptor goes to the device as a kernel parameter (no host buffer, no
// copy), and its only other preparation is a memset of the scratch.
//
// Limits: at most kMaxCells cells per map and kMaxPoints points per update
// (about 2.9 MiB of scratch, held by every GPU that loads the library until the
// process exits).  Every call shares the array and it keeps the last call's
// contents; the call clears what must start at zero.  Calls whose GPU work
// overlaps (e.g. on two streams) race on the array.
#include <cuda_runtime.h>
#include <string.h>

#include <cmath>
#include <cstddef>
#include <mutex>

#include "em.h"
#include "em_host.h"
#include "em_internal.cuh"

using namespace em;

namespace {

constexpr int32_t kMaxCells = EM_NOALLOC_MAX_CELLS;
constexpr int64_t kMaxPoints = EM_NOALLOC_MAX_POINTS;
constexpr int kMaxCloudsNA = EM_NOALLOC_MAX_CLOUDS;

constexpr size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

static_assert(kMaxCloudsNA <= kDescClouds, "the descriptor travels as a kernel parameter");

// Scratch layout.  The part that must start at zero (control blocks, marks and
// the accumulators of this call's cells) is contiguous, so one memset
// as long as the map is clears it.
constexpr size_t kOffCtl = 0;
constexpr size_t kOffBCtl = kOffCtl + up256(sizeof(MapCtl));
constexpr size_t kOffZero = kOffBCtl + up256(sizeof(BatchCtl));  // the map's part of the zeroed scratch
struct Layout {
  size_t mark, rej, cnt, acc, thr, cthr, end;
};
// coarse: blocks of the coarse grid
constexpr Layout layout(size_t cells, size_t coarse) {
  Layout o{};
  o.mark = kOffZero;
  o.rej = o.mark + up256((cells + 31) / 32 * sizeof(uint32_t));
  o.cnt = o.rej + up256(cells * sizeof(uint32_t));
  o.acc = o.cnt + up256(cells * sizeof(uint32_t));
  o.thr = o.acc + up256(cells * sizeof(CellAcc));  // end of the zeroed part
  o.cthr = o.thr + up256(cells * sizeof(float));
  o.end = o.cthr + up256(coarse * sizeof(float));
  return o;
}
// coarse entries of a map of at most kMaxCells cells: (W/8 + 3)(H/8 + 3) <= kMaxCells/64 + 3 (W + H)/8 + 9,
// and W + H <= kMaxCells + 1
static_assert(kMaxCells <= kFlagCells, "no tile flags");
constexpr size_t kMaxCoarse = (size_t)kMaxCells / 64 + 3 * ((size_t)kMaxCells + 1) / 8 + 10;
constexpr size_t kScratchBytes = layout(kMaxCells, kMaxCoarse).end;

constexpr int kMaxDevices = 64;
std::mutex g_mu;
unsigned char* g_addr[kMaxDevices] = {};

}  // namespace

// The scratch itself.  In host code this name is only a stand-in for the
// device array: its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

namespace {

int na_status(cudaError_t e, const char* what) {
  return e == cudaSuccess ? EM_OK : map_record_error(what, e);
}

// Device address of the scratch on the current device, looked up once per
// device with that device current.
int scratch_address(int dev, unsigned char** out) {
  if (dev < 0 || dev >= kMaxDevices) return EM_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) return na_status(e == cudaSuccess ? cudaErrorInvalidSymbol : e, "cudaGetSymbolAddress");
    g_addr[dev] = static_cast<unsigned char*>(p);
  }
  *out = g_addr[dev];
  return EM_OK;
}

bool na_params_ok(const em_params* p) {
  if (!p || p->width < 1 || p->height < 1 || p->width > (1 << 22) || p->height > (1 << 22)) return false;
  if (!(std::isfinite(p->resolution) && p->resolution > 0.f)) return false;
  const float f[] = {p->noise_a0, p->noise_a1, p->noise_a2, p->var_min, p->min_range, p->mahalanobis_k,
                     p->outlier_variance, p->time_variance, p->ray_step, p->cleanup_normal_thresh};
  for (float v : f)
    if (!std::isfinite(v)) return false;
  return p->var_min > 0.f && !std::isnan(p->max_range) && p->max_range >= p->min_range &&
         p->outlier_variance >= 0.f && p->time_variance >= 0.f && p->ray_step >= 0.f &&
         p->wall_num_thresh >= 0 && p->cleanup_min_age >= 0 && std::isfinite(p->drift_flatness) &&
         p->drift_flatness >= 0.f && p->drift_flatness <= 1.f &&
         !(p->flags & EM_F_UPPER);  // the upper-bound layer is not one of the caller's layers here
}

}  // namespace

extern "C" int em_update_noalloc(const em_params* params, int64_t shift_x, int64_t shift_y, int32_t t_now,
                                 float* h, float* var, int32_t* t_last, const float* nx, const float* ny,
                                 const float* nz, const em_cloud* clouds, int32_t n_clouds, em_stream_t stream) {
  if (!na_params_ok(params) || !h || !var || !t_last || !clouds || n_clouds < 1 || t_now < 1)
    return EM_ERR_INVALID_ARG;
  if (!word_aligned(h) || !word_aligned(var) || !word_aligned(t_last) || !word_aligned(nx) || !word_aligned(ny) ||
      !word_aligned(nz))
    return EM_ERR_INVALID_ARG;
  if ((params->cleanup_normal_thresh > 0.f || params->drift_flatness > 0.f) && (!nx || !ny || !nz))
    return EM_ERR_INVALID_ARG;
  if ((int64_t)params->width * params->height > kMaxCells || n_clouds > kMaxCloudsNA) return EM_ERR_CAPACITY;
  int64_t total = 0;
  for (int i = 0; i < n_clouds; ++i) {
    const em_cloud& c = clouds[i];
    if (c.n < 0 || (c.stride != 3 && c.stride != 4) || (c.n > 0 && !c.points) || !word_aligned(c.points))
      return EM_ERR_INVALID_ARG;
    for (int k = 0; k < 12; ++k)
      if (!std::isfinite(c.pose[k])) return EM_ERR_INVALID_ARG;
    total += c.n;
  }
  if (total > kMaxPoints) return EM_ERR_CAPACITY;

  int dev = 0;
  int rc = na_status(cudaGetDevice(&dev), "cudaGetDevice");
  if (rc) return rc;
  unsigned char* base = nullptr;
  rc = scratch_address(dev, &base);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  const int32_t W = params->width, H = params->height, ncell = W * H;

  // descriptor, built here and handed to every kernel by value
  MapDesc desc;
  memset(&desc, 0, sizeof(desc));
  BatchDev* b = &desc.b;
  MapDev* m = &desc.m;
  CloudDev* cd = desc.c;
  m->h = h;
  m->var = var;
  m->t_last = t_last;
  m->nx = const_cast<float*>(nx);
  m->ny = const_cast<float*>(ny);
  m->nz = const_cast<float*>(nz);
  set_item_grid(*m, W, H, params->ray_step > 0.f, params->drift_flatness > 0.f);
  const Layout lay = layout((size_t)ncell, m->CW ? (size_t)coarse_size(W, H) : 0);
  m->mark = reinterpret_cast<uint32_t*>(base + lay.mark);
  m->rej = reinterpret_cast<uint32_t*>(base + lay.rej);
  if (params->wall_num_thresh > 0) m->cnt = reinterpret_cast<uint32_t*>(base + lay.cnt);
  m->acc = reinterpret_cast<CellAcc*>(base + lay.acc);
  m->thr = reinterpret_cast<float*>(base + lay.thr);
  m->cthr = reinterpret_cast<float*>(base + lay.cthr) + coarse_first(W);
  m->ctl = reinterpret_cast<MapCtl*>(base + kOffCtl);
  m->cell_begin = 0;
  m->z_ref = clouds[0].pose[11];
  m->W = W;
  m->H = H;
  const double r = (double)params->resolution;
  m->x0 = (float)(r * ((double)shift_x - 0.5 * W));
  m->y0 = (float)(r * ((double)shift_y - 0.5 * H));
  m->res = params->resolution;
  m->inv_res = (float)(1.0 / (double)params->resolution);
  m->t_now = t_now;
  m->a0 = params->noise_a0; m->a1 = params->noise_a1; m->a2 = params->noise_a2; m->var_min = params->var_min;
  m->min_range = params->min_range; m->max_range = params->max_range; m->k = params->mahalanobis_k;
  m->v_out = params->outlier_variance; m->sigma_t2 = params->time_variance; m->ray_step = params->ray_step;
  m->alpha_n = params->cleanup_normal_thresh; m->wall = params->wall_num_thresh;
  m->min_age = params->cleanup_min_age;
  m->drift_flat = params->drift_flatness;
  m->excl_b = params->excl_b; m->excl_c = params->excl_c; m->excl_d = params->excl_d;
  m->excl_tan = (float)std::tan((double)params->excl_theta);
  m->ovl_r2 = params->overlap_radius * params->overlap_radius; m->ovl_dz = params->overlap_dz;
  m->ref_x = clouds[0].pose[3];
  m->ref_y = clouds[0].pose[7];
  int64_t begin = 0;
  for (int i = 0; i < n_clouds; ++i) {
    cd[i].pts = clouds[i].points;
    cd[i].n = clouds[i].n;
    cd[i].begin = begin;
    cd[i].stride = clouds[i].stride;
    cd[i].map = 0;
    for (int row = 0; row < 3; ++row) {
      for (int k = 0; k < 3; ++k) cd[i].R[row * 3 + k] = clouds[i].pose[row * 4 + k];
      cd[i].t[row] = clouds[i].pose[row * 4 + 3];
    }
    begin += clouds[i].n;
  }
  b->n_maps = 1;
  b->n_clouds = n_clouds;
  b->n_points = total;
  b->n_cells = pad_tile(ncell);
  b->n_items = (int64_t)m->IW * m->IH;
  b->ctl = reinterpret_cast<BatchCtl*>(base + kOffBCtl);

  rc = na_status(cudaMemsetAsync(base + kOffCtl, 0, lay.thr - kOffCtl, s), "cudaMemsetAsync");
  if (rc) return rc;
  const int64_t cells = pad_tile(ncell);
  UpdateKind kind = params_kind(*params, kValueGroup);
  kind.stencils = 0;  // not the per-cell filters
  kind.by_value = true;
  const Sequence q = update_sequence(kind, total, cells);
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < q.n && e == cudaSuccess; ++i) e = run(q.k[i], &desc, s);
  return na_status(e, "em_update_noalloc launch");
}
