// em_internal.cuh -- device-side descriptors and kernel launchers of libem.so.
//
// One update is a "batch": one or more maps, each with one or more clouds.
// The plain em_update is a batch of one map and one cloud.  All sizes that
// change from update to update live in device memory (BatchDev / MapDev /
// CloudDev), so the same kernels serve the plain, multi-cloud and batched
// forms, and launches can be captured in a CUDA graph.
//
// Work spaces of a batch:
//   points  the clouds of all maps concatenated (per-point kernels, 1D grid);
//   cells   the cells of all maps concatenated, each map's range padded to a
//           multiple of kTile cells, so every tile of kTile cells lies in one
//           map (per-cell kernels, 1D grid over tiles: uneven maps balance);
//   items   logical blocks of 32 x 8 cells, one warp's work in k_cells.
//
// Pipeline of one update (Section II-A of the paper: transform, height update
// and ray casting in the same iteration, then per-cell passes):
//   k_pre      only with the wall rule or the drift compensation: points per
//              cell, and the drift sums                (Section II-C, II-D)
//   k_cells    only with the ray march or the drift compensation: moves the
//              estimates by the drift, ray thresholds of the pre-update map and
//              their largest per block of 8 x 8 cells  (Section II-D, II-E)
//   k_points   per point: transform, noise variance, cell, wall rule and
//              Mahalanobis gate against the pre-update map, exact integer sums
//              into the cell's accumulator (Section II-C); then its ray, marched
//              against the pre-update thresholds       (Section II-E)
//   k_sums     only with maps beyond kFlatCells: Eq. 1/2 for the cells of the table
//   k_write    per cell: Eq. 1/2 in information form from the sums; removal of
//              penetrated cells not written recently   (Section II-C, II-E, II-F)
//   k_stencils normals, smoothing, in-painting         (Section II-A, II-I)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace em {

constexpr int kTile = 1024;  // cells per tile of the cell space
// The ray march's coarse grid: per block of kCoarse x kCoarse logical cells the
// largest ray threshold of the block (a chunk of samples whose lowest z is not
// below it cannot mark any cell).
constexpr int kCoarseShift = 3;
constexpr int kCoarse = 1 << kCoarseShift;
inline int32_t coarse_dim(int32_t cells) { return (cells + kCoarse - 1) >> kCoarseShift; }
// the grid in memory, with its rim: rows of coarse_stride(W) blocks; block (0, 0) is entry coarse_first(W)
inline int32_t coarse_stride(int32_t W) { return coarse_dim(W) + 2; }
inline int64_t coarse_size(int32_t W, int32_t H) { return (int64_t)coarse_stride(W) * (coarse_dim(H) + 2); }
inline int32_t coarse_first(int32_t W) { return coarse_stride(W) + 1; }


// per-map counters (device), in em_stats order
enum StatIdx {
  kStUpdates = 0, kStIn, kStValid, kStInMap, kStAccepted, kStRejected, kStWall, kStCellsUpdated,
  kStCleared, kStRaySamples, kStDriftPoints, kStCount
};

// per-map device control block
struct MapCtl {
  unsigned long long stats[kStCount];
  int32_t err;         // first device-side error code of this map (sticky until read)
  float drift_last;    // height error added by the last drift compensation
  int32_t pad[2];
  // drift-compensation sums (k_pre; read by k_cells, zero between updates)
  long long drift_h;           // sum of the errors' fixed-point high parts
  unsigned long long drift_l;  // ... and low parts (value h 2^27 + l, 2^-44 m units)
  unsigned long long drift_n;  // points in the sum
};

// per-batch device control block (zero between updates)
struct BatchCtl {
  int32_t next[3];           // per part, work counter of k_points: runs of at most kRayRun 32-point batches
  int32_t scattered;         // of the sampled batches of a large update, those whose points lie far apart (k_cells)
  // grid barrier of the persistent kernel (k_persist.cu): blocks done, the abort
  // flag of a barrier wait that ran out, and block tickets
  int32_t bar_done;
  int32_t bar_abort;
  unsigned long long bar_ticket;
};

// Accumulator of one cell: the exact fixed-point sums of its accepted points'
// weights and weighted heights (value h 2^27 + l each), one 32-byte sector, so
// the four words of a run of points go to L2 as one sector's reductions.  Zero
// between updates.  kAccTouched in wl: a point was accepted whose weight is
// zero in fixed point (the low parts' sum stays below 2^58).
struct __align__(32) CellAcc {
  unsigned long long wh, wl, th, tl;
};
constexpr unsigned long long kAccTouched = 1ull << 63;

// Large updates whose points come in no order go through them in parts
// (point_pass.cuh): at least kSplitPoints points, and more than half of
// kOrderSamples sampled batches scattered.
constexpr int kParts = 3;
constexpr uint32_t kSplitPoints = 1u << 20;
constexpr int kOrderSamples = 64;

// Updates of more than kFlagCells cells (all maps together) of which the points can
// touch half at most keep a flag per tile, so that clouds on a few cells of large maps
// do not cost a read of all their accumulators (64 maps of 250,000 cells, 2,000
// points each, with rays: 213 us without flags, 190 with).  In smaller updates the flags would
// be a few sectors that every warp writes: without them a raw depth image took 45 us
// instead of 49, four depth cameras 36.8 instead of 38.5; and where the points are as
// many as the cells most tiles are touched anyhow (64-map batch, 14 M points on 6.8 M
// cells: 2196 us without, 2212 with).
constexpr int64_t kFlagCells = 1 << 20;
inline bool use_flags(int64_t n_cells, int64_t n_points) { return n_cells > kFlagCells && n_cells >= 2 * n_points; }

// Maps of at most kFlatCells cells hold an accumulator per cell (up to 40 bytes a
// cell, 21 MB).  Larger ones would hold gigabytes for the few cells an update
// touches: their updates keep the sums of the cells the points fall into in a table
// of 3/2 slots per point, keyed by cell, open addressing (SumTable).  8192 x 8192
// cells with rays, after an update of 262,144 points: 3.5 GB with an accumulator
// per cell, 1.1 GB with the table.
constexpr int64_t kFlatCells = 1 << 19;
inline int64_t table_slots(int64_t cells) { return cells + cells / 2 + 1; }  // of an update that touches that many
struct SumTable {
  unsigned long long* keys;  // batch cell + 1 of the slot's cell; 0 = free.  Zero between updates, as the rest
  CellAcc* acc;              // one slot more than `slots`: it takes what finds no slot (never, by the table's size)
  uint32_t* rej;
  uint32_t* cnt;
  uint32_t slots;            // 0: no table
};

constexpr int kItemW = 32, kItemH = 8;  // k_cells: logical cells per warp item

// device-side error word value for a failed internal consistency check (EM_ERR_CUDA)
constexpr int32_t kErrInternal = -3;
// ... and for a bounded device-side wait that ran out (EM_ERR_TIMEOUT)
constexpr int32_t kErrTimeout = -4;

// point status codes (trace)
enum PointStatus : uint8_t { kPtNonFinite = 0, kPtRange = 1, kPtOutside = 2, kPtFused = 3, kPtRejected = 4, kPtWall = 5 };

struct MapDev {
  // layers, physical ring layout [py][px], px = (ix + ox) mod W
  float* h;
  float* var;       // +inf = empty cell
  int32_t* t_last;
  float* nx;        // normals (may be null)
  float* ny;
  float* nz;
  float* smooth;    // may be null
  float* inpaint;   // may be null
  float* upper;     // upper bound of the ground height (Section II-H), +inf where none; may be null
  uint32_t* mark;   // visibility marks, one bit per physical cell, zero between updates
  float* thr;       // per LOGICAL cell [iy][ix]: h - sqrt(var_eff) of the pre-update map, -inf if empty
                    // (with the upper-bound layer an empty cell's bound); k_refresh: -inf where marked
  float* cthr;      // per coarse block [by][bx] (CW x CH of them, rows CS apart, a rim of -inf blocks
                    // around them): the largest thr of its cells
  MapCtl* ctl;
  CellAcc* acc;     // per physical cell, or per slot of the table
  uint32_t* rej;    // rejected points per physical cell or slot, zero between updates
  uint32_t* cnt;    // wall rule: points per physical cell or slot, zero between updates; null without the rule
  unsigned long long* keys;  // the table's keys; null: acc, rej and cnt are per cell
  uint8_t* touched; // per tile of kTile cells: some point of this update fell into it; null when the update
                    // keeps no flags (use_flags): all tiles count as touched
  int64_t ibegin;   // this map's first item in the batch's item space (maps with the ray march or drift)
  int32_t IW, IH;   // items per row and column; 0 x 0 without the ray march and the drift compensation
  int32_t CW, CH, CS;  // coarse blocks per row and column (0 x 0 without the ray march), row stride
  int64_t cell_begin;  // this map's first cell in the batch cell space (multiple of kTile)
  int32_t W, H, ox, oy;
  float x0, y0, res, inv_res;  // inv_res = 1 / res rounded to float
  float drift_flat;    // drift compensation: flat iff previous normal n_z >= this; 0 = off
  float excl_b, excl_c, excl_tan, excl_d;  // exclusion ramp (tan of its angle); excl_d <= 0 = off
  float ovl_r2, ovl_dz, ref_x, ref_y;      // overlap clearance: radius^2, height gap, robot position
  float z_ref;         // reference height of empty cells in the fusion sums: the z of the
                       // first cloud's sensor origin (any fixed value gives the same result
                       // up to rounding; one near the points keeps the terms small)
  int32_t t_now;       // index of this update
  // method parameters
  float a0, a1, a2, var_min, min_range, max_range, k, v_out, sigma_t2, ray_step, alpha_n;
  int32_t wall, min_age;
  uint32_t flags;
};

struct CloudDev {
  const float* pts;
  int64_t n;
  int64_t begin;   // first index of this cloud in the batch point space
  int32_t stride;
  int32_t map;
  float R[9];
  float t[3];
};

struct BatchDev {
  int32_t n_maps, n_clouds;
  int64_t n_points;
  int64_t n_cells;     // padded size of the cell space
  int64_t n_items;     // k_cells items of all maps
  const MapDev* maps;
  const CloudDev* clouds;
  int32_t* tr_ix;      // trace (null unless EM_F_TRACE)
  int32_t* tr_iy;
  uint8_t* tr_status;
  BatchCtl* ctl;
  SumTable tab;        // sums of the maps with keys
  uint32_t passes;     // kPass* bits: optional passes some map of the batch needs
  long long wait_budget;  // SM clock cycles a grid barrier of the persistent kernel may wait
};
// The descriptor of an update of one map with few clouds travels as a kernel
// parameter: nothing to upload before the first kernel, and the fields are read
// from the constant bank instead of through two dependent global loads.
constexpr int kDescClouds = 8;
struct MapDesc {
  BatchDev b;
  MapDev m;
  CloudDev c[kDescClouds];
};
static_assert(sizeof(MapDesc) <= 4096, "a kernel parameter");
// What the passes see of either form.
struct MapView : BatchDev {};
__device__ __forceinline__ const BatchDev& view(const BatchDev* p) { return *p; }
__device__ __forceinline__ MapView view(const MapDesc& d) {
  MapView v;
  static_cast<BatchDev&>(v) = d.b;
  v.n_maps = 1;
  v.maps = &d.m;
  v.clouds = d.c;
  return v;
}
__device__ __forceinline__ const MapDev& map_at(const BatchDev& b, int i) { return b.maps[i]; }
__device__ __forceinline__ const MapDev& map_at(const MapView& b, int) { return b.maps[0]; }

enum : uint32_t { kPassPre = 1u, kPassCells = 2u };

// The coarse grid and the items of k_cells of a map of W x H cells.
inline void set_item_grid(MapDev& d, int32_t W, int32_t H, bool ray, bool drift) {
  d.CW = ray ? coarse_dim(W) : 0;
  d.CH = ray ? coarse_dim(H) : 0;
  d.CS = ray ? coarse_stride(W) : 0;
  d.IW = ray || drift ? (W + kItemW - 1) / kItemW : 0;
  d.IH = ray || drift ? (H + kItemH - 1) / kItemH : 0;
}

inline int64_t pad_tile(int64_t cells) { return (cells + kTile - 1) / kTile * kTile; }
// The kernels read points and layers as 4-byte words: a buffer that does not
// start on a 4-byte boundary is refused on the host (it would fault on the device).
inline bool word_aligned(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

// number of SMs of the current device (cached)
int sm_count();

// ---- the kernels of an update
// One launch: every kernel of an update takes the descriptor -- its device
// address, or the descriptor itself (MapDesc) -- and k_points also the part, so a
// launch is plain data that can go to a stream or become a graph node.
struct Launch {
  const void* fn;  // null: nothing to launch
  unsigned grid, block;
  size_t smem;
  bool coop;
  int slot;        // EM_PROF_* slot of its time
  const char* name;
  int part;        // k_points: the part of the points
};
// What an update needs: the optional passes some map of it uses.
struct UpdateKind {
  int32_t ray_group;  // samples per chunk and lanes per marched chunk
  bool ray;
  bool drift;
  bool wall;
  bool ext;           // some map uses the exclusion area, the upper-bound layer or the table of sums
  bool persistent;
  bool by_value;      // the kernels take a MapDesc
  uint32_t slots;     // of the update's table; 0: every map has its own accumulators
  uint32_t stencils;  // EM_F_* of the per-cell filters
  bool operator==(const UpdateKind& o) const {
    return ray_group == o.ray_group && ray == o.ray && drift == o.drift && wall == o.wall && ext == o.ext &&
           persistent == o.persistent && by_value == o.by_value && stencils == o.stencils && slots == o.slots;
  }
};
constexpr int kMaxLaunches = 16;
struct Sequence {
  int n = 0;
  Launch k[kMaxLaunches];
  void add(const Launch& l) {
    if (l.fn) k[n++] = l;
  }
};
// The launches of an update in stream order; grids for n_points points and
// n_cells (padded) cells, which bound what the descriptor holds.
#define EM_KERNEL(k, by_value) ((by_value) ? (const void*)&k<MapDesc> : (const void*)&k<const BatchDev*>)
constexpr int kValueGroup = 8;  // the one ray_group built for MapDesc
Sequence update_sequence(const UpdateKind& k, int64_t n_points, int64_t n_cells);
// desc: the kernel's descriptor argument (a const BatchDev* or a MapDesc)
cudaError_t run(const Launch& l, const void* desc, cudaStream_t s);

// Launch a kernel that begins with begin_after_previous(): it may start while the
// kernel before it on the stream ends.
template <class... P, class... A>
cudaError_t launch_after(void (*k)(P...), int grid, int block, cudaStream_t s, A... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, P(args)...);
}
// The sequence as a chain of kernel nodes.
cudaError_t build_graph(const Sequence& q, const BatchDev* b, cudaGraph_t* out);

Launch pre_launch(int64_t n_points, bool ext, bool by_value);
Launch cells_launch(int64_t n_cells, bool by_value);
Launch refresh_launch(int64_t n_cells, bool by_value);
Launch points_launch(int64_t n_points, int group, bool ray, bool ext, int part, bool by_value);
Launch sums_launch(uint32_t slots, bool by_value);
Launch write_launch(int64_t n_cells, bool by_value);
// The whole update but the drift compensation and the stencils (points per
// cell, thresholds, points, write) in one cooperative launch with grid
// barriers; barrier waits are bounded by the descriptor's wait_budget.  fn is
// null when the device cannot run it.
Launch persist_launch(int group, bool ext);
long long clock_budget(long long us);  // SM clock cycles of that many microseconds
Launch stencils_launch(int64_t n_cells, bool by_value);

// ---- launchers of the other kernels (each returns cudaGetLastError())
// The bounded wait of the persistent kernel on a word that nothing sets: one
// block, budget wait_us; *timed_out (device memory) becomes 1 when it runs out.
cudaError_t launch_wait_selftest(const unsigned long long* word, int* timed_out, int wait_us, cudaStream_t s);
cudaError_t launch_shift_clear(const MapDev& m, int32_t dx, int32_t dy, cudaStream_t s);
cudaError_t launch_layers_out(const MapDev& m, uint32_t mask, float* dst, cudaStream_t s);
// Layer reads of up to kMaxReadJobs maps in one launch (the jobs are the kernel parameters).
constexpr int kMaxReadJobs = 32;
struct ReadJob {
  MapDev m;
  uint32_t mask;
  float* dst;
};
struct ReadJobs {
  int n;
  ReadJob job[kMaxReadJobs];
};
cudaError_t launch_layers_out_multi(const ReadJobs& jobs, cudaStream_t s);
static_assert(sizeof(ReadJobs) <= 32000, "the read jobs must fit a kernel's parameter block");
cudaError_t launch_layers_in(const MapDev& m, uint32_t mask, const float* src, cudaStream_t s);
cudaError_t launch_fill_map(const MapDev& m, cudaStream_t s);

// ---- small device helpers shared by the kernels

// Start of every kernel of an update: it may have been launched while the
// kernel before it on the stream still ran (launch.cu), so it waits for that
// one's end and memory, then lets the next one be launched in the same way.
// What the kernel before may have written -- layers, and the caller's points --
// was not read-only while this one ran, so no kernel reads with __ldg.
__device__ __forceinline__ void begin_after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
}

__device__ __forceinline__ int32_t clamp_floor(float q) {
  float f = floorf(q);
  f = fminf(fmaxf(f, -1.0e9f), 1.0e9f);
  return (int32_t)f;
}

// physical index of logical cell (ix, iy), both in range
__device__ __forceinline__ int32_t phys_index(const MapDev& m, int32_t ix, int32_t iy) {
  int32_t px = ix + m.ox;
  px -= (px >= m.W) ? m.W : 0;
  int32_t py = iy + m.oy;
  py -= (py >= m.H) ? m.H : 0;
  return py * m.W + px;
}

// logical coordinates of physical cell p
__device__ __forceinline__ void logical_of(const MapDev& m, int32_t p, int32_t& lx, int32_t& ly) {
  const int32_t py = p / m.W, px = p - py * m.W;
  lx = px - m.ox;
  lx += (lx < 0) ? m.W : 0;
  ly = py - m.oy;
  ly += (ly < 0) ? m.H : 0;
}

// effective variance of a cell at update t_now (lazy time variance)
__device__ __forceinline__ float var_eff(const MapDev& m, float var, int32_t t_last) {
  return __fmaf_rn(m.sigma_t2, (float)(m.t_now - t_last), var);
}

// index of the cloud that holds batch point g (clouds sorted by begin)
__device__ __forceinline__ int find_cloud(const CloudDev* cl, int n_clouds, int64_t g) {
  int lo = 0, hi = n_clouds - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (cl[mid].begin <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The same, tried first on cloud `hint` (the cloud of the caller's previous
// point: passes walk the point space in order, so it usually holds g); an
// empty cloud never holds g, so the answer is the search's.
__device__ __forceinline__ int find_cloud(const CloudDev* cl, int n_clouds, int64_t g, int hint) {
  if ((unsigned)hint < (unsigned)n_clouds && cl[hint].begin <= g && g < cl[hint].begin + cl[hint].n) return hint;
  return find_cloud(cl, n_clouds, g);
}

// Whether this update's points go in parts (k_cells has run).
__device__ __forceinline__ bool in_parts(const BatchDev& b) {
  return b.n_points >= kSplitPoints && b.ctl->scattered > kOrderSamples / 2;
}

// Where the sums of batch cell g are, for the lanes that want it: the cell's slot
// of the table, taken now when the cell has none yet.  At most as many cells as the
// table is sized for, so a free slot is always found; should it not be, the sums go
// to the spare slot and the map reports an internal error.  Multiplicative hashing
// (Knuth, The Art of Computer Programming 3, 6.4), linear probing.  Called by whole
// warps, with a warp's vote per probe: with a loop per lane a warp whose lanes needed
// different numbers of probes stayed split in two for the rest of its batch (points
// and rays of 262,144 points on 1,000,000 cells: 76 us, 54 as it is).  No look before the
// exchange: a line that SMs of both dies read while others write it costs more (no
// rays: 29 us with a look, 26 without).
__device__ __forceinline__ uint32_t slot_of(bool want, const SumTable& t, const MapDev& m, int64_t g) {
  const unsigned long long key = (unsigned long long)g + 1ull;
  uint32_t s = (uint32_t)(((key * 0x9E3779B97F4A7C15ull) >> 32) * t.slots >> 32);
  for (uint32_t i = 0; i < t.slots && __any_sync(0xffffffffu, want); ++i) {
    if (want) {
      const unsigned long long k = atomicCAS(t.keys + s, 0ull, key);
      if (k == 0ull || k == key) want = false;
      else s = s + 1 == t.slots ? 0 : s + 1;
    }
  }
  if (want) {
    atomicCAS(&m.ctl->err, 0, kErrInternal);
    s = t.slots;
  }
  return s;
}

// index of the map whose cell range holds batch cell g (maps sorted by cell_begin)
__device__ __forceinline__ int find_map_cell(const MapDev* maps, int n_maps, int64_t g) {
  int lo = 0, hi = n_maps - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (maps[mid].cell_begin <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The blocks that share a pass: a kernel's own grid, or the blocks of the
// persistent kernel (k_persist.cu) that the pass runs on.
struct Grid {
  int bid, nb;
};
__device__ __forceinline__ Grid own_grid() { return Grid{(int)blockIdx.x, (int)gridDim.x}; }

// Iterate over the tiles of the cell space: for each tile the map it lies in
// (block-uniform) and the tile's first physical cell.  body(m, map, p0, count).
template <class V, class F>
__device__ __forceinline__ void for_each_tile(const V& b, Grid gr, F body) {
  const int64_t n_tiles = b.n_cells / kTile;
  for (int64_t t = gr.bid; t < n_tiles; t += gr.nb) {
    const int64_t g0 = t * kTile;
    const int mi = find_map_cell(b.maps, b.n_maps, g0);
    const MapDev& m = map_at(b, mi);
    const int64_t p0 = g0 - m.cell_begin;
    const int32_t ncell = m.W * m.H;
    if (p0 >= ncell) continue;  // padding at the end of a map
    const int32_t cnt = (int32_t)(ncell - p0 < kTile ? ncell - p0 : kTile);
    body(m, mi, (int32_t)p0, cnt);
  }
}
}  // namespace em
