// point_pass.cuh -- the device passes over the points (k_point.cu):
//
//   pre_pass     points per cell for the wall rule, drift-compensation sums
//   points_pass  every point once: transform, variance, cell, wall rule and gate
//                against the pre-update state, exact sums into the cell's
//                accumulator; then the point's ray, marched against the
//                pre-update thresholds with an exact chunk test
//
// Each pass runs on the blocks of a Grid: its own kernel's, or the persistent
// kernel's (k_persist.cu).
#pragma once

#include "em_point.cuh"

namespace em {

constexpr int kPointThreads = 256;
constexpr int kPointWarps = kPointThreads / 32;
constexpr int kRayRun = 8;  // batches per take from the work counter, at most
constexpr uint32_t kMinSpan = 8;

// Large updates whose points come in no order go through them in parts, the
// first ones small: between them k_refresh takes the marked cells out of the
// thresholds and the coarse grid, so the later parts skip what the earlier ones
// have decided (64-map batch, 14 M points: 4.15 -> 2.35 ms).  Points in a
// sensor's order go in one part: their march is cheap, and parts break its
// locality (32-robot round 601 -> 689 us).  Part i holds the places
// part_first(i) .. part_first(i + 1) - 1 of every 32 batches.
__device__ __forceinline__ uint32_t part_first(int i) { return i <= 0 ? 0u : i == 1 ? 2u : i == 2 ? 8u : 32u; }

// Block-contiguous partition of the point space into chunks of whole warps.
__device__ __forceinline__ void block_range(int64_t n, Grid gr, int64_t& beg, int64_t& end) {
  int64_t per = (n + gr.nb - 1) / gr.nb;
  per = (per + 31) & ~int64_t(31);
  beg = (int64_t)gr.bid * per;
  end = beg + per < n ? beg + per : n;
}

// Add a block's, warp's or lane's drift-compensation sums to the map's.
__device__ __forceinline__ void drift_add(const MapDev& m, long long h, unsigned long long l,
                                          unsigned long long n) {
  atomicAdd(reinterpret_cast<unsigned long long*>(&m.ctl->drift_h), (unsigned long long)h);
  atomicAdd(&m.ctl->drift_l, l);
  atomicAdd(&m.ctl->drift_n, n);
}

struct PreSmem {
  float4 stage[kPointWarps][24];
  int map;
  long long h[kPointWarps];
  unsigned long long l[kPointWarps], n[kPointWarps];
};

// Before the thresholds and the points: for maps with the wall rule the points
// of every cell (valid and in the map, before any rejection); for maps with
// drift compensation (Section II-D) the errors of the points in flat cells
// that hold an estimate (previous normal n_z >= drift_flatness; a NaN normal is
// not flat), summed exactly per map.
template <bool kExt, class V>
__device__ __forceinline__ void pre_pass(const V& b, Grid gr, PreSmem& S) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t beg, end;
  block_range(b.n_points, gr, beg, end);
  int dmap = -1;
  long long dh = 0;
  unsigned long long dl = 0, dn = 0;
  int hint = -1;
  for (int64_t wbase = beg + warp * 32; wbase < end; wbase += kPointThreads) {
    const int c0 = find_cloud(b.clouds, b.n_clouds, wbase, hint);
    hint = c0;
    const CloudDev& cl0 = b.clouds[c0];
    const MapDev& m0 = map_at(b, cl0.map);
    if (wbase + 32 <= cl0.begin + cl0.n && m0.drift_flat <= 0.f && !m0.cnt) continue;  // nothing for a whole warp
    float px, py, pz;
    const int ci = load_warp_points(b, wbase, end, S.stage[warp], px, py, pz, hint);
    const int64_t g = wbase + lane;
    const CloudDev& c = b.clouds[ci];
    const MapDev& m = map_at(b, c.map);
    const PointGeom pg = point_geom<kExt>(m, c, px, py, pz);
    const bool inm = g < end && pg.in_range && in_map(m, pg.ix, pg.iy);
    const int32_t key = inm ? phys_index(m, pg.ix, pg.iy) : 0;
    // one count per run of lanes in the same cell
    int head, len;
    key_runs(inm && m.cnt ? (unsigned long long)(uint32_t)c.map << 32 | (uint32_t)key : ~0ull, head, len);
    const bool counts = inm && m.cnt && lane == head;
    uint32_t q = (uint32_t)key;
    if (kExt && b.tab.slots) {
      const uint32_t s = slot_of(counts && m.keys, b.tab, m, m.cell_begin + key);
      if (m.keys) q = s;
    }
    if (counts) atomicAdd(&m.cnt[q], (uint32_t)len);
    if (inm && m.drift_flat > 0.f) {
      // the three loads are independent: all in flight at once
      const float var = m.var[key], nz = m.nz[key], hc = m.h[key];
      if (isfinite(var) && nz >= m.drift_flat) {
        if (c.map != dmap) {
          if (dmap >= 0) drift_add(map_at(b, dmap), dh, dl, dn);
          dmap = c.map;
          dh = 0;
          dl = dn = 0;
        }
        const Fix e = to_fix(__fsub_rn(pg.z, hc));
        dh += e.h;
        dl += e.l;
        ++dn;
      }
    }
  }
  // One atomic triple per block when the block's sums all belong to one map (the
  // usual case): every block adding to the same three words of that map would
  // otherwise queue at one L2 slice.  Else per lane.
  if (threadIdx.x == 0) S.map = -1;
  __syncthreads();
  if (dn) atomicMax(&S.map, dmap);
  __syncthreads();
  const int bm = S.map;
  if (bm < 0) {  // block-uniform: no drift sums
    __syncthreads();  // the shared memory is free again
    return;
  }
  if (__syncthreads_and(dn == 0 || dmap == bm)) {
    for (int o = 16; o > 0; o >>= 1) {
      dh += __shfl_xor_sync(kFull, dh, o);
      dl += __shfl_xor_sync(kFull, dl, o);
      dn += __shfl_xor_sync(kFull, dn, o);
    }
    if (lane == 0) {
      S.h[warp] = dh;
      S.l[warp] = dl;
      S.n[warp] = dn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      long long th = 0;
      unsigned long long tl = 0, tn = 0;
      for (int w = 0; w < kPointWarps; ++w) {
        th += S.h[w];
        tl += S.l[w];
        tn += S.n[w];
      }
      drift_add(map_at(b, bm), th, tl, tn);
    }
  } else if (dmap >= 0 && dn) {
    drift_add(map_at(b, dmap), dh, dl, dn);
  }
  __syncthreads();  // the shared memory is free again
}

// ---- the points' sums

// A warp's finished runs on their way to the accumulators: lanes 4 j .. 4 j + 3
// add the four words of one run, so a warp-wide reduction touches 8 sectors,
// not 32 (12.6 M runs into 64 maps of 106 k cells in random order: 251 us
// against 390 us with a lane per run and 739 us with an array per word).
struct AccStage {
  CellAcc sum[32];
  CellAcc* dst[32];
};

// Gate the warp's points against their cells' pre-update state and add them to
// the accumulators: runs of equal cells in consecutive lanes are first reduced
// by a segmented scan of the exact sums.  Every lane takes part; returns the
// lane's status (meaningful where inm).
template <bool kExt, class V>
__device__ __forceinline__ uint8_t add_points(const V& b, const MapDev& m, int map, bool one_map, bool inm, uint32_t p,
                                              float z, float d, AccStage& A) {
  const int lane = threadIdx.x & 31;
  Fix fw{0, 0u}, ft{0, 0u};
  uint8_t st = kPtOutside;
  uint32_t q = p;  // where the cell's sums are
  if (kExt && b.tab.slots) {  // the first lane of a run looks its slot up
    const bool keyed = inm && m.keys;
    int head, len;
    key_runs(keyed ? (unsigned long long)(m.cell_begin + p) : ~0ull, head, len);
    const uint32_t s = __shfl_sync(kFull, slot_of(keyed && lane == head, b.tab, m, m.cell_begin + p), head);
    if (keyed) q = s;
  }
  if (inm) {
    const float var = m.var[p], h = m.h[p];  // the loads are independent: all in flight at once
    const int32_t tl = m.t_last[p];
    const int32_t cnt = m.cnt ? (int32_t)m.cnt[q] : 0;
    const bool valid = isfinite(var);
    const float ve = valid ? var_eff(m, var, tl) : 0.f;
    const float vp = point_variance(m, d);
    const float dz = __fsub_rn(z, h);
    if (m.cnt && valid && cnt > m.wall && z < h) {
      st = kPtWall;
    } else if (valid && m.k > 0.f && __fmul_rn(dz, dz) > __fmul_rn(__fmul_rn(m.k, m.k), __fadd_rn(ve, vp))) {
      // |z - h| / sqrt(sigma_m^2 + sigma_p^2) > k  <=>  (z - h)^2 > k^2 (sigma_m^2 + sigma_p^2)  (k > 0)
      st = kPtRejected;
    } else {
      st = kPtFused;
      const float wgt = __frcp_rn(vp);
      fw = to_fix(wgt);
      ft = to_fix(__fmul_rn(wgt, valid ? dz : __fsub_rn(z, m.z_ref)));
    }
  }
  // a segmented inclusive scan over the runs, as many steps as the longest run
  // needs; within a run of at most 32 lanes the 27-bit low parts and the counts
  // (accepted | rejected << 16) fit 32 bits
  uint32_t nn = st == kPtFused ? 1u : st == kPtRejected ? (1u << 16) : 0u;
  const uint32_t tag = inm ? q : 0xffffffffu;
  const uint32_t prev = __shfl_up_sync(kFull, tag, 1);  // (every lane takes part in the shuffles)
  bool first = lane == 0 || prev != tag;
  if (!one_map) {
    const int before = __shfl_up_sync(kFull, map, 1);
    first = first || before != map;
  }
  const unsigned heads = __ballot_sync(kFull, first);
  const int head = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
  const bool tail = inm && (lane == 31 || (heads >> (lane + 1)) & 1u);
  const int maxrun = (int)__reduce_max_sync(kFull, inm ? (unsigned)(lane - head + 1) : 1u);
  long long wh = fw.h, th = ft.h;
  uint32_t wl = fw.l, tl = ft.l;
  for (int o = 1; o < maxrun; o <<= 1) {
    const long long awh = __shfl_up_sync(kFull, wh, o), ath = __shfl_up_sync(kFull, th, o);
    const uint32_t awl = __shfl_up_sync(kFull, wl, o), atl = __shfl_up_sync(kFull, tl, o);
    const uint32_t an = __shfl_up_sync(kFull, nn, o);
    if (lane - o >= head) {
      wh += awh;
      th += ath;
      wl += awl;
      tl += atl;
      nn += an;
    }
  }
  // the run's last lane holds its sums
  if (tail) {
    if (m.touched) m.touched[q / kTile] = 1;  // every writer stores the same (maps with keys have no flags)
    if (nn >> 16) atomicAdd(&m.rej[q], nn >> 16);
    if ((nn & 0xffffu) && (wh | (long long)wl) == 0) atomicOr(&m.acc[q].wl, kAccTouched);
  }
  const bool add = tail && (nn & 0xffffu);
  const unsigned am = __ballot_sync(kFull, add);
  const int runs = __popc(am);
  if (add) {
    const int k = __popc(am & ((1u << lane) - 1u));
    A.sum[k] = CellAcc{(unsigned long long)wh, wl, (unsigned long long)th, tl};
    A.dst[k] = m.acc + q;
  }
  __syncwarp();
  for (int k = lane >> 2; k < runs; k += 8)
    atomicAdd(reinterpret_cast<unsigned long long*>(A.dst[k]) + (lane & 3),
              reinterpret_cast<const unsigned long long*>(&A.sum[k])[lane & 3]);
  __syncwarp();
  return st;
}

// Statistics of the points: a warp counts for the map its batches lie in, one
// counter per lane, and adds the counters to the map's when the map changes.
enum PointStat { kPsValid = 0, kPsInMap, kPsAccepted, kPsRejected, kPsWall, kPsSamples, kPointStats };
__device__ __forceinline__ int stat_of(int k) {
  return k == kPsValid      ? kStValid
         : k == kPsInMap    ? kStInMap
         : k == kPsAccepted ? kStAccepted
         : k == kPsRejected ? kStRejected
         : k == kPsWall     ? kStWall
                            : kStRaySamples;
}
template <class V>
__device__ __forceinline__ void add_counts(const V& b, int map, unsigned long long v) {
  const int lane = threadIdx.x & 31;
  if (map >= 0 && lane < kPointStats && v) atomicAdd(&map_at(b, map).ctl->stats[stat_of(lane)], v);
}

// ---- the rays

// Narrow [lo, hi] (metres along the ray) to where the track o + (s/d) v stays
// inside [a0, a1); false when it never does.  An estimate (the sample range
// gets 1 mm + 1 step of slack and every sample is tested exactly), so a fast
// division does: its 2-ulp error is micrometres at tens of metres.
__device__ __forceinline__ bool slab(float o, float v, float d, float a0, float a1, float& lo, float& hi) {
  if (v == 0.f) return o >= a0 && o < a1;
  const float dv = __fdividef(d, v);
  const float sa = (a0 - o) * dv;
  const float sb = (a1 - o) * dv;
  lo = fmaxf(lo, fminf(sa, sb));
  hi = fminf(hi, fmaxf(sa, sb));
  return true;
}

// Per-ray set-up, made by one lane and read by the lanes that test and march
// the ray's chunks.  Sample k lies at q = a + k b in coarse-block units (x, y:
// an eighth of the position in cells, an exact scaling) and at z = az + k bz,
// i.e. the track o + (k step / d) (R p_s) measured from the map corner.
// Samples per ray are capped at 2^24 - 1, so the float sample index is exact.
constexpr int32_t kMaxRayK = (1 << 24) - 1;

struct RaySetup {
  float ax, bx, ay, by, az, bz;
  float vx, vy, vz, d;  // for the Eq. 4 guard
  int32_t ix, iy, k_lo, n, map;
  int32_t cn;           // samples per chunk
};

// floor(8 t) -- the cell -- and floor(t) -- the block -- of a position in block
// units by one add rounded down: t + 1.5 2^20 lands where the float spacing is
// 1/8 (t + 1.5 2^23: 1), so its bits hold the floor plus a constant.  Exact for
// cells below 2^22; the bits grow with t everywhere, so anything farther out
// fails the map's box test.
__device__ __forceinline__ int32_t cell_of(float t) { return __float_as_int(__fadd_rd(t, 1572864.0f)) - 0x49C00000; }
__device__ __forceinline__ int32_t block_of(float t) { return __float_as_int(__fadd_rd(t, 12582912.0f)) - 0x4B400000; }
static_assert(kCoarse == 8, "cell_of");

// Shared memory of the points pass.  Per warp one buffer serves in turn the
// points on their way in, the runs on their way out and the queue of chunks.
constexpr int kRayQ = 256;   // queued chunks per warp (a ring)
constexpr int kMarkQ = 160;  // samples below their threshold: 31 waiting and 4 x 32 of a round
struct ChunkQueue {
  int2 chunk[kRayQ];      // {ray | samples << 8, first sample}
  uint32_t mark[kMarkQ];  // sample | ray << 24
};
union WarpBuf {
  float4 stage[24];
  AccStage acc;
  ChunkQueue q;
};
// The warps' rays, one array per field (lanes reading the fields of different
// rays hit different banks).
struct RaySmem {
  float ax[kPointThreads], bx[kPointThreads], ay[kPointThreads], by[kPointThreads], az[kPointThreads],
      bz[kPointThreads];
  float vx[kPointThreads], vy[kPointThreads], vz[kPointThreads], d[kPointThreads];
  int32_t ix[kPointThreads], iy[kPointThreads], k_lo[kPointThreads], n[kPointThreads], map[kPointThreads],
      cn[kPointThreads];
};
struct FlushBuf {
  int map;
  unsigned long long sum[kPointStats];
};
template <bool kRay>
struct PointsSmem {
  union {
    float4 stage[24];
    AccStage acc;
  } w[kPointWarps];
  FlushBuf flush;
};
template <>
struct PointsSmem<true> {
  WarpBuf w[kPointWarps];
  RaySmem ray;
  FlushBuf flush;
};

__device__ __forceinline__ void put_ray(RaySmem& S, int t, const RaySetup& r) {
  S.ax[t] = r.ax; S.bx[t] = r.bx; S.ay[t] = r.ay; S.by[t] = r.by; S.az[t] = r.az; S.bz[t] = r.bz;
  S.vx[t] = r.vx; S.vy[t] = r.vy; S.vz[t] = r.vz; S.d[t] = r.d;
  S.ix[t] = r.ix; S.iy[t] = r.iy; S.k_lo[t] = r.k_lo; S.n[t] = r.n; S.map[t] = r.map; S.cn[t] = r.cn;
}

// One lane: sample k of ray sr of the warp lies below its cell's threshold.
// Nothing the march reads for its tests is written here: a line that the SMs of
// both dies read while others write it costs far more than the looks it saves
// (thresholds or block flags updated in place took the 64-map batch from 4.0 to
// 6.3 ms and one depth frame from 59 to 112 us).
template <bool kExt, class V>
__device__ __forceinline__ void mark_sample(const V& b, const RaySmem& S, int sr, uint32_t k) {
  const MapDev& m = map_at(b, S.map[sr]);
  const float kf = (float)k;
  // the sample again, by the march's rounded arithmetic
  const int32_t cx = cell_of(__fmaf_rn(kf, S.bx[sr], S.ax[sr])), cy = cell_of(__fmaf_rn(kf, S.by[sr], S.ay[sr]));
  const int32_t p = phys_index(m, cx, cy);
  if (kExt && !isfinite(m.var[p])) {
    // an empty cell (its threshold is the upper bound): the sample lowers the
    // bound (Section II-H); float minimum through the ordered bits
    const int z = __float_as_int(__fmaf_rn(kf, S.bz[sr], S.az[sr]));
    if (z >= 0) atomicMin(reinterpret_cast<int*>(m.upper + p), z);
    else atomicMax(reinterpret_cast<unsigned int*>(m.upper + p), (unsigned)z);
    return;
  }
  // many rays graze the same surface cells: nothing to do when the bit is already
  // set (bits are only ever set during this kernel, so a stale read can only
  // cost a redundant atomic, never a lost mark)
  uint32_t* const word = m.mark + (p >> 5);
  const uint32_t bit = 1u << (p & 31);
  const bool guard = m.alpha_n > 0.f;
  float n0 = 0.f, n1 = 0.f, n2 = 1.f;
  if (guard) {  // (read with the mark, not after it)
    n0 = m.nx[p];
    n1 = m.ny[p];
    n2 = m.nz[p];
  }
  if (*word & bit) return;
  if (guard) {  // Eq. 4
    if (!(isfinite(n0) && isfinite(n1) && isfinite(n2))) { n0 = 0.f; n1 = 0.f; n2 = 1.f; }
    const float rd = S.d[sr];
    const float rx = __fdiv_rn(S.vx[sr], rd), ry = __fdiv_rn(S.vy[sr], rd), rz = __fdiv_rn(S.vz[sr], rd);
    const float dot = fabsf(__fmaf_rn(rx, n0, __fmaf_rn(ry, n1, __fmul_rn(rz, n2))));
    if (!(dot > m.alpha_n)) return;
  }
  atomicOr(word, bit);
}

// Each warp takes 32 consecutive points, adds them to their cells, and marches
// their rays: every lane sets up one ray (the k range inside the map box and
// before the point, its chunk length) and tests its ray's chunks one after
// another; the warp queues the chunks that may mark a cell and marches them
// 4 x 32 / G at a time, G lanes per chunk and one sample per lane and round
// (4 gathers in flight).
template <int G, bool kRay, bool kExt, class V>
__device__ __forceinline__ void points_pass(const V& b, Grid gr, int part, PointsSmem<kRay>& SM) {
  constexpr int kU = G >= 4 ? 4 : G;         // samples per lane and march round, all of one chunk
  constexpr int kLPC = G / kU;               // lanes per chunk in the march
  constexpr int kFQ = 32 / kLPC;             // chunks per march round (at most 32)
  constexpr int kCU = 4;                     // chunks per lane and test round (their loads in flight together)
  constexpr int kQ = kRayQ;
  static_assert(kQ >= kFQ - 1 + 32 * kCU && kFQ <= 32, "queue capacity");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // warps take runs of consecutive 32-point batches, the first by their index
  // in the grid, the others from the work counter (rays of uneven maps differ in
  // length: the counter balances them); a run mostly lies in one cloud and map.
  // Runs are as long as leaves every warp of the grid two of them, at most
  // kRayRun batches.
  const uint32_t n_points = (uint32_t)b.n_points;  // below 2^31
  // the part's batches: `len` of every 32, those at places first .. of the
  // bit-reversed order, so that every part samples the whole clouds (points
  // that go in one part: all of them, in order)
  uint32_t first = 0, len = 32;
  if (kRay && in_parts(b)) {
    first = part_first(part);
    len = part_first(part + 1) - first;
  } else if (part > 0) {
    return;
  }
  // A batch is 32 points, or 16 or 8 while that leaves every warp at most one: a
  // small update is as slow as its slowest warp, and the tests and the march of
  // fewer rays are spread over the same 32 lanes (43,018 points of two dome
  // LiDARs: 64 -> 57 us an update).  Two batches per warp gave those 54 us, but
  // 76,800 points of a camera 33 for 28; batches of 4 gain nothing more.
  const uint32_t warps = (uint32_t)gr.nb * kPointWarps;
  uint32_t span = 32;
  while (span > kMinSpan && (n_points + span / 2 - 1) / (span / 2) <= warps) span /= 2;
  uint32_t n_batches = (n_points + span - 1) / span;
  if (len < 32) n_batches = (n_batches + 31) / 32 * len;
  const uint32_t run_len = max(1u, min((uint32_t)kRayRun, n_batches / (2 * warps)));
  const uint32_t n_runs = (n_batches + run_len - 1) / run_len;
  int cmap = -1;  // the map the warp counts for, and this lane's counter
  unsigned long long count = 0;
  int hint = -1;  // the cloud of the warp's previous batch
  uint32_t run = (uint32_t)gr.bid * kPointWarps + warp;
  uint32_t index = run * run_len;
  while (run < n_runs) {
    const uint32_t batch = len < 32 ? index / len * 32 + (__brev(first + index % len) >> 27) : index;
    const uint32_t p0 = batch * span;
    if (p0 < n_points) {
    // ---- the points: transform, gate, sums
    float px, py, pz;
    const uint32_t p1 = min(p0 + span, n_points), g = p0 + lane;
    const int ci = load_warp_points(b, p0, p1, SM.w[warp].stage, px, py, pz, hint);
    const bool live = g < p1;
    const CloudDev& c = b.clouds[ci];
    const int32_t map = c.map;
    const MapDev& m = map_at(b, map);
    const PointGeom pg = point_geom<kExt>(m, c, px, py, pz);
    const bool inm = live && pg.in_range && in_map(m, pg.ix, pg.iy);
    const uint32_t cell = inm ? (uint32_t)phys_index(m, pg.ix, pg.iy) : 0u;
    const int map0 = __shfl_sync(kFull, map, 0);
    const bool one_map = __all_sync(kFull, map == map0);
    const uint8_t st = add_points<kExt>(b, m, map, one_map, inm, cell, pg.z, pg.d, SM.w[warp].acc);
    if (b.tr_status && live) {
      b.tr_ix[g] = pg.finite ? pg.ix : INT32_MIN;
      b.tr_iy[g] = pg.finite ? pg.iy : INT32_MIN;
      b.tr_status[g] = !pg.finite ? kPtNonFinite : !pg.in_range ? kPtRange : st;
    }
    const bool ok = live && pg.in_range;
    if (one_map) {
      if (map0 != cmap) {
        add_counts(b, cmap, count);
        count = 0;
        cmap = map0;
      }
      const unsigned nv = __popc(__ballot_sync(kFull, ok)), ni = __popc(__ballot_sync(kFull, inm));
      const unsigned na = __popc(__ballot_sync(kFull, st == kPtFused)),
                     nr = __popc(__ballot_sync(kFull, st == kPtRejected));
      count += lane == kPsValid      ? nv
               : lane == kPsInMap    ? ni
               : lane == kPsAccepted ? na
               : lane == kPsRejected ? nr
               : lane == kPsWall     ? ni - na - nr
                                     : 0u;
    } else if (ok) {  // a batch across a map boundary: per lane
      atomicAdd(&m.ctl->stats[kStValid], 1ull);
      if (inm) {
        atomicAdd(&m.ctl->stats[kStInMap], 1ull);
        atomicAdd(&m.ctl->stats[st == kPtFused ? kStAccepted : st == kPtRejected ? kStRejected : kStWall], 1ull);
      }
    }
    if constexpr (kRay) {
    RaySmem& S = SM.ray;
    ChunkQueue& Q = SM.w[warp].q;
    const int wb = warp * 32;  // the warp's rays in S
    // ---- set-up: one ray per lane
    RaySetup r;
    r.n = 0;
    r.map = map;
    r.cn = 1;
    if (ok && m.ray_step > 0.f) {
      // clip the sample range to the map box (conservative by 1 mm + 1 step)
      float lo = 0.f, hi = pg.d;
      const float ext_x = __fmul_rn((float)m.W, m.res), ext_y = __fmul_rn((float)m.H, m.res);
      if (pg.d > 0.f && slab(c.t[0], pg.vx, pg.d, m.x0, m.x0 + ext_x, lo, hi) &&
          slab(c.t[1], pg.vy, pg.d, m.y0, m.y0 + ext_y, lo, hi) && lo <= hi + 1e-3f) {
        const float step = m.ray_step;
        const float kl = floorf(__fdividef(lo - 1e-3f, step)) - 1.f;
        const float kh = ceilf(__fdividef(hi + 1e-3f, step)) + 1.f;
        const int32_t k_lo = kl < 1.f ? 1 : kl > (float)kMaxRayK ? kMaxRayK : (int32_t)kl;
        int32_t k_hi = kh > (float)kMaxRayK ? kMaxRayK : (int32_t)kh;
        // last k with k * step < d, decided exactly as sample by sample
        // (the estimate is within a few units of the answer; past kMaxRayK the
        // range is capped anyway, so the searches stop there)
        float kf = fminf(floorf(__fdividef(pg.d, step)), (float)kMaxRayK);  // an estimate, made exact just below
        int32_t k_last = (int32_t)kf;
        for (int it = 0; it < 64 && k_last > 0 && !(__fmul_rn((float)k_last, step) < pg.d); ++it) --k_last;
        for (int it = 0; it < 64 && k_last < kMaxRayK && __fmul_rn((float)(k_last + 1), step) < pg.d; ++it) ++k_last;
        if (k_last < k_hi) k_hi = k_last;
        const float cstep = __fdiv_rn(step, pg.d);  // f_k = k * step / d
        // in cells, then in blocks (an exact scaling: every sample's cell is that of the unscaled track)
        const float bx = __fmul_rn(__fmul_rn(cstep, pg.vx), m.inv_res);
        const float by = __fmul_rn(__fmul_rn(cstep, pg.vy), m.inv_res);
        r.ax = __fmul_rn(__fmul_rn(__fsub_rn(c.t[0], m.x0), m.inv_res), 1.f / kCoarse);
        r.ay = __fmul_rn(__fmul_rn(__fsub_rn(c.t[1], m.y0), m.inv_res), 1.f / kCoarse);
        r.bx = __fmul_rn(bx, 1.f / kCoarse);
        r.by = __fmul_rn(by, 1.f / kCoarse);
        r.az = c.t[2];
        r.bz = __fmul_rn(cstep, pg.vz);
        r.vx = pg.vx; r.vy = pg.vy; r.vz = pg.vz;
        r.d = pg.d;
        r.ix = pg.ix;
        r.iy = pg.iy;
        r.k_lo = k_lo;
        r.n = k_hi >= k_lo ? k_hi - k_lo + 1 : 0;
        // a chunk and the next chunk's first sample span about kCoarse cells per axis at
        // most, so they touch at most 2 x 2 blocks (a rounding case that touches more is
        // marched untested)
        const float span = fmaxf(fmaxf(fabsf(bx), fabsf(by)), 1e-6f);
        r.cn = (int32_t)fminf((float)G, fmaxf(1.f, floorf(__fdividef((float)kCoarse, span))));
      }
    }
    // samples of the march, per map
    if (one_map) {
      const unsigned t = __reduce_add_sync(kFull, (unsigned)r.n);  // 32 (2^24 - 1) at most
      if (lane == kPsSamples) count += t;
    } else if (r.n > 0) {
      atomicAdd(&m.ctl->stats[kStRaySamples], (unsigned long long)r.n);
    }
    put_ray(S, wb + lane, r);
    __syncwarp();
    // ---- the chunks of the warp's rays against the coarse grid, kCU consecutive
    // chunks of one ray per lane and round.  A ray has nq such quads.  When
    // the rays' lengths differ (points in random order), lanes that each test
    // only their own ray would idle while the longest ray is tested: the quads
    // are then dealt out in order across the lanes (quad j of the warp goes to
    // lane j mod 32 in round j / 32), which the warp does when that saves at
    // least a quarter of the rounds.
    const int32_t nch = r.n > 0 ? (r.n + r.cn - 1) / r.cn : 0;
    const int32_t nq = (nch + kCU - 1) / kCU;
    const int32_t qmax = (int32_t)__reduce_max_sync(kFull, (unsigned)nq);
    const int32_t qtot = (int32_t)__reduce_add_sync(kFull, (unsigned)nq);
    const bool flat = 4 * ((qtot + 31) >> 5) <= 3 * qmax;  // warp-uniform
    const int32_t rounds = flat ? (qtot + 31) >> 5 : qmax;
    int32_t qinc = nq;  // inclusive scan of the quads over the lanes
    if (flat) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(kFull, qinc, o);
        if (lane >= o) qinc += t;
      }
    }
    int qh = 0, qn = 0, mn = 0;  // chunk queue: head and length; mark queue: length (warp-uniform)
    for (int32_t it = 0; it < rounds; ++it) {
      // this lane's quad: ray `src`, chunks c0 .. c0 + kCU - 1
      int src = lane;
      int32_t c0 = it * kCU;
      bool act = it < nq;
      if (flat) {
        const int32_t j = it * 32 + lane;
        int o = 0;  // lanes whose quads all come before quad j: the owner of quad j
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
          const int32_t v = __shfl_sync(kFull, qinc, o + s - 1);
          if (v <= j) o += s;
        }
        act = j < qtot;
        src = o < 32 ? o : 31;
        c0 = (j - __shfl_sync(kFull, qinc - nq, src)) * kCU;
      }
      const int sr = wb + src;
      const int32_t cn = S.cn[sr], kq = S.k_lo[sr] + c0 * cn;  // the quad's first sample
      const int32_t left = act ? S.n[sr] - c0 * cn : 0;        // samples from there on
      const float ax = S.ax[sr], bx = S.bx[sr], ay = S.ay[sr], by = S.by[sr], az = S.az[sr], bz = S.bz[sr];
      // The round's chunks and their end samples: chunk u is tested over its own
      // samples and the next chunk's first one (a superset, so the test stays
      // exact), so neighbouring chunks share an end and its block.  Blocks
      // outside the map are those of the grid's rim, which holds -inf.  All loads
      // of the round come first (no branches between them), then the tests.
      const MapDev& m = map_at(b, S.map[sr]);
      const float* ct = m.cthr;
      const int32_t CW = m.CW, CH = m.CH, CS = m.CS;
      int32_t xb[kCU + 1], yb[kCU + 1];
      float zc[kCU + 1], ve[kCU + 1];
#pragma unroll
      for (int u = 0; u <= kCU; ++u) {
        const float kf = (float)(kq + min(u * cn, max(left - 1, 0)));
        xb[u] = min(max(block_of(__fmaf_rn(kf, bx, ax)), -1), CW);
        yb[u] = min(max(block_of(__fmaf_rn(kf, by, ay)), -1), CH);
        zc[u] = __fmaf_rn(kf, bz, az);
        ve[u] = left > 0 ? ct[yb[u] * CS + xb[u]] : __int_as_float(0xff800000);
      }
#pragma unroll
      for (int u = 0; u < kCU; ++u) {
        const int32_t dx = xb[u + 1] - xb[u], dy = yb[u + 1] - yb[u];
        // the two other corners of the 2 x 2 box, when the chunk crosses a block row and column
        float mx = fmaxf(ve[u], ve[u + 1]);
        if (left > 0 && dx != 0 && dy != 0) mx = fmaxf(mx, fmaxf(ct[yb[u] * CS + xb[u + 1]], ct[yb[u + 1] * CS + xb[u]]));
        // more than 2 x 2 blocks (not for the chunk lengths above): march it untested
        const bool wide = (unsigned)(dx + 1) > 2u || (unsigned)(dy + 1) > 2u;
        const int32_t cnt = min(cn, left - u * cn);
        const bool keep = cnt > 0 && (wide || fminf(zc[u], zc[u + 1]) < mx);
        // ---- queue the chunks that may mark a cell
        const unsigned km = __ballot_sync(kFull, keep);
        if (keep)
          Q.chunk[(qh + qn + __popc(km & ((1u << lane) - 1u))) & (kQ - 1)] =
              make_int2(src | (cnt << 8), kq + u * cn);
        qn += __popc(km);
      }
      __syncwarp();
      // ---- march the queued chunks, kFQ at a time (all of them after the last test)
      const bool last = it + 1 >= rounds;
      while (qn >= kFQ || (last && qn > 0)) {
        // lane: chunk qi, samples sj, sj + kLPC, ...; every threshold first (kU gathers
        // in flight), then the samples below theirs go to the mark queue: a few lanes
        // in a hundred, so marking them where they are found would run a long branch
        // for one or two lanes at a time
        const int qi = lane / kLPC, sj = lane % kLPC;
        const int2 e = Q.chunk[(qh + qi) & (kQ - 1)];
        const int32_t ne = qi < qn ? e.x >> 8 : 0;
        const int mr = qi < qn ? e.x & 31 : 0, sm = wb + mr;
        const MapDev& mm = map_at(b, S.map[sm]);
        const int32_t Wm = mm.W, Hm = mm.H;
        const float* tm = mm.thr;
        const float mx0 = S.ax[sm], mbx = S.bx[sm], my0 = S.ay[sm], mby = S.by[sm], mz0 = S.az[sm], mbz = S.bz[sm];
        const int32_t rix = S.ix[sm], riy = S.iy[sm];
        const float kf0 = (float)(e.y + sj);
        float zz[kU], th[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const float kf = kf0 + (float)(u * kLPC);
          const int32_t cx = cell_of(__fmaf_rn(kf, mbx, mx0));
          const int32_t cy = cell_of(__fmaf_rn(kf, mby, my0));
          const bool in = sj + u * kLPC < ne && (uint32_t)cx < (uint32_t)Wm && (uint32_t)cy < (uint32_t)Hm &&
                          !(cx == rix && cy == riy);
          zz[u] = __fmaf_rn(kf, mbz, mz0);
          th[u] = in ? tm[cy * Wm + cx] : __int_as_float(0xff800000);  // logical index; -inf: never below
        }
        bool any = false;
#pragma unroll
        for (int u = 0; u < kU; ++u) any |= zz[u] < th[u];
        if (__any_sync(kFull, any)) {
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const bool below = zz[u] < th[u];
            const unsigned bm = __ballot_sync(kFull, below);
            if (below)
              Q.mark[mn + __popc(bm & ((1u << lane) - 1u))] = (uint32_t)(e.y + sj + u * kLPC) | (uint32_t)mr << 24;
            mn += __popc(bm);
          }
          __syncwarp();
          while (mn >= 32) {
            mn -= 32;
            const uint32_t v = Q.mark[mn + lane];
            mark_sample<kExt>(b, S, wb + (int)(v >> 24), v & 0xffffffu);
          }
          __syncwarp();
        }
        const int took = min(qn, kFQ);
        qh = (qh + took) & (kQ - 1);
        qn -= took;
        __syncwarp();
      }
    }
    if (lane < mn) {
      const uint32_t v = Q.mark[lane];
      mark_sample<kExt>(b, S, wb + (int)(v >> 24), v & 0xffffffu);
    }
    __syncwarp();
    }
    }  // a batch of the clouds
    // the next batch of the run, or the next run
    ++index;
    if (index >= (run + 1) * run_len || index >= n_batches) {
      uint32_t t = 0;
      if (lane == 0) t = (uint32_t)atomicAdd(&b.ctl->next[part], 1);
      run = warps + __shfl_sync(kFull, t, 0);
      index = run * run_len;
    }
  }
  // the warps' counts: one atomic per block and counter when the block saw one
  // map last, else one per warp
  FlushBuf& F = SM.flush;
  if (threadIdx.x == 0) F.map = cmap;
  if (threadIdx.x < kPointStats) F.sum[threadIdx.x] = 0;
  __syncthreads();
  if (cmap == F.map) {
    if (lane < kPointStats && count) atomicAdd(&F.sum[lane], count);
  } else {
    add_counts(b, cmap, count);
  }
  __syncthreads();
  if (threadIdx.x < kPointStats && F.map >= 0 && F.sum[threadIdx.x])
    atomicAdd(&map_at(b, F.map).ctl->stats[stat_of(threadIdx.x)], F.sum[threadIdx.x]);
  __syncthreads();  // the shared memory is free again
}

}  // namespace em
