// cell_pass.cuh -- the device passes over the cells (k_cell.cu):
//
//   cells_pass  before the points: estimates moved by the drift, ray thresholds
//               of the pre-update map and their largest per coarse block
//   refresh_pass  between parts of the points: marked cells out of both
//   sums_pass   after them: new state of the cells whose sums are in the table
//   write_pass  every cell's new state from its sums, removal of marked cells,
//               overlap clearance
//
// Each pass runs on the blocks of a Grid: its own kernel's, or the persistent
// kernel's (k_persist.cu).
#pragma once

#include "em_point.cuh"

namespace em {

constexpr int kCellThreads = 256;

// Do the points of a large update come in a sensor's order?  kOrderSamples
// batches of 32 consecutive points, spread over the clouds, one warp's loads for
// one block each; a batch counts as scattered when more than half of its
// neighbouring points lie farther apart than half the nearer one's distance.
template <class V>
__device__ __forceinline__ void sample_order(const V& b, Grid gr) {
  if (b.n_points < kSplitPoints) return;
  const int lane = threadIdx.x & 31;
  const int64_t n_batches = b.n_points / 32;  // whole ones
  int scattered = 0;
  for (int k = gr.bid; k < kOrderSamples; k += gr.nb) {
    const int64_t g = n_batches * k / kOrderSamples * 32 + lane;
    const CloudDev& c = b.clouds[find_cloud(b.clouds, b.n_clouds, g)];
    float px, py, pz;
    load_point(c, g - c.begin, px, py, pz);
    const float qx = __shfl_down_sync(kFull, px, 1), qy = __shfl_down_sync(kFull, py, 1),
                qz = __shfl_down_sync(kFull, pz, 1);
    const float dx = qx - px, dy = qy - py, dz = qz - pz;
    const float near = fminf(px * px + py * py + pz * pz, qx * qx + qy * qy + qz * qz);
    const bool far = lane < 31 && dx * dx + dy * dy + dz * dz > 0.25f * near;  // false for NaN
    scattered += __popc(__ballot_sync(kFull, far)) > 16;
  }
  if (lane == 0 && scattered) atomicAdd(&b.ctl->scattered, scattered);
}

// One warp per item: body(map, item column, item row), called by whole warps.
template <class V, class F>
__device__ __forceinline__ void for_each_item(const V& b, Grid gr, F body) {
  const int warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  for (int64_t g = (int64_t)gr.bid * warps + warp; g < b.n_items; g += (int64_t)gr.nb * warps) {
    int lo = 0, hi = b.n_maps - 1;  // the last map whose items start at or before g
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (b.maps[mid].ibegin <= g) lo = mid; else hi = mid - 1;
    }
    const MapDev& m = map_at(b, lo);
    const int32_t q = (int32_t)(g - m.ibegin);
    const int32_t ty = q / m.IW;
    body(m, q - ty * m.IW, ty);
  }
}

// The item's coarse blocks from the lanes' column maxima, and the rim entries
// beside blocks at the map's edge.
__device__ __forceinline__ void put_coarse(const MapDev& m, int32_t tx, int32_t ty, float mx) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < kCoarse; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
  const int32_t cx = tx * (kItemW / kCoarse) + lane / kCoarse;
  if (lane % kCoarse != 0 || cx >= m.CW) return;
  float* const c = m.cthr + ty * m.CS + cx;
  const int l = cx == 0 ? -1 : 0, r = cx == m.CW - 1 ? 1 : 0, t = ty == 0 ? -1 : 0, d = ty == m.CH - 1 ? 1 : 0;
  for (int y = t; y <= d; ++y)
    for (int x = l; x <= r; ++x) c[y * m.CS + x] = x == 0 && y == 0 ? mx : __int_as_float(0xff800000);
}

// One warp per item of kItemW x kItemH logical cells: a lane's column of 8
// cells gives 24 independent loads, rows are coalesced in both layouts, and the
// item's four coarse blocks are maxima over 8 lanes.  The thresholds go to
// logical order, so the march indexes them without the ring wrap.
static_assert(kItemH == kCoarse && kItemW == 32 && kItemW % kCoarse == 0, "items hold whole coarse blocks");
template <class V>
__device__ __forceinline__ void cells_pass(const V& b, Grid gr) {
  if (threadIdx.x < 32) sample_order(b, gr);
  for_each_item(b, gr, [&](const MapDev& m, int32_t tx, int32_t ty) {
    const int lane = threadIdx.x & 31;
    const int32_t W = m.W, lx = tx * kItemW + lane, y0 = ty * kItemH;
    const int32_t rows = lx < W ? min(kItemH, m.H - y0) : 0;
    int32_t px = lx + m.ox;
    px -= px >= W ? W : 0;
    const bool drift = m.drift_flat > 0.f, ray = m.ray_step > 0.f;
    float var[kItemH], h[kItemH];
    int32_t tl[kItemH], p[kItemH];
#pragma unroll
    for (int r = 0; r < kItemH; ++r) {  // all loads first
      int32_t py = y0 + r + m.oy;
      py -= py >= m.H ? m.H : 0;
      p[r] = py * W + px;
      var[r] = r < rows ? m.var[p[r]] : __int_as_float(0x7f800000);
      h[r] = r < rows ? m.h[p[r]] : 0.f;
      tl[r] = r < rows ? m.t_last[p[r]] : 0;
    }
    if (drift) {
      // height drift compensation (Section II-D): every estimate moves by the mean
      // error of this update's points in flat cells (k_pre summed them exactly, so
      // every thread derives the same mean)
      const unsigned long long n = m.ctl->drift_n;
      const float mean = n ? __fdiv_rn(fixed_to_float(fix128(m.ctl->drift_h, m.ctl->drift_l)), (float)n) : 0.f;
      if (tx == 0 && ty == 0 && lane == 0) {  // once per map
        atomicAdd(&m.ctl->stats[kStDriftPoints], n);
        m.ctl->drift_last = mean;
      }
#pragma unroll
      for (int r = 0; r < kItemH; ++r) {
        if (r < rows && isfinite(var[r]) && n) {
          h[r] = __fadd_rn(h[r], mean);
          m.h[p[r]] = h[r];
        }
      }
    }
    if (!ray) return;
    // Eq. 3: h - sqrt(var_eff); an empty cell is never penetrated (-inf).  With
    // the upper-bound layer it holds the cell's bound instead, so a ray sample
    // below the bound takes the march's candidate path and lowers it (Section II-H)
    float mx = __int_as_float(0xff800000);
#pragma unroll
    for (int r = 0; r < kItemH; ++r) {
      if (r >= rows) continue;
      float t = __int_as_float(0xff800000);
      if (isfinite(var[r])) t = __fsub_rn(h[r], __fsqrt_rn(var_eff(m, var[r], tl[r])));
      else if (m.upper) t = m.upper[p[r]];
      m.thr[(y0 + r) * W + lx] = t;
      mx = fmaxf(mx, t);  // a NaN never marks: skipped
    }
    put_coarse(m, tx, ty, mx);
  });
}

// Between two parts of the points: a marked cell stays marked, so its threshold
// becomes -inf; an empty cell's is its bound as lowered so far; and the coarse
// blocks' maxima are taken again.
template <class V>
__device__ __forceinline__ void refresh_pass(const V& b, Grid gr) {
  if (!in_parts(b)) return;
  for_each_item(b, gr, [&](const MapDev& m, int32_t tx, int32_t ty) {
    if (m.ray_step <= 0.f) return;
    const int lane = threadIdx.x & 31;
    const int32_t W = m.W, lx = tx * kItemW + lane, y0 = ty * kItemH;
    const int32_t rows = lx < W ? min(kItemH, m.H - y0) : 0;
    int32_t px = lx + m.ox;
    px -= px >= W ? W : 0;
    float t[kItemH];
    uint32_t mark[kItemH];
#pragma unroll
    for (int r = 0; r < kItemH; ++r) {  // all loads first
      int32_t py = y0 + r + m.oy;
      py -= py >= m.H ? m.H : 0;
      const int32_t p = py * W + px;
      t[r] = r < rows ? m.thr[(y0 + r) * W + lx] : __int_as_float(0xff800000);
      mark[r] = r < rows ? (m.mark[p >> 5] >> (p & 31)) & 1u : 0u;
      if (m.upper && r < rows && !isfinite(m.var[p])) t[r] = m.upper[p];
    }
    float mx = __int_as_float(0xff800000);
#pragma unroll
    for (int r = 0; r < kItemH; ++r) {
      if (r >= rows) continue;
      if (mark[r]) t[r] = __int_as_float(0xff800000);
      if (mark[r] || m.upper) m.thr[(y0 + r) * W + lx] = t[r];
      mx = fmaxf(mx, t[r]);
    }
    put_coarse(m, tx, ty, mx);
  });
}

// New state of a cell from its complete sums; acc: some point was accepted, rej:
// rejected points (Section II-C: every rejection adds outlier_variance; then
// Eq. 1 and Eq. 2 for all accepted points at once in information form).
__device__ __forceinline__ void fused_state(const MapDev& m, float h, float var, int32_t tl, __int128 qw, __int128 qt,
                                            bool acc, uint32_t rej, float& h_new, float& var_new) {
  const float sw = fixed_to_float(qw), st = fixed_to_float(qt);
  if (isfinite(var)) {
    const float vprior = __fadd_rn(var_eff(m, var, tl), __fmul_rn((float)(int)rej, m.v_out));
    if (!acc) {
      h_new = h;
      var_new = vprior;
    } else {
      const float lam = __fadd_rn(__frcp_rn(vprior), sw);
      h_new = __fadd_rn(h, __fdiv_rn(st, lam));
      var_new = __frcp_rn(lam);
    }
  } else {
    h_new = __fadd_rn(m.z_ref, __fdiv_rn(st, sw));
    var_new = __frcp_rn(sw);
  }
}

// A cell's accumulator with one 32-byte load.
__device__ __forceinline__ CellAcc load_acc(const CellAcc* p) {
  CellAcc a;
  asm volatile("ld.global.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(a.wh), "=l"(a.wl), "=l"(a.th), "=l"(a.tl)
               : "l"(p)
               : "memory");
  return a;
}
__device__ __forceinline__ void clear_acc(CellAcc* p) {
  asm volatile("st.global.v4.u64 [%0], {%1, %1, %1, %1};" ::"l"(p), "l"(0ull) : "memory");
}

// The cells of maps with keys: a slot of the table per thread and round.  Freed
// slots, sums and counts go back to zero.  The cells are written now, so write_pass,
// which runs after this, finds them too young to remove (Section II-E).
template <class V>
__device__ __forceinline__ void sums_pass(const V& b, Grid gr) {
  const SumTable& t = b.tab;
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)gr.bid * kCellThreads; base < t.slots; base += (int64_t)gr.nb * kCellThreads) {
    const int64_t i = base + threadIdx.x;
    const unsigned long long key = i < t.slots ? t.keys[i] : 0ull;
    int updated = -1;  // the map whose cell this lane writes
    if (key) {
      const CellAcc a = load_acc(t.acc + i);
      const uint32_t rej = t.rej[i];
      const int64_t g = (int64_t)(key - 1ull);
      const int mi = find_map_cell(b.maps, b.n_maps, g);
      const MapDev& m = map_at(b, mi);
      const int32_t c = (int32_t)(g - m.cell_begin);
      const bool acc = (a.wh | a.wl) != 0;
      if (acc || rej) {
        float hn, vn;
        fused_state(m, m.h[c], m.var[c], m.t_last[c], fix128((long long)a.wh, a.wl & ~kAccTouched),
                    fix128((long long)a.th, a.tl), acc, rej, hn, vn);
        m.h[c] = hn;
        m.var[c] = vn;
        m.t_last[c] = m.t_now;
        if (m.upper) m.upper[c] = __int_as_float(0x7f800000);  // observed: no bound (Section II-H)
        updated = mi;
      }
      t.keys[i] = 0ull;
      if (acc) clear_acc(t.acc + i);
      if (rej) t.rej[i] = 0;
      if (m.cnt) t.cnt[i] = 0;
    }
    const unsigned same = __match_any_sync(kFull, updated);
    if (updated >= 0 && lane == __ffs(same) - 1)
      atomicAdd(&map_at(b, updated).ctl->stats[kStCellsUpdated], (unsigned long long)__popc(same));
  }
}

// One block per tile of kTile cells, a cell per thread and round: the sums of
// the tile's four rounds are in flight together.  Sums, counts, marks and the
// tile's flag go back to zero for the next update.  Tiles start on multiples of
// kTile cells, so a tile owns whole mark words.
constexpr int kWriteRounds = kTile / kCellThreads;
template <class V>
__device__ __forceinline__ void write_pass(const V& b, Grid gr) {
  const int lane = threadIdx.x & 31;
  if (gr.bid == 0 && threadIdx.x == 0) {
    for (int i = 0; i < kParts; ++i) b.ctl->next[i] = 0;
    b.ctl->scattered = 0;
  }
  for_each_tile(b, gr, [&](const MapDev& m, int, int32_t p0, int32_t count) {
    const int32_t tile = p0 / kTile;
    if (p0 == 0 && threadIdx.x == 0) {  // once per map
      atomicAdd(&m.ctl->stats[kStUpdates], 1ull);
      m.ctl->drift_h = 0;
      m.ctl->drift_l = 0;
      m.ctl->drift_n = 0;
    }
    const bool touched = m.acc && !m.keys && (!m.touched || m.touched[tile] != 0);
    const bool overlap = m.ovl_dz > 0.f;
    CellAcc a[kWriteRounds];
    uint32_t rej[kWriteRounds], mark[kWriteRounds];
#pragma unroll
    for (int k = 0; k < kWriteRounds; ++k) {
      const int32_t i = k * kCellThreads + threadIdx.x, c = p0 + i;
      a[k] = CellAcc{0, 0, 0, 0};
      rej[k] = 0;
      mark[k] = i < count ? m.mark[c >> 5] : 0u;
      if (touched && i < count) {
        a[k] = load_acc(m.acc + c);
        rej[k] = m.rej[c];
        if (m.cnt && m.cnt[c]) m.cnt[c] = 0;
      }
    }
    unsigned updated = 0, cleared = 0;
#pragma unroll
    for (int k = 0; k < kWriteRounds; ++k) {
      const int32_t i = k * kCellThreads + threadIdx.x, c = p0 + i;
      const bool acc = (a[k].wh | a[k].wl) != 0;  // (an accepted point leaves a weight or kAccTouched)
      const bool mk = (mark[k] >> (c & 31)) & 1u;
      const bool fused = acc || rej[k] != 0;
      // overlap clearance (Section II-F): an estimate whose cell centre lies within
      // overlap_radius of the robot (the first cloud's sensor origin) and whose
      // height is more than overlap_dz from the robot's belongs to another floor
      bool near = false;
      if (overlap && i < count) {
        int32_t lx, ly;
        logical_of(m, c, lx, ly);
        const float cx = __fsub_rn(__fmaf_rn(__fadd_rn((float)lx, 0.5f), m.res, m.x0), m.ref_x);
        const float cy = __fsub_rn(__fmaf_rn(__fadd_rn((float)ly, 0.5f), m.res, m.y0), m.ref_y);
        near = __fmaf_rn(cx, cx, __fmul_rn(cy, cy)) <= m.ovl_r2;
      }
      if (!(fused || mk || near)) continue;
      float h = m.h[c], var = m.var[c];
      int32_t tl = m.t_last[c];
      bool gone = false;
      if (fused) {
        if (acc) clear_acc(m.acc + c);
        if (rej[k]) m.rej[c] = 0;
        float hn, vn;
        fused_state(m, h, var, tl, fix128((long long)a[k].wh, a[k].wl & ~kAccTouched),
                    fix128((long long)a[k].th, a[k].tl), acc, rej[k], hn, vn);
        h = hn;
        var = vn;
        m.h[c] = h;
        m.var[c] = var;
        m.t_last[c] = m.t_now;
        if (m.upper) m.upper[c] = __int_as_float(0x7f800000);  // observed: no bound (Section II-H)
        ++updated;
      } else if (mk && isfinite(var) && m.t_now - tl >= (m.min_age > 1 ? m.min_age : 1)) {
        gone = true;  // penetrated and not written recently (a cell written now has age 0)
        ++cleared;
      }
      if (!gone && near && isfinite(var) && fabsf(__fsub_rn(h, m.z_ref)) > m.ovl_dz) gone = true;
      if (gone) {
        m.h[c] = __int_as_float(0x7fc00000);
        m.var[c] = __int_as_float(0x7f800000);
      }
    }
    // the mark words are reset after their readers (one warp each) have read them
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kWriteRounds; ++k)
      if (lane == 0 && mark[k]) m.mark[(p0 + k * kCellThreads + (int)threadIdx.x) >> 5] = 0u;
    const unsigned nu = __reduce_add_sync(kFull, updated), nc = __reduce_add_sync(kFull, cleared);
    if (lane == 0 && nu) atomicAdd(&m.ctl->stats[kStCellsUpdated], (unsigned long long)nu);
    if (lane == 0 && nc) atomicAdd(&m.ctl->stats[kStCleared], (unsigned long long)nc);
    if (m.touched) {
      __syncthreads();  // every thread has read the tile's flag
      if (threadIdx.x == 0 && touched) m.touched[tile] = 0;
    }
  });
}

// What an update that stopped half way left behind: everything that is zero
// between updates goes back to zero.  One block, after every other block of the
// launch has left (64 maps of 250,000 cells: 0.6 GB, some milliseconds).
template <class V>
__device__ __forceinline__ void clear_scratch(const V& b) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < kParts; ++i) b.ctl->next[i] = 0;
    b.ctl->scattered = 0;
  }
  for (int mi = 0; mi < b.n_maps; ++mi) {
    const MapDev& m = map_at(b, mi);
    const int32_t ncell = m.W * m.H;
    const bool flat = m.acc && !m.keys;
    for (int32_t c = threadIdx.x; c < ncell; c += blockDim.x) {
      if (flat) {
        clear_acc(m.acc + c);
        m.rej[c] = 0;
        if (m.cnt) m.cnt[c] = 0;
      }
      if (c % 32 == 0) m.mark[c / 32] = 0;
      if (m.touched && c % kTile == 0) m.touched[c / kTile] = 0;
    }
    if (threadIdx.x == 0) {
      m.ctl->drift_h = 0;
      m.ctl->drift_l = 0;
      m.ctl->drift_n = 0;
    }
  }
  for (int64_t i = threadIdx.x; i < b.tab.slots; i += blockDim.x) {
    b.tab.keys[i] = 0ull;
    clear_acc(b.tab.acc + i);
    b.tab.rej[i] = 0;
    if (b.tab.cnt) b.tab.cnt[i] = 0;
  }
}

}  // namespace em
