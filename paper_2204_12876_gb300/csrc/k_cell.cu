// k_cell.cu -- the kernels over the cells (cell_pass.cuh), launched before and
// after the points.
//
// Eq. 1 and Eq. 2 for all accepted points of a cell at once, in information form:
//   Lambda = 1 / (sigma_m^2 + n_rej v_out) + sum_i 1/sigma_p,i^2
//   h'     = h_ref + sum_i (z_i - h_ref) / sigma_p,i^2 / Lambda,   sigma_m^2' = 1 / Lambda
// with h_ref = h for a valid cell (an empty cell has 1/sigma_m^2 = 0 and h_ref =
// the map's reference height z_ref).  Applying Eq. 1/2 point after point gives
// the same result in exact arithmetic.
//
// The two sums are exact: every float32 term is a fixed-point integer with 44
// fractional bits (kept as h 2^27 + l) and the integers are added.  Integer
// addition is associative, so the result is the same for every order of the
// points and every split of the work, bit for bit (no float atomics).
#include "cell_pass.cuh"
#include "em.h"

namespace em {

// Latency-bound on one map (9 us cold for 250 x 250 cells: two dependent loads
// and the square roots), DRAM-bound on many (37 us for the 64-map batch's 6.8 M
// cells, 43 cold).  It takes the place of a threshold pass in the point kernel and a
// one-thread-per-block coarse kernel (12 us alone on one map).
template <class D>
__global__ void __launch_bounds__(kCellThreads) k_cells(const __grid_constant__ D d) {
  begin_after_previous();
  cells_pass(view(d), own_grid());
}

// Latency-bound: a slot's key, its sums and its cell's state are dependent reads, the
// last one scattered (16 us for 491,521 slots, 113,000 of them in use).
template <class D>
__global__ void __launch_bounds__(kCellThreads) k_sums(const __grid_constant__ D d) {
  begin_after_previous();
  sums_pass(view(d), own_grid());
}

// DRAM-bound on many maps (106 us for the 64-map batch; 556 MB in 132 us cold: 36
// bytes of sums and 12 of state per touched cell, read and written); 8-12 us cold
// on one.
template <class D>
__global__ void __launch_bounds__(kCellThreads) k_write(const __grid_constant__ D d) {
  begin_after_previous();
  write_pass(view(d), own_grid());
}

// Skips (one load a block) when the points went in one part.
template <class D>
__global__ void __launch_bounds__(kCellThreads) k_refresh(const __grid_constant__ D d) {
  begin_after_previous();
  refresh_pass(view(d), own_grid());
}

// n_cells bounds the items but for partial last rows and columns (the pass strides over the grid)
static Launch item_launch(const void* fn, int64_t n_cells, int slot, const char* name) {
  constexpr int kThreads = kCellThreads;
  const int64_t blocks = n_cells / (kItemW * kItemH * (kThreads / 32)) + 1;
  const int64_t cap = (int64_t)sm_count() * 16;
  return {fn, (unsigned)(blocks < cap ? blocks : cap), kThreads, 0, false, slot, name, 0};
}
Launch cells_launch(int64_t n_cells, bool by_value) {
  return item_launch(EM_KERNEL(k_cells, by_value), n_cells, EM_PROF_COUNT, "k_cells");
}
Launch refresh_launch(int64_t n_cells, bool by_value) {
  return item_launch(EM_KERNEL(k_refresh, by_value), n_cells, EM_PROF_RAY, "k_refresh");
}

Launch sums_launch(uint32_t slots, bool by_value) {
  if (!slots) return {};
  const int64_t blocks = ((int64_t)slots + kCellThreads - 1) / kCellThreads, cap = (int64_t)sm_count() * 8;
  return {EM_KERNEL(k_sums, by_value), (unsigned)(blocks < cap ? blocks : cap), kCellThreads, 0, false, EM_PROF_FUSE,
          "k_sums", 0};
}

Launch write_launch(int64_t n_cells, bool by_value) {
  const int64_t tiles = n_cells / kTile;  // a block per tile
  const int64_t cap = (int64_t)sm_count() * 8;
  const unsigned grid = (unsigned)(tiles < 1 ? 1 : tiles < cap ? tiles : cap);
  return {EM_KERNEL(k_write, by_value), grid, kCellThreads, 0, false, EM_PROF_FUSE, "k_write", 0};
}

}  // namespace em
