// k_point.cu -- the kernels over the points (point_pass.cuh).
//
// Fusion (Section II-C of the paper): every point is gated against its cell's
// pre-update estimate (wall rule, then the Mahalanobis gate) and its exact
// fixed-point terms are added to the cell's accumulator with integer
// reductions, so the result does not depend on the points' order; k_write
// turns the sums into the new estimate.  No grouping of the points by cell: the
// reductions of a 407,040-point depth image, or of 14 M points in random order
// over 64 maps, cost less than a counting sort by tile and a fusion from shared
// memory did (count, range, scatter and fusion kernels: 1130 us of the 64-map
// batch, where gate and sums without rays take 380; 184 us of the depth image's
// kernels, now 18), and one launch takes the place of four.
//
// Visibility (Section II-E): one ray per valid point.  The ray from the sensor
// origin o (the pose translation) to the point is sampled at s_k = o + (k step / d) (R p_s) for
// k = 1, 2, ... while k step < d (computed as a + k b in cell units: one FMA
// per coordinate).  A sample inside the map, outside the point's own cell,
// below the cell's threshold h - sqrt(sigma_m^2) of the pre-update map (Eq. 3;
// the threshold layer is -inf for empty cells) and -- when alpha_n > 0 -- with
// |rhat . n| > alpha_n for the cell's previous normal (Eq. 4; a NaN normal
// counts as (0, 0, 1)) marks the cell in a bitmask (atomicOr: idempotent, so
// the marks do not depend on thread order).  Only the k whose samples can lie
// inside the map's box are visited.
//
// Most samples of a scan pass far above the surface.  k_cells keeps, per
// block of kCoarse x kCoarse cells, the largest threshold of the block.  The
// march cuts each ray into chunks of at most G samples spanning at most
// kCoarse cells per axis; a chunk's samples lie in the cells between those of
// its first sample and the next chunk's first sample (both coordinates and z
// are monotone in k, and the same rounded arithmetic gives every sample), so
// when the lower of those two heights is not below the largest threshold of
// the (at most 2 x 2) blocks they span, none of its samples can mark a cell
// and it is skipped -- an exact test, not a heuristic.
//
// What bounds it: issue and latency (one depth frame of 4 x 76,800 points: 23.5 M
// warp instructions before the tests went to block coordinates on a rimmed grid
// and the marks to a queue, 20 M then; 66 -> 58 us per update), on scattered
// points the gathers of thresholds from L2 (1.4 G sectors for the 64-map batch,
// which the parts with refreshed thresholds cut to about a third).  256 threads
// and 64 registers, four blocks per SM: one resident wave that takes runs of
// batches from a counter (the builds that read an uploaded descriptor spill 32 bytes
// a thread at that, those with the descriptor as a parameter none).  Measured and not kept: one test for the beam of a warp's
// 32 rays before the rays' own (no fewer instructions: rays of an image row
// have 4 to 8 chunks); thresholds or block maxima updated in place by the march
// (mark_sample).
#include "em.h"
#include "point_pass.cuh"

namespace em {

template <bool kExt, class D>
__global__ void __launch_bounds__(kPointThreads) k_pre(const __grid_constant__ D d) {
  __shared__ PreSmem S;
  begin_after_previous();
  pre_pass<kExt>(view(d), own_grid(), S);
}

template <int G, bool kRay, bool kExt, class D>
__global__ void __launch_bounds__(kPointThreads, 4) k_points(const __grid_constant__ D d, int part) {
  __shared__ PointsSmem<kRay> S;
  begin_after_previous();
  points_pass<G, kRay, kExt>(view(d), own_grid(), part, S);
}

int sm_count() {
  static int cached[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 148;
  if (!cached[dev]) {
    int sms = 148;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cached[dev] = sms;
  }
  return cached[dev];
}

// Blocks for n points, `span` of them per warp at least.
static int point_grid(int64_t n, int span, int per_sm) {
  const int64_t want = (n + span * kPointWarps - 1) / (span * kPointWarps);
  const int64_t cap = (int64_t)sm_count() * per_sm;
  return (int)(want < 1 ? 1 : want < cap ? want : cap);
}

Launch pre_launch(int64_t n_points, bool ext, bool by_value) {
  if (n_points <= 0) return {};
  const void* fn = by_value ? (ext ? (const void*)&k_pre<true, MapDesc> : (const void*)&k_pre<false, MapDesc>)
                   : ext    ? (const void*)&k_pre<true, const BatchDev*>
                            : (const void*)&k_pre<false, const BatchDev*>;
  return {fn, (unsigned)point_grid(n_points, 32, 16), kPointThreads, 0, false, EM_PROF_SCATTER, "k_pre", 0};
}

template <bool kExt>
static const void* points_kernel(int g) {
  switch (g) {
    case 1: return (const void*)&k_points<1, true, kExt, const BatchDev*>;
    case 2: return (const void*)&k_points<2, true, kExt, const BatchDev*>;
    case 4: return (const void*)&k_points<4, true, kExt, const BatchDev*>;
    case 16: return (const void*)&k_points<16, true, kExt, const BatchDev*>;
    case 32: return (const void*)&k_points<32, true, kExt, const BatchDev*>;
    default: return (const void*)&k_points<8, true, kExt, const BatchDev*>;
  }
}
// The descriptor by value: kValueGroup samples per chunk only.
template <bool kRay, bool kExt>
static const void* points_kernel_value() {
  return (const void*)&k_points<kValueGroup, kRay, kExt, MapDesc>;
}

Launch points_launch(int64_t n_points, int group, bool ray, bool ext, int part, bool by_value) {
  if (n_points <= 0) return {};
  const void* fn;
  if (by_value)
    fn = ray ? (ext ? points_kernel_value<true, true>() : points_kernel_value<true, false>())
         : ext ? points_kernel_value<false, true>()
               : points_kernel_value<false, false>();
  else
    fn = ray ? (ext ? points_kernel<true>(group) : points_kernel<false>(group))
         : ext ? (const void*)&k_points<8, false, true, const BatchDev*>
               : (const void*)&k_points<8, false, false, const BatchDev*>;
  return {fn, (unsigned)point_grid(n_points, kMinSpan, 4), kPointThreads, 0, false, EM_PROF_RAY, "k_points", part};
}

}  // namespace em
