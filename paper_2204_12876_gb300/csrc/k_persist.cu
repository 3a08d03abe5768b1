// k_persist.cu -- the batched form in one persistent launch: the passes of an
// update over every map of a batch (transform, noise, binning, wall rule, gate,
// Eq. 1/2 fusion, ray march and removal; Section II-A to II-E of the paper) in
// one cooperative kernel whose blocks are all resident, with a grid-wide
// barrier wherever a pass needs the one before:
//
//   points per cell (maps with the wall rule), thresholds and coarse grids
//   | points: gate, sums, ray march (blocks take runs from the work counter); for
//   |   scattered points in parts, the thresholds refreshed between them
//   | new state of the table's cells (maps beyond kFlatCells)
//   | new state of every cell, removal of marked cells, overlap clearance
//
// The stencils (normals, smoothing, in-painting) follow as their own kernels.
// The passes share one shared-memory buffer; each one ends with a block
// barrier, so the next pass of the same block never writes into it early.
// A barrier hands out tickets from one counter: barrier j of a launch holds
// tickets [j nb, (j + 1) nb), and a block waits until the counter reaches the
// end of its barrier's range.  The last block to finish the launch sets the
// counter back to zero.  Every wait is bounded by a clock64 budget: a wait
// that runs out raises the abort flag, writes EM_ERR_TIMEOUT into the maps'
// error words, and every block leaves at its next barrier; the last one to leave
// then clears the update's scratch, so the next update starts as after a whole one.
#include "cell_pass.cuh"
#include "em.h"
#include "point_pass.cuh"

namespace em {

constexpr int kPersistThreads = 256;
static_assert(kPersistThreads == kPointThreads && kPersistThreads == kCellThreads, "the passes share one block size");

constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }
// the passes run one after another and share one shared-memory buffer
constexpr size_t kPersistSmem = cmax(sizeof(PointsSmem<true>), sizeof(PreSmem));
constexpr size_t kPersistAlign = 32;
static_assert(kPersistAlign >= alignof(PointsSmem<true>) && kPersistAlign >= alignof(PreSmem),
              "the buffer starts where the passes' structs may");

// Wait until *word >= target, or until `abort` is raised, for at most budget
// SM clock cycles; true when the word got there.
__device__ __forceinline__ bool wait_at_least(const unsigned long long* word, unsigned long long target,
                                              const int* abort, long long budget) {
  const long long t0 = clock64();
  while (*(const volatile unsigned long long*)word < target) {
    if ((abort && *(const volatile int*)abort) || clock64() - t0 > budget) return false;
    __nanosleep(100);
  }
  return true;
}

// Barrier of all nb blocks of the launch; false when this block should leave.
__device__ __forceinline__ bool grid_barrier(const BatchDev& b, int nb, long long budget, int& s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    BatchCtl* c = b.ctl;
    __threadfence();  // this block's writes before its arrival
    const unsigned long long t = atomicAdd(&c->bar_ticket, 1ull);
    const unsigned long long target = (t / (unsigned long long)nb + 1ull) * (unsigned long long)nb;
    bool ok = wait_at_least(&c->bar_ticket, target, &c->bar_abort, budget);
    if (!ok && atomicExch(&c->bar_abort, 1) == 0) {  // the first block to give up records it
      for (int mi = 0; mi < b.n_maps; ++mi) atomicCAS(&b.maps[mi].ctl->err, 0, kErrTimeout);
    }
    __threadfence();  // the other blocks' writes before this block goes on
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <int G, bool kExt>
__global__ void __launch_bounds__(kPersistThreads, 4) k_persist(const BatchDev* __restrict__ bp) {
  extern __shared__ __align__(kPersistAlign) unsigned char sm[];
  __shared__ int s_ok;
  begin_after_previous();
  const BatchDev& b = *bp;
  const long long budget = b.wait_budget;
  const int nb = gridDim.x, bid = blockIdx.x;
  const Grid all{bid, nb};
  bool ok = true;
  if (b.passes & (kPassPre | kPassCells)) {
    if (b.passes & kPassPre) pre_pass<kExt>(b, all, *reinterpret_cast<PreSmem*>(sm));
    if (b.passes & kPassCells) cells_pass(b, all);
    ok = grid_barrier(b, nb, budget, s_ok);
  }
  const int parts = ok && in_parts(b) ? kParts : 1;  // (the same for every block)
  for (int i = 0; ok && i < parts; ++i) {
    if (i > 0) {
      refresh_pass(b, all);
      ok = grid_barrier(b, nb, budget, s_ok);
      if (!ok) break;
    }
    points_pass<G, true, kExt>(b, all, i, *reinterpret_cast<PointsSmem<true>*>(sm));
    ok = grid_barrier(b, nb, budget, s_ok);
  }
  if (ok && b.tab.slots) {
    sums_pass(b, all);
    ok = grid_barrier(b, nb, budget, s_ok);
  }
  if (ok) write_pass(b, all);
  // the last block to leave makes the barrier state ready for the next launch; when a
  // wait ran out, some blocks left before their share of the sums, the marks and
  // write_pass, so it also clears what those passes hand on
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_ok = atomicAdd(&b.ctl->bar_done, 1) == nb - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s_ok) return;
  if (*(const volatile int*)&b.ctl->bar_abort) clear_scratch(b);
  __syncthreads();  // (every thread has read the abort flag)
  if (threadIdx.x == 0) {
    b.ctl->bar_ticket = 0ull;
    b.ctl->bar_done = 0;
    b.ctl->bar_abort = 0;
    __threadfence();
  }
}

__global__ void k_wait_selftest(const unsigned long long* word, int* timed_out, long long budget) {
  if (threadIdx.x == 0) *timed_out = wait_at_least(word, 1ull, nullptr, budget) ? 0 : 1;
}

long long clock_budget(long long us) {
  int dev = 0, khz = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) != cudaSuccess || khz <= 0) khz = 2000000;
  return (long long)khz * us / 1000;
}

namespace {

template <int G, bool kExt>
Launch persist_launch_t() {
  // per device, once: the shared-memory limit above the static 48 KB, and the
  // blocks that fit at once (the cooperative launch needs all of them resident)
  static int per_sm[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return {};
  const void* fn = (const void*)&k_persist<G, kExt>;
  int& n = per_sm[dev];
  if (n == 0) {
    int v = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPersistSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, fn, kPersistThreads, kPersistSmem) != cudaSuccess) {
      cudaGetLastError();
      return {};
    }
    n = v > 0 ? v : -1;
  }
  if (n < 0) return {};
  return {fn, (unsigned)(n * sm_count()), kPersistThreads, kPersistSmem, true, EM_PROF_PERSIST, "k_persist", 0};
}

template <bool kExt>
Launch persist_launch_g(int g) {
  switch (g) {
    case 1: return persist_launch_t<1, kExt>();
    case 2: return persist_launch_t<2, kExt>();
    case 4: return persist_launch_t<4, kExt>();
    case 16: return persist_launch_t<16, kExt>();
    case 32: return persist_launch_t<32, kExt>();
    default: return persist_launch_t<8, kExt>();
  }
}

}  // namespace

Launch persist_launch(int group, bool ext) { return ext ? persist_launch_g<true>(group) : persist_launch_g<false>(group); }

cudaError_t launch_wait_selftest(const unsigned long long* word, int* timed_out, int wait_us, cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(word, timed_out, clock_budget(wait_us));
  return cudaGetLastError();
}

}  // namespace em
