// em_host.h -- host-side internals shared by the translation units of libem.so
// (the map object itself stays private to em_api.cu).
#pragma once

#include <cuda_runtime.h>

#include "em.h"
#include "em_internal.cuh"

namespace em {

int map_device(const em_map* m);
uint32_t map_flags(const em_map* m);
int32_t map_cells(const em_map* m);
const em_params& map_params(const em_map* m);
// The passes an update of a map with these parameters needs.
UpdateKind params_kind(const em_params& p, int32_t ray_group);
UpdateKind map_kind(const em_map* m, int32_t ray_group);

// Start one update of map m: advances its update index and returns its
// device descriptor (pt_begin / pt_count are left to the caller).
MapDev map_begin_update(em_map* m, int64_t points);
void map_end_update(em_map* m, cudaStream_t s, int64_t points);
void map_undo_update(em_map* m, int64_t points);

// An update of map m failed after some of its kernels were launched: its scratch
// (sums, marks, counters) may not be zero.  map_clean clears it before the next
// update, on that update's stream; nothing to do otherwise.
void map_set_dirty(em_map* m);
int map_clean(em_map* m, cudaStream_t s);

// One update of map m from at most kDescClouds clouds (checked by the caller),
// total points, as a batch of that map alone does it (no trace, no profiling).
int map_update_one(em_map* m, const em_cloud* clouds, int32_t n_clouds, int64_t total, cudaStream_t s);

// Can an update of that many points of this map run without allocating?
bool map_has_room(const em_map* m, int64_t points);

// Device memory of a table of sums, zeroed; cnt only when the wall rule may count.
cudaError_t table_alloc(SumTable* t, int64_t slots, bool cnt, int64_t* bytes);
void table_free(SumTable* t);
cudaError_t table_clear(const SumTable& t, cudaStream_t s);

// Copy layers, ring offsets, shift and update index of src into dst (same size).
int map_copy_state(em_map* dst, const em_map* src, cudaStream_t s);

// Write the layers in mask (em_get_layers layout) to dst, a pointer the device
// can write (device memory or mapped page-locked host memory), on stream s.
int map_read_layers(em_map* m, uint32_t mask, float* dst, cudaStream_t s);
// The same for n maps, kMaxReadJobs per launch.
int maps_read_layers(em_map* const* maps, const uint32_t* masks, float* const* dst, int n, cudaStream_t s);

// Record a CUDA error for em_last_cuda_error() and map it to a status code.
int map_record_error(const char* what, cudaError_t e);

}  // namespace em
