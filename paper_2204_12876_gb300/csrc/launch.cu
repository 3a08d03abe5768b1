// launch.cu -- the kernels of an update as a list of launches: the per-map,
// batched and allocation-free forms run the same list, on a stream or as a graph.
#include "em.h"
#include "em_internal.cuh"

namespace em {

Sequence update_sequence(const UpdateKind& k, int64_t n_points, int64_t n_cells) {
  Sequence q;
  // EM_BATCH_PERSISTENT: the passes in one launch (k_persist.cu), when the device
  // can run it and no map needs the drift compensation
  const Launch p = k.persistent && !k.drift ? persist_launch(k.ray_group, k.ext) : Launch{};
  if (p.fn) {
    q.add(p);
  } else {
    if (k.wall || k.drift) q.add(pre_launch(n_points, k.ext));
    if (k.ray || k.drift) q.add(cells_launch(n_cells));
    const int parts = k.ray && n_points >= (int64_t)kSplitPoints ? kParts : 1;
    for (int i = 0; i < parts; ++i) {
      if (i > 0) q.add(refresh_launch(n_cells));
      q.add(points_launch(n_points, k.ray_group, k.ray, k.ext, i));
    }
    q.add(write_launch(n_cells));
  }
  if (k.stencils & EM_F_NORMALS) q.add(normals_launch(n_cells));
  if (k.stencils & (EM_F_SMOOTH | EM_F_MEDIAN | EM_F_GAUSS)) q.add(smooth_launch(n_cells));
  if (k.stencils & EM_F_INPAINT) q.add(inpaint_launch(n_cells));
  return q;
}

cudaError_t run(const Launch& l, const BatchDev* b, cudaStream_t s) {
  void* args[] = {(void*)&b, (void*)&l.part};  // (a kernel takes as many as it has parameters)
  return l.coop ? cudaLaunchCooperativeKernel(l.fn, dim3(l.grid), dim3(l.block), args, l.smem, s)
                : cudaLaunchKernel(l.fn, dim3(l.grid), dim3(l.block), args, l.smem, s);
}

// Nodes are added one by one instead of captured from a stream: a capture can be
// broken by any other thread of the process that synchronises the device.
cudaError_t build_graph(const Sequence& q, const BatchDev* b, cudaGraph_t* out) {
  *out = nullptr;
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaGraphCreate(&g, 0);
  cudaGraphNode_t prev = nullptr;
  for (int i = 0; i < q.n && e == cudaSuccess; ++i) {
    const Launch& l = q.k[i];
    void* args[] = {(void*)&b, (void*)&l.part};
    cudaKernelNodeParams p = {};
    p.func = const_cast<void*>(l.fn);
    p.gridDim = dim3(l.grid);
    p.blockDim = dim3(l.block);
    p.sharedMemBytes = (unsigned)l.smem;
    p.kernelParams = args;
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddKernelNode(&node, g, prev ? &prev : nullptr, prev ? 1 : 0, &p);
    if (e == cudaSuccess && l.coop) {
      cudaKernelNodeAttrValue v = {};
      v.cooperative = 1;
      e = cudaGraphKernelNodeSetAttribute(node, cudaKernelNodeAttributeCooperative, &v);
    }
    prev = node;
  }
  if (e != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return e;
  }
  *out = g;
  return cudaSuccess;
}

}  // namespace em
