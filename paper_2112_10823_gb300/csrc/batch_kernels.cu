// Launch of the batched persistent solve (batch_kernel.cuh).
#include <algorithm>
#include "cg_internal.h"

namespace cgk {

template <bool kMixed>
const void* batch_kernel_of(bool jacobi);  // batch_f64.cu, batch_mixed.cu

const void* batch_kernel_ptr(bool mixed, bool jacobi) {
  return mixed ? batch_kernel_of<true>(jacobi) : batch_kernel_of<false>(jacobi);
}

// A batch may hold systems of both column widths: room for either ring.
size_t batch_smem_bytes(bool mixed) {
  return std::max(solve_smem_bytes(mixed, false), solve_smem_bytes(mixed, true));
}

int batch_blocks_per_sm(bool mixed, bool jacobi) {
  int nb = 0;
  const void* k = batch_kernel_ptr(mixed, jacobi);
  const size_t smem = batch_smem_bytes(mixed);
  cudaError_t e = ensure_smem_attr(k, smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, kThreads, smem);
  return e == cudaSuccess ? nb : -1;
}

// Cooperative launch (all CTAs co-resident: the ranks of a group wait on
// each other), through cudaLaunchKernelEx so that it can be captured in a
// CUDA graph.
cudaError_t launch_batch(const BatchParams& B, bool mixed, bool jacobi, int nblocks, cudaStream_t s) {
  const void* k = batch_kernel_ptr(mixed, jacobi);
  const size_t smem = batch_smem_bytes(mixed);
  cudaError_t e = ensure_smem_attr(k, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nblocks);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  void* args[] = {const_cast<BatchParams*>(&B)};
  return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace cgk
