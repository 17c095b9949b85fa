// The batched persistent solve: many systems in one cooperative launch.
// Each CTA takes tasks (a system and its rank in the system's group of CTAs)
// from a queue; the CG arithmetic of every task is the single-system solve's
// (cg_solve.cuh).  One translation unit per value type instantiates the kernel
// (batch_*.cu).
#pragma once
#include "cg_solve.cuh"

namespace cgk {

// A task of the computing warps or of the producer warp; false if the ring did
// not drain in time (a task that ended in a timeout has drained it all the same).
template <bool kMixed, bool kJacobi, typename C>
__device__ __noinline__ bool batch_task(unsigned char* smem, const TaskState* tk, int32_t stream_rows, int32_t keep) {
  using T = std::conditional_t<kMixed, float, double>;
  using Ring = RingSmem<T, C>;
  const Ring sm{smem};
  if (threadIdx.x >= kBlock) {
    const int end = producer(sm, tk->P.A, tk->rank, false, keep != 0, tk->P.wait_limit_ns);
    if (end != kStreamDone) solve_fail(tk->P, threadIdx.x == kBlock);
    return end != kStreamLost;
  }
  solve_task<kMixed, kJacobi, false, false>(sm, tk, stream_rows);
  stop_producer(sm);
  return true;
}

// Many systems in one persistent launch: each CTA takes tasks (a system and
// its rank in the system's group) from the queue, in queue order, until it is
// empty.  The host orders the queue longest estimated time per CTA first,
// with a group's ranks next to each other; a group's first ranks wait at its
// first group barrier until CTAs that free up have taken the rest.  Between
// tasks the whole CTA joins, every warp's ring drained; a CTA whose ring did
// not drain in time takes no more.
template <bool kMixed, bool kJacobi>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
    cg_batch_kernel(const __grid_constant__ BatchParams B) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int32_t task_id;
  __shared__ TaskState task;
  using T = std::conditional_t<kMixed, float, double>;
  ring_init(RingSmem<T, int32_t>{smem_raw});
  for (;;) {
    if (threadIdx.x == 0) task_id = atomicAdd(B.next, 1);
    __syncthreads();
    const int t = task_id;
    if (t >= B.queue->ntasks) break;
    const BatchTask tk = B.queue->task[t];
    ring_reset(RingSmem<T, int32_t>{smem_raw});
    task_load(&task, B.sys[tk.sys], tk.rank);
    const int32_t stream_rows = B.queue->stream_rows, keep = B.queue->keep;
    const bool drained = task.P.A.col16 ? batch_task<kMixed, kJacobi, uint16_t>(smem_raw, &task, stream_rows, keep)
                                       : batch_task<kMixed, kJacobi, int32_t>(smem_raw, &task, stream_rows, keep);
    if (!__syncthreads_and(drained)) break;
  }
}

template <bool kMixed>
const void* batch_kernel_of(bool jacobi) {
  return jacobi ? reinterpret_cast<const void*>(cg_batch_kernel<kMixed, true>)
                : reinterpret_cast<const void*>(cg_batch_kernel<kMixed, false>);
}

}  // namespace cgk
