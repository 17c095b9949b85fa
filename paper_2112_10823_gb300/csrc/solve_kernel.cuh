// The persistent kernel of a single-system solve.  One translation unit per
// value and column type instantiates its variants (solve_*.cu), so that they
// compile side by side.
#pragma once
#include "cg_solve.cuh"

namespace cgk {

// One system on the whole grid: CTA c is rank c of the group.  kJacobi:
// preconditioned by M = diag(A) (P.dinv).  C: type of the stored columns.
template <bool kMixed, bool kJacobi, bool kSmallShare, typename C>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
    cg_solve_kernel(const __grid_constant__ SolveParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // the step loop streams FP32 values in the mixed solve
  using Ring = RingSmem<std::conditional_t<kMixed, float, double>, C>;
  const Ring sm{smem_raw};
  __shared__ TaskState task;
  ring_init(sm);
  task_load(&task, P, blockIdx.x);
  if (threadIdx.x >= kBlock) {
    if (producer(sm, P.A, blockIdx.x, false, P.A.keep != 0, P.wait_limit_ns) != kStreamDone) solve_fail(P, threadIdx.x == kBlock);
    return;
  }
  // the neighbour wait at the end of a step pays off on large shares (160^3:
  // 1.6 % faster); on small ones the group barrier is faster (64^3: 1 %, 16^3: 9 %)
  solve_task<kMixed, kJacobi, kSmallShare, !kSmallShare>(sm, &task, P.stream_rows);
  stop_producer(sm);
}

template <bool kMixed, typename C>
const void* solve_kernel_of(bool jacobi, bool small) {
  if (jacobi)
    return small ? reinterpret_cast<const void*>(cg_solve_kernel<kMixed, true, true, C>)
                 : reinterpret_cast<const void*>(cg_solve_kernel<kMixed, true, false, C>);
  return small ? reinterpret_cast<const void*>(cg_solve_kernel<kMixed, false, true, C>)
               : reinterpret_cast<const void*>(cg_solve_kernel<kMixed, false, false, C>);
}

}  // namespace cgk
