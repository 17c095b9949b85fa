// CSR product and the persistent conjugate-gradient solves.
//
// Classical CG (the paper's Sec. 5.3 solver; no preconditioner), one
// cooperative launch per solve (or, batched, per set of systems):
//   setup     r = b - A x, p = r, rho = r.r, ||b||^2          (product + 2 sums)
//   each step q = A p, gamma = p.q                            (product fused with the sum)
//             alpha = rho/gamma; r -= alpha q, rho' = r.r     (update fused with the sum)
//             stop if sqrt(rho') <= tol ||b||
//             beta = rho'/rho; x += alpha p; p = r + beta p   (x update deferred here)
//   exit      ||b - A x|| / ||b||                             (true residual)
// alpha, beta and the stopping test are computed on the device by every CTA
// from the same deterministic sums, so no host synchronisation happens per
// step and every CTA takes the same branch.  Each CTA owns a fixed range of
// rows (a run of product steps) for all phases, so only the two sums and the
// gather of p need synchronisation across the CTAs that share the system: two
// sums through accumulators (or the group barrier, see acc_words) and one barrier
// or neighbour wait per step.  A single-system solve uses the whole grid
// as one group; a batched solve gives each system its own group of CTAs (one
// CTA for most systems) and lets CTAs take systems from a queue.
//
// The mixed-precision variant keeps an FP32 copy of the values and an FP32
// shadow of p: the product is FP32 (FP32 accumulation); sums, alpha, beta, x
// and r stay FP64; every `replace_every` steps, and before accepting
// convergence, r is replaced by the FP64 true residual b - A x.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <set>
#include <utility>
#include "cg_device.cuh"

namespace cgk {

// y = A x (same partition and stream as the solve; one pass, every table read
// once: evict-first).
template <typename C>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
    spmv_kernel(const __grid_constant__ DevCsr A, const double* x, double* y, int32_t* err) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using Ring = RingSmem<double, C>;
  const Ring sm{smem_raw};
  ring_init(sm);
  const unsigned long long lim = 2000000000ull;
  if (threadIdx.x >= kBlock) {
    if (producer(sm, A, blockIdx.x, true, A.keep != 0, lim) != kStreamDone && threadIdx.x == kBlock) atomicExch(err, kETIMEOUT);
    return;
  }
  const int bw = blockIdx.x * kWarps + (threadIdx.x >> 5);
  const int s = A.warp_step[bw], s1 = A.warp_step[bw + 1];
  const PassIo io = pass_io(A, 1, nullptr, y, lim);
  load_first_steps(sm, io, s, s1);
  if (threadIdx.x == 0) sm.state()->io = io;
  cta_sync();
  ring_pass<Ring>(smem_raw, s, s1, x, false);
  if ((threadIdx.x & 31) == 0 && sm.stream(threadIdx.x >> 5)->failed) {
    atomicExch(err, kETIMEOUT);
    *reinterpret_cast<volatile int32_t*>(sm.stop()) = 1;
  }
}

// The same of a mixed-precision handle, whose streams hold FP32 values: its FP64
// values directly from global memory, a warp per step.  What bounds it is the
// latency of a step's chain (step, columns, x, FMAs), so as many warps as 64
// registers allow (32 per SM) work on steps of their own, in small blocks, whose
// warps give way to the next steps at once (blocks of 64, 128, 256 threads: Q1
// 160^3 232, 238, 250 us; 48 registers spill: 267).  Q1 64^3 20.8 us, 160^3 232;
// the former CSR ring 25.0 and 239, a warp per stream (19 per SM) 27.1 and 350.
constexpr int kDirectThreads = 64, kDirectBlocks = 16;

template <typename C, bool kKeep>
__global__ void __launch_bounds__(kDirectThreads, kDirectBlocks)
    spmv_direct_kernel(const __grid_constant__ DevCsr A, const double* x, double* y) {
  using Ring = RingSmem<float, C>;
  const int64_t s = (static_cast<int64_t>(blockIdx.x) * kDirectThreads + threadIdx.x) >> 5;
  if (s >= A.nsteps) return;
  direct_pass<Ring, kKeep>(A, A.step_chunk[s], A.step_entry[s], static_cast<int>(s), static_cast<int>(s) + 1, x,
                    y);
}

// Opt a kernel in to `bytes` of dynamic shared memory, and ask for the
// smallest shared-memory carveout that holds them (the rest of the SM's
// 256 KB serves as L1 for the product's gathers), once per (kernel, device).
cudaError_t ensure_smem_attr(const void* kernel, size_t bytes) {
  static std::mutex mu;
  static std::set<std::pair<const void*, int>> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (done.count({kernel, dev})) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  int max_sm = 0;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&max_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess && max_sm > 0) {
    // a hint: CUDA picks the nearest supported carveout that the launch fits in
    const size_t need = bytes + 1024;  // + the CTA's reserved shared memory
    int pct = static_cast<int>((need * 100 + static_cast<size_t>(max_sm) - 1) / static_cast<size_t>(max_sm));
    if (pct > 100) pct = 100;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
  }
  if (e == cudaSuccess) done.insert({kernel, dev});
  return e;
}

cudaError_t launch_spmv(const DevCsr& A, const double* x, double* y, int32_t* err, cudaStream_t s) {
  if (A.val64 != nullptr) {
    const unsigned blocks = static_cast<unsigned>((static_cast<int64_t>(A.nsteps) * 32 + kDirectThreads - 1) / kDirectThreads);
    auto run = [&](auto kernel) { kernel<<<blocks, kDirectThreads, 0, s>>>(A, x, y); };
    if (A.keep) A.col16 ? run(spmv_direct_kernel<uint16_t, true>) : run(spmv_direct_kernel<int32_t, true>);
    else A.col16 ? run(spmv_direct_kernel<uint16_t, false>) : run(spmv_direct_kernel<int32_t, false>);
    return cudaGetLastError();
  }
  const size_t smem = solve_smem_bytes(false, A.col16 != 0);
  const void* k = A.col16 ? reinterpret_cast<const void*>(spmv_kernel<uint16_t>)
                          : reinterpret_cast<const void*>(spmv_kernel<int32_t>);
  cudaError_t e = ensure_smem_attr(k, smem);
  if (e != cudaSuccess) return e;
  if (A.col16) spmv_kernel<uint16_t><<<A.nblocks, kThreads, smem, s>>>(A, x, y, err);
  else spmv_kernel<int32_t><<<A.nblocks, kThreads, smem, s>>>(A, x, y, err);
  return cudaGetLastError();
}

template <bool kMixed, typename C>
const void* solve_kernel_of(bool jacobi, bool small);  // solve_*.cu

const void* solve_kernel_ptr(bool mixed, bool jacobi, bool col16, bool small) {
  if (mixed) return col16 ? solve_kernel_of<true, uint16_t>(jacobi, small) : solve_kernel_of<true, int32_t>(jacobi, small);
  return col16 ? solve_kernel_of<false, uint16_t>(jacobi, small) : solve_kernel_of<false, int32_t>(jacobi, small);
}

size_t solve_smem_bytes(bool mixed, bool col16, bool local) {
  if (mixed) return col16 ? ring_smem_bytes<float, uint16_t>(local) : ring_smem_bytes<float, int32_t>(local);
  return col16 ? ring_smem_bytes<double, uint16_t>(local) : ring_smem_bytes<double, int32_t>(local);
}

int solve_blocks_per_sm(bool mixed, bool jacobi) {
  int nb = 1 << 20;
  for (const bool small : {false, true})  // every variant must fit (one CTA per SM)
    for (const bool col16 : {false, true}) {
      const void* k = solve_kernel_ptr(mixed, jacobi, col16, small);
      const size_t smem = solve_smem_bytes(mixed, col16, small);
      cudaError_t e = ensure_smem_attr(k, smem);
      int nk = 0;
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nk, k, kThreads, smem);
      if (e != cudaSuccess) return -1;
      nb = std::min(nb, nk);
    }
  return nb;
}

cudaError_t launch_solve(const SolveParams& P, bool mixed, cudaStream_t s) {
  void* args[] = {const_cast<SolveParams*>(&P)};
  // the small-share kernel: every CTA's rows fit its shared r, and the
  // solve runs in this one launch
  const bool small = small_share(P.A, P.chunk_iters), col16 = P.A.col16 != 0;
  const void* k = solve_kernel_ptr(mixed, P.dinv != nullptr, col16, small);
  const size_t smem = solve_smem_bytes(mixed, col16, small);
  cudaError_t e = ensure_smem_attr(k, smem);
  if (e != cudaSuccess) return e;
  return cudaLaunchCooperativeKernel(k, dim3(P.A.nblocks), dim3(kThreads), args, smem, s);
}

// dinv[i] = 1 / diag(A)_i (the diagonal summed over row i's entries in
// column i, in storage order); err <- first row (+1) without a positive one.
__global__ void jacobi_dinv_kernel(const CsrSource src, int64_t row0, int64_t row1, double* __restrict__ dinv,
                                   int32_t* err) {
  for (int64_t i = row0 + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < row1;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    double d = 0.0;
    for (int64_t k = src.row_ptr[i] - src.e_first; k < src.row_ptr[i + 1] - src.e_first; ++k)
      if (src.col_idx[k] - src.base == i) d += src.val[k];
    if (d > 0.0) {
      dinv[i] = 1.0 / d;
    } else {
      dinv[i] = 0.0;
      atomicCAS(err, 0, static_cast<int32_t>(i + 1));
    }
  }
}

cudaError_t launch_jacobi_dinv(const CsrSource& src, int64_t row0, int64_t row1, double* dinv, int32_t* err,
                               cudaStream_t s) {
  if (row1 <= row0) return cudaSuccess;
  const int64_t blocks = (row1 - row0 + 255) / 256;
  jacobi_dinv_kernel<<<static_cast<unsigned>(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(src, row0, row1, dinv, err);
  return cudaGetLastError();
}

// ---- self-test of the bounded wait: thread 0 of one CTA arrives at the
// group barrier of the solves (group_barrier_t0) for a group of two CTAs that
// no other CTA joins, so its wait must run out after limit_ns, raise the
// abort flag, record the site and report kETIMEOUT through the control block.
__global__ void wait_timeout_selftest_kernel(SolveCtrl* ctrl, unsigned long long limit_ns) {
  __shared__ unsigned long long target;
  if (threadIdx.x == 0) {
    target = 0;
    const bool ok = group_barrier_t0(ctrl, &target, 2u, limit_ns, kSelftestSite);
    ctrl->status = ok ? kOK : kETIMEOUT;
  }
}

cudaError_t launch_wait_timeout_selftest(SolveCtrl* ctrl, unsigned long long limit_ns, cudaStream_t s) {
  wait_timeout_selftest_kernel<<<1, 32, 0, s>>>(ctrl, limit_ns);
  return cudaGetLastError();
}

// ---- cost of the solves' group-wide synchronisations on the whole grid
// (one CTA per SM, the solve kernel's block): `iters` times, between CTA
// barriers as in a solve step, warp 0 of every CTA either meets the others at
// the group barrier (mode 0: group_barrier_t0), or runs a group sum (mode 1:
// publishes the CTA's value in one of two alternating slots, meets the others
// at the barrier, and sums the group's values exactly with fx_warp_sum_array: the
// general form of the solves' group_sum; the sums of a step usually go through
// the accumulators, which it does not time).  The waits are the
// solves' bounded ones: a wait that gives up raises ctrl->abort, after which
// every CTA stops.  out[rank] keeps the sums live.
__global__ void __launch_bounds__(kBlock, kCtasPerSm)
    sync_probe_kernel(SolveCtrl* ctrl, double* partials, int iters, int mode, unsigned long long limit_ns,
                      double* out) {
  __shared__ unsigned long long target;
  __shared__ int ok;
  __shared__ double total;
  const int nb = static_cast<int>(gridDim.x), rank = static_cast<int>(blockIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    target = 0;
    ok = 1;
    total = 0.0;
  }
  __syncthreads();
  double acc = 0.0;
  for (int k = 0; k < iters; ++k) {
    if (warp == 0) {
      double* part = partials + static_cast<size_t>(k & 1) * nb;
      int good = 1;
      if (lane == 0) {
        if (mode == 1) part[rank] = static_cast<double>(rank + k);
        good = group_barrier_t0(ctrl, &target, static_cast<unsigned int>(nb), limit_ns, kProbeSite) ? 1 : 0;
      }
      good = __shfl_sync(0xffffffffu, good, 0);
      if (good && mode == 1) {
        const double sum = fx_warp_sum_array(part, nb);
        if (lane == 0) total = sum;
      }
      if (lane == 0 && !good) ok = 0;
    }
    __syncthreads();
    if (!ok) break;
    acc += total;
    __syncthreads();  // total is rewritten by the next sum
  }
  if (threadIdx.x == 0) out[rank] = acc;
}

cudaError_t launch_sync_probe(SolveCtrl* ctrl, double* partials, int iters, int mode, int nblocks,
                              unsigned long long limit_ns, double* out, cudaStream_t s) {
  void* args[] = {&ctrl, &partials, &iters, &mode, &limit_ns, &out};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(sync_probe_kernel), dim3(nblocks), dim3(kBlock),
                                     args, 0, s);
}

}  // namespace cgk
