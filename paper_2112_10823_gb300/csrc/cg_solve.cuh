// The CG solve body shared by the single-system and the batched kernels:
// one CTA's share of one
// system, its matrix streamed by every warp for itself.
#pragma once
#include <cmath>
#include "cg_device.cuh"

namespace cgk {

// Leave the solve after a failed wait: record the status (thread 0 of the
// computing warps; lane 0 of the producer warp).  Waits on other CTAs have
// recorded their site; the others are the matrix stream's.
__device__ __forceinline__ void solve_fail(const SolveParams& P, bool first) {
  if (first) {
    if (atomicExch(&P.ctrl->abort, 1) == 0) atomicCAS(&P.ctrl->timeout_site, 0, kStreamSite);
    atomicExch(&P.ctrl->status, kETIMEOUT);
    atomicExch(&P.ctrl->phase, kPhaseDone);
  }
  __syncwarp();
}

// Systems whose CTAs hold at most kLocalRows rows each (small, L2-resident
// shares), solved in one launch, use the small-share kernels: r of the CTA's
// rows lives in shared memory (only the owning CTA ever reads it; three
// accesses per step), and x is updated behind the barrier of the r.r sum,
// where the wait is longer than the update.  Larger shares keep r in global
// memory and update x together with p (one pass over p).  Both compute the
// same bits.

// Rows per thread in flight in the vector phases (all loads of a batch
// issued before any is used): as many as the registers that the product
// leaves allow without spilling (96 per thread at 20 warps per CTA; the
// Jacobi variants carry dinv as well, the fused x and p update three vectors).
template <bool kJacobi, bool kSmallShare>
__host__ __device__ constexpr int vec_rows() {
  return kSmallShare ? (kJacobi ? 3 : 4) : (kJacobi ? 2 : 3);
}

// What a solve task needs, in shared memory: the phases of a step read it from
// there, so that nothing but a few indices stays in registers across the
// product, whose registers are then its own.
struct TaskState {
  SolveParams P;
  int32_t rank;
  int32_t row0, row1;  // the CTA's rows
  int32_t warp_step[kWarps + 1];
};

// Copies the parameters of a task into shared memory (all threads of the CTA
// call; ends with a CTA barrier).
__device__ __forceinline__ void task_load(TaskState* tk, const SolveParams& P, int rank) {
  static_assert(sizeof(SolveParams) % 4 == 0 && sizeof(SolveParams) / 4 <= kBlock, "a word per thread");
  if (threadIdx.x < sizeof(SolveParams) / 4)
    reinterpret_cast<uint32_t*>(&tk->P)[threadIdx.x] = reinterpret_cast<const uint32_t*>(&P)[threadIdx.x];
  if (threadIdx.x <= kWarps) tk->warp_step[threadIdx.x] = P.A.warp_step[rank * kWarps + threadIdx.x];
  if (threadIdx.x == 0) {
    tk->rank = rank;
    tk->row0 = P.A.block_row[rank];
    tk->row1 = P.A.block_row[rank + 1];
  }
  __syncthreads();
}

// A solve task: share `rank` (of P.group CTAs) of the CG
// iteration on one system, from its start or from the state a previous
// launch saved, for at most P.chunk_iters steps.  kSmallShare: the small-share
// kernel (above): r in shared memory, x updated by warps 1.. behind the
// barrier of the r.r sum; it runs a solve in one launch.
//
// Scalars live in the CTA state in shared memory (thread 0 updates them
// between CTA barriers; every thread reads them after one).
//
// The computing warps call this while the producer warp runs the CTA's stream,
// and stop it afterwards, whichever way this returns.
template <bool kMixed, bool kJacobi, bool kSmallShare, bool kNeighborWait, typename Ring>
__device__ __forceinline__ void solve_task(const Ring& sm, const TaskState* const tk, const int32_t stream_rows) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SolveParams& P = tk->P;
  // kNeighborWait: the single-system kernel for large shares (P.flags set
  // when the group has several CTAs); the small-share and batched kernels
  // always use the group barrier.
  auto neighbor = [&] { return kNeighborWait && P.flags != nullptr; };
  CtaState* const st = sm.state();
  SumScratch* const ss = sm.sums();
  constexpr int kVR = vec_rows<kJacobi, kSmallShare>();

  // Group-wide sum of nv values per thread (nv <= 3), fused with the vote of
  // the computing warps (`ok`: this thread's waits all succeeded).  Each warp
  // sums its lanes exactly in fixed point; warp 0 combines the warps and sums
  // the group's CTA values, exactly and order-independently, so that every CTA
  // gets the same bits: through the accumulators slot, slot + 1, .. (slot >= 0:
  // the sums of a step, see acc_words), or in the general form: it publishes the
  // CTA's values, meets the other CTAs of the group at the barrier and sums the
  // values in fixed point.  Lane 0 then runs fin(sums), which updates the CTA
  // state; one CTA barrier publishes it.  In the general form two slots of
  // partials (3 nb values each) alternate so that a fast CTA publishing the next
  // sum never overwrites values a slow CTA still reads.
  // `side()` runs in warps 1.. while warp 0 does this: work of the step that
  // needs no group-wide value yet, hidden behind the wait.
  // Returns false in every thread if a wait gave up, here or anywhere before.
  auto group_sum = [&](bool ok, int nv, double v0, double v1, double v2, int slot, auto&& fin, auto&& side) -> bool {
    const double vin[kMaxSumValues] = {v0, v1, v2};
    FxPart fp[kMaxSumValues];
#pragma unroll
    for (int j = 0; j < kMaxSumValues; ++j)
      if (j < nv) fp[j] = fx_warp(vin[j]);
    const bool wok = __all_sync(0xffffffffu, ok);
    if (lane == 0) {
#pragma unroll
      for (int j = 0; j < kMaxSumValues; ++j)
        if (j < nv) ss->part[j][warp] = fp[j];
      ss->ok[warp] = wok ? 1 : 0;
    }
    cta_sync();
    if (warp == 0) {
      const bool valid = lane < kWarps;
      bool good = __all_sync(0xffffffffu, valid ? ss->ok[lane] != 0 : true);
      FxPart cp[kMaxSumValues];
#pragma unroll
      for (int j = 0; j < kMaxSumValues; ++j)
        if (j < nv) cp[j] = fx_combine(valid ? ss->part[j][lane] : FxPart{0, 0, 0}, valid);
      double sum[kMaxSumValues] = {0.0, 0.0, 0.0};
      const int nb = P.group, rank = tk->rank;
      bool summed = false;
      if (good && nb > 1 && slot >= 0) {
        // lane j: value j
        const int j = slot + lane;
        FxPart mine = cp[0];
        if (nv > 1 && lane == 1) mine = cp[1];
        const int eb = lane < nv ? st->acc_exp[j] : 1;
        if (__all_sync(0xffffffffu, eb != 0)) {
          bool in = true;
          double v = 0.0;
          if (lane < nv) {
            unsigned long long* const word = P.ctrl->acc[j];
            unsigned long long lo, hi;
            acc_words(mine, eb, &lo, &hi);
            asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(lo) : "memory");
            asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(word + 1), "l"(hi) : "memory");
            const unsigned long long lo0 = st->acc_seen[j][0], hi0 = st->acc_seen[j][1];
            good = acc_wait(P.ctrl, word, lo0, hi0, static_cast<unsigned int>(nb), P.wait_limit_ns, &lo, &hi);
            st->acc_seen[j][0] = lo;
            st->acc_seen[j][1] = hi;
            in = acc_sum(lo - lo0, hi - hi0, static_cast<unsigned int>(nb), eb, &v);
            if (in) st->acc_exp[j] = acc_exponent(v);
          }
          good = __all_sync(0xffffffffu, good);
          summed = __all_sync(0xffffffffu, in);
#pragma unroll
          for (int q = 0; q < 2; ++q) sum[q] = __shfl_sync(0xffffffffu, v, q);
        }
      }
      if (good && !summed) {
#pragma unroll
        for (int j = 0; j < kMaxSumValues; ++j)
          if (j < nv) sum[j] = fx_value(cp[j]);
        if (nb > 1) {
          const int ps = st->slot;
          double* part = P.partials + static_cast<size_t>(ps) * kMaxSumValues * nb;
          int bar_ok = 1;
          if (lane == 0) {
#pragma unroll
            for (int j = 0; j < kMaxSumValues; ++j)
              if (j < nv) part[j * nb + rank] = sum[j];
            bar_ok = group_barrier_t0(P.ctrl, &st->target, static_cast<unsigned int>(nb), P.wait_limit_ns, ++st->site);
          }
          good = __shfl_sync(0xffffffffu, bar_ok, 0) != 0;
          __syncwarp();
          if (good) {
#pragma unroll
            for (int j = 0; j < kMaxSumValues; ++j)
              if (j < nv) sum[j] = fx_warp_sum_array(part + j * nb, nb);
            if (lane == 0) st->slot = ps ^ 1;
          }
          if (slot >= 0 && lane < nv) st->acc_exp[slot + lane] = acc_exponent(lane == 0 ? sum[0] : sum[1]);
        }
      }
      if (lane == 0) {
        st->ok = good ? 1 : 0;
        if (good) fin(sum);
      }
    } else {
      side();
    }
    cta_sync();
    return st->ok != 0;
  };
  auto no_side = [] {};
  // Group barrier of all threads: every write before it is visible to every
  // CTA of the group after it.
  auto group_sync = [&]() -> bool {
    cta_sync();
    if (tid == 0)
      st->ok =
          group_barrier_t0(P.ctrl, &st->target, static_cast<unsigned int>(P.group), P.wait_limit_ns, ++st->site) ? 1 : 0;
    cta_sync();
    return st->ok != 0;
  };
  // End of a step in a single-system solve (P.flags set): instead of a group
  // barrier, the CTA publishes this step's number in its epoch flag once its
  // p is written (release pattern as in the group barrier) and waits until
  // the CTAs that own the columns its rows reach (ranks dep_lo..dep_hi) have
  // published the same step: the next product gathers p only from them.
  // Reusing p in place is safe: a CTA overwrites its p only once it has the step's
  // r.r, i.e. every CTA's arrival at that sum, and a CTA arrives only after its
  // p.q, whose value depends on every p that its product has gathered.  Those loads
  // have returned before the arrival is even computed, so no fence is needed
  // between them (in the general form of the sums the barrier has its fences).
  auto neighbor_sync = [&]() -> bool {
    cta_sync();
    if (warp == 0) {
      const int rank = tk->rank;
      SolveCtrl* const ctrl = P.ctrl;
      const unsigned long long epoch = static_cast<unsigned long long>(st->k);
      if (lane == 0) {
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(P.flags + rank), "l"(epoch) : "memory");
      }
      bool good = true;
      unsigned long long t0 = 0;
      uint32_t spins = 0;
      for (int q0 = st->dep_lo; q0 <= st->dep_hi && good; q0 += 32) {
        const int q = q0 + lane;
        if (q <= st->dep_hi && q != rank) {
          for (;;) {
            unsigned long long v;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(P.flags + q) : "memory");
            if (v >= epoch) break;
            if ((++spins & 255u) == 0) {
              if (*reinterpret_cast<const volatile int32_t*>(&ctrl->abort)) { good = false; break; }
              const unsigned long long now = global_timer_ns();
              if (t0 == 0) t0 = now;
              else if (now - t0 > P.wait_limit_ns) {
                atomicExch(&ctrl->abort, 1);
                atomicExch(&ctrl->timeout_site, kNeighborSite);
                good = false;
                break;
              }
            }
          }
        }
      }
      good = __all_sync(0xffffffffu, good);
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      if (lane == 0) st->ok = good ? 1 : 0;
    }
    cta_sync();
    return st->ok != 0;
  };
  // r_i of the CTA's rows: in shared memory in the small-share kernel
  auto residual = [&]() -> double* {
    if constexpr (kSmallShare) return sm.local() - tk->row0;
    else return P.r;
  };

  load_first_steps(sm, pass_io(P.A, 0, nullptr, nullptr, 0), tk->warp_step[warp], tk->warp_step[warp + 1]);
  // ---- state: saved by an earlier launch of this solve (written by another
  // kernel, so read through L2), or fresh
  if (tid == 0) {
    st->io = pass_io(P.A, stream_rows, P.p, P.q, P.wait_limit_ns);
    st->slot = 0;
    st->site = 0;
    st->ok = 1;
    st->flags = 0;
    st->target = 0;
    st->k = 0;
    st->pass = kPassSetup;
    const SolveCtrl* const ctrl = P.ctrl;
    for (int j = 0; j < 3; ++j) {  // (zero in a new solve)
      st->acc_seen[j][0] = __ldcg(&ctrl->acc_seen[j][0]);
      st->acc_seen[j][1] = __ldcg(&ctrl->acc_seen[j][1]);
      st->acc_exp[j] = __ldcg(&ctrl->acc_exp[j]);
    }
    if (__ldcg(&ctrl->phase) == kPhaseRunning) {
      st->target = __ldcg(&ctrl->rounds) * static_cast<unsigned long long>(P.group);
      st->slot = __ldcg(&ctrl->slot);
      st->rho = __ldcg(&ctrl->rho);
      st->bnorm2 = __ldcg(&ctrl->bnorm2);
      st->k = __ldcg(&ctrl->iters);
      const double rel = __ldcg(&ctrl->relres_rec);
      st->rr = rel * rel * st->bnorm2;  // reported only (the next step recomputes it)
      st->thresh2 = (P.tol * P.tol) * st->bnorm2;
      st->pass = kPassStep;
    }
    const long long k = st->k;
    st->k_end = P.chunk_iters > 0 && P.chunk_iters < P.maxit - k ? k + P.chunk_iters : P.maxit;
    st->dep_lo = 0x7fffffff;  // smallest and largest column of the CTA's rows, first
    st->dep_hi = -1;
  }
  cta_sync();
  if (neighbor()) {
    const DevCsr& A = P.A;
    // the CTAs whose p the product gathers: ranks owning the CTA's column range
    int cmin = 0x7fffffff, cmax = -1;
    for (int k = tk->warp_step[0] + tid; k < tk->warp_step[kWarps]; k += kBlock) {
      const int c = A.step_cmax[k];
      if (c >= 0) {
        cmin = min(cmin, A.step[k].w);
        cmax = max(cmax, c);
      }
    }
    cmin = static_cast<int>(__reduce_min_sync(0xffffffffu, static_cast<unsigned int>(cmin)));
    cmax = __reduce_max_sync(0xffffffffu, cmax);
    if (lane == 0) {
      atomicMin(&st->dep_lo, cmin);
      atomicMax(&st->dep_hi, cmax);
    }
    cta_sync();
    if (tid == 0) {
      auto owner = [&](int c) {  // the rank whose row range holds row c
        int lo = 0, hi = P.group - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (A.block_row[mid] <= c) lo = mid;
          else hi = mid - 1;
        }
        return lo;
      };
      if (st->dep_hi < 0) {  // no entries: nothing to wait for
        st->dep_lo = 1;
        st->dep_hi = 0;
      } else {
        st->dep_lo = owner(st->dep_lo);
        st->dep_hi = owner(st->dep_hi);
      }
    }
    cta_sync();
  }

  // One product per turn, q = A p in a step (with p.q) and q = A x in the other
  // passes: a single copy of the product's code, whatever it is for.
  for (;;) {
    const int pass = st->pass;
    const bool step = pass == kPassStep;
    double acc_g = 0.0;
    if constexpr (kMixed) {
      if (step) {
        acc_g = ring_pass<Ring>(sm.base, tk->warp_step[warp], tk->warp_step[warp + 1], P.p32, true);
      } else {
        const int bw = tk->rank * kWarps + warp;
        direct_pass<Ring>(P.A, P.A.warp_chunk[bw].x, P.A.warp_entry[bw], tk->warp_step[warp], tk->warp_step[warp + 1], P.x, P.q);
      }
    } else {
      acc_g = ring_pass<Ring>(sm.base, tk->warp_step[warp], tk->warp_step[warp + 1], step ? P.p : P.x, step);
    }
    const bool ok = sm.stream(warp)->failed == 0;

    if (!step) {
      // ---- d = b - A x.  Setup: r = d, p = z = dinv .* r (Jacobi) or r,
      // rho = r.z, rr = r.r, ||b||^2.  Replacement: r, rr and rho take the true
      // residual's values.  End: the true residual's norm.
      cta_sync();  // the CTA's rows of q are complete
      double acc_rr = 0.0, acc_bb = 0.0, acc_rz = 0.0;
      {
        double* const r = residual();
        for (int i = tk->row0 + tid; i < tk->row1; i += kBlock) {
          const double bi = P.b[i];
          const double ri = bi - P.q[i];
          double zi = ri;
          if constexpr (kJacobi) zi = P.dinv[i] * ri;
          if (pass != kPassEnd) r[i] = ri;
          if (pass == kPassSetup) {
            P.p[i] = zi;
            if constexpr (kMixed) P.p32[i] = static_cast<float>(zi);
          }
          acc_rr = fma(ri, ri, acc_rr);
          if constexpr (kJacobi) acc_rz = fma(ri, zi, acc_rz);
          acc_bb = fma(bi, bi, acc_bb);
        }
      }
      if (!group_sum(ok, kJacobi ? 3 : 2, acc_rr, acc_bb, acc_rz, -1, [&](const double* sum) {
            if (pass == kPassEnd) {
              if (tk->rank == 0) {
                SolveCtrl* const ctrl = P.ctrl;
                const int32_t f = st->flags;
                ctrl->status = (f & kFlagBreakdown) ? kEBREAKDOWN : ((f & kFlagDone) ? kOK : kENOTCONV);
                ctrl->iters = st->k;
                ctrl->rho = st->rho;
                ctrl->bnorm2 = st->bnorm2;
                ctrl->relres_rec = sqrt(st->rr / st->bnorm2);
                ctrl->relres_true = sqrt(sum[0] / st->bnorm2);
                ctrl->phase = kPhaseDone;
              }
              return;
            }
            st->rr = sum[0];
            st->rho = kJacobi ? sum[2] : sum[0];
            if (pass == kPassSetup) {
              st->bnorm2 = sum[1];
              // Stopping test sqrt(rr) <= tol ||b|| evaluated as rr <= tol^2 ||b||^2
              // (no square root on the critical path; the same test up to rounding).
              st->thresh2 = (P.tol * P.tol) * sum[1];
            }
            if (sum[0] <= st->thresh2) st->flags |= kFlagDone;
          }, no_side)) {
        solve_fail(P, tid == 0);
        return;
      }
      if (pass == kPassEnd) return;
      if (pass == kPassSetup && st->bnorm2 == 0.0) {  // b = 0: the solution is 0
        for (int i = tk->row0 + tid; i < tk->row1; i += kBlock) P.x[i] = 0.0;
        if (tk->rank == 0 && tid == 0) {
          SolveCtrl* const ctrl = P.ctrl;
          ctrl->status = kOK;
          ctrl->iters = 0;
          ctrl->rho = 0.0;
          ctrl->bnorm2 = 0.0;
          ctrl->relres_rec = 0.0;
          ctrl->relres_true = 0.0;
          ctrl->phase = kPhaseDone;
        }
        return;
      }
      if (pass == kPassReplace && !(st->flags & kFlagDone)) {
        // the step's p update, on the true residual
        const double beta = st->beta;
        const double* const r = residual();
        for (int i = tk->row0 + tid; i < tk->row1; i += kBlock) {
          double zi = r[i];
          if constexpr (kJacobi) zi = P.dinv[i] * zi;
          const double pi = fma(beta, P.p[i], zi);
          P.p[i] = pi;
          if constexpr (kMixed) P.p32[i] = static_cast<float>(pi);
        }
      }
    } else {
      // alpha = rho / gamma, once per CTA (an FP64 division is slow)
      if (!group_sum(ok, 1, acc_g, 0.0, 0.0, 0, [&](const double* sum) {
            const double gamma = sum[0];
            if (!(gamma > 0.0) || !isfinite(gamma)) st->flags |= kFlagBreakdown;  // not SPD, or overflow
            else st->alpha = st->rho / gamma;
          }, no_side)) {
        solve_fail(P, tid == 0);
        return;
      }
      if (!(st->flags & kFlagBreakdown)) {
        // ---- r -= alpha q; rr = r.r and (Jacobi) r.z   (kVR rows per thread in flight)
        double acc_r = 0.0, acc_z = 0.0;
        {
          const double alpha = st->alpha;
          const int row1 = tk->row1;
          const double* const q = P.q;
          const double* const dinv = P.dinv;
          double* const r = residual();
          for (int base = tk->row0 + tid; base < row1; base += kVR * kBlock) {
            double qv[kVR] = {}, rv[kVR] = {}, dv[kVR] = {};
#pragma unroll
            for (int u = 0; u < kVR; ++u) {
              const int i = base + u * kBlock;
              if (i < row1) {
                qv[u] = q[i];
                rv[u] = r[i];
                if constexpr (kJacobi) dv[u] = dinv[i];
              }
            }
#pragma unroll
            for (int u = 0; u < kVR; ++u) {
              const int i = base + u * kBlock;
              if (i < row1) {
                const double rn = fma(-alpha, qv[u], rv[u]);
                r[i] = rn;
                acc_r = fma(rn, rn, acc_r);
                if constexpr (kJacobi) acc_z = fma(rn, dv[u] * rn, acc_z);
              }
            }
          }
        }
        // kSmallShare: x += alpha p by warps 1.. while warp 0 does the sum below (x is
        // needed again only by the next residual replacement or at the end)
        auto side_x = [&] {
          if constexpr (kSmallShare) {
            const double alpha = st->alpha;
            const int row1 = tk->row1;
            const double* const p = P.p;
            double* const x = P.x;
            for (int base = tk->row0 + tid - 32; base < row1; base += 2 * (kBlock - 32)) {
              double pv[2] = {}, xv[2] = {};
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int i = base + u * (kBlock - 32);
                if (i < row1) {
                  pv[u] = p[i];
                  xv[u] = x[i];
                }
              }
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const int i = base + u * (kBlock - 32);
                if (i < row1) x[i] = fma(alpha, pv[u], xv[u]);
              }
            }
          }
        };
        if (!group_sum(true, kJacobi ? 2 : 1, acc_r, acc_z, 0.0, 1, [&](const double* sum) {
              const long long k = st->k + 1;
              st->k = k;
              const double rr = sum[0], rho_new = kJacobi ? sum[1] : sum[0];
              st->rr = rr;
              // beta keeps the recurrence's own ratio (rho_new: the recursive r.z
              // of this step), also when r is replaced below
              st->beta = rho_new / st->rho;
              bool replace = false;
              if constexpr (kMixed)
                replace = (P.replace_every > 0 && k % P.replace_every == 0) || rr <= st->thresh2;
              if (replace) {
                st->flags |= kFlagReplace;
              } else {
                if (rr <= st->thresh2) st->flags |= kFlagDone;
                st->rho = rho_new;
              }
            }, side_x)) {
          solve_fail(P, tid == 0);
          return;
        }
        // ---- x += alpha p (large shares); p = z + beta p   (z = dinv .* r, or r)
        // unless the residual is replaced first or the solve is done
        const bool upd_p = !(st->flags & (kFlagReplace | kFlagDone));
        if (!kSmallShare || upd_p) {
          const double alpha = st->alpha, beta = st->beta;
          const int row1 = tk->row1;
          double* const x = P.x;
          double* const p = P.p;
          float* const p32 = P.p32;
          const double* const dinv = P.dinv;
          const double* const r = residual();
          for (int base = tk->row0 + tid; base < row1; base += kVR * kBlock) {
            double pv[kVR] = {}, zv[kVR] = {}, xv[kVR] = {};
#pragma unroll
            for (int u = 0; u < kVR; ++u) {
              const int i = base + u * kBlock;
              if (i < row1) {
                pv[u] = p[i];
                zv[u] = r[i];
                if constexpr (kJacobi) zv[u] = dinv[i] * zv[u];
                if constexpr (!kSmallShare) xv[u] = __ldcs(x + i);  // x is not read again this step: evict-first
              }
            }
#pragma unroll
            for (int u = 0; u < kVR; ++u) {
              const int i = base + u * kBlock;
              if (i < row1) {
                if constexpr (!kSmallShare) __stcs(x + i, fma(alpha, pv[u], xv[u]));
                if (upd_p) {
                  const double pn = fma(beta, pv[u], zv[u]);
                  p[i] = pn;
                  if constexpr (kMixed) p32[i] = static_cast<float>(pn);
                }
              }
            }
          }
        }
      }
    }

    // ---- what comes next, and the wait before the next product gathers
    const int32_t f = st->flags;
    // a replacement comes before the step limit: it alone tells whether a mixed
    // solve has converged
    const bool last = (f & (kFlagDone | kFlagBreakdown)) || (!(f & kFlagReplace) && st->k >= P.maxit);
    const bool next_step = !last && !(f & kFlagReplace);
    bool synced;
    if constexpr (kNeighborWait)
      synced = step && next_step && neighbor() ? neighbor_sync() : group_sync();
    else
      synced = group_sync();
    if (!synced) { solve_fail(P, tid == 0); return; }
    if (next_step && pass != kPassSetup && st->k >= st->k_end) {
      // end of this launch's share of the solve: save the state (identical in
      // every CTA of the group; x, r, p are complete after the barrier)
      if (tk->rank == 0 && tid == 0) {
        SolveCtrl* const ctrl = P.ctrl;
        ctrl->iters = st->k;
        ctrl->rho = st->rho;
        ctrl->bnorm2 = st->bnorm2;
        ctrl->relres_rec = sqrt(st->rr / st->bnorm2);
        ctrl->rounds = st->target / static_cast<unsigned long long>(P.group);
        ctrl->slot = st->slot;
        for (int j = 0; j < 3; ++j) {
          ctrl->acc_seen[j][0] = st->acc_seen[j][0];
          ctrl->acc_seen[j][1] = st->acc_seen[j][1];
          ctrl->acc_exp[j] = st->acc_exp[j];
        }
        ctrl->phase = kPhaseRunning;
      }
      return;
    }
    if (tid == 0) {
      st->pass = last ? kPassEnd : (f & kFlagReplace) ? kPassReplace : kPassStep;
      st->flags = f & ~kFlagReplace;
    }
    cta_sync();
  }
}

}  // namespace cgk
