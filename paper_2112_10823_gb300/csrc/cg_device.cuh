// Device-side building blocks of the CG kernels: PTX wrappers for 1-D TMA
// bulk copies and mbarriers, deterministic reductions, the bounded grid
// barrier of the persistent solve, and the CSR product fed by a TMA ring.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>
#include "cg_internal.h"

namespace cgk {

// ------------------------------------------------------------------ PTX

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Makes mbarrier initialisation visible to the async (TMA) proxy.
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// 1-D bulk copy global -> shared (TMA), completion counted on `bar`.
// dst and src 16-byte aligned, bytes a non-zero multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// The same copy with an L2 eviction policy (createpolicy): used for data read
// once per pass, so that it does not push reused data out of L2.
__device__ __forceinline__ void bulk_g2s_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                              uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ int ld_volatile_i32(const int32_t* p) {
  return *reinterpret_cast<const volatile int32_t*>(p);
}

// Barrier of the computing warps only (named barrier 1): the producer warp
// takes no part in it.
__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kBlock) : "memory"); }

__device__ __forceinline__ void st_release_shared(uint32_t* p, uint32_t v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_acquire_shared(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

// threadIdx.x, read anew: what is computed from it is not kept in registers
// from one pass over the matrix to the next (the compiler would move it out of
// the step loop, and spill it).
__device__ __forceinline__ int fresh_tid() {
  int t;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  return t;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// ------------------------------------------------------------ reductions

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;  // identical in every lane (IEEE addition is commutative)
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of `v` over the CTA in a fixed order (FP64 adds); every thread gets the
// same value.  `red` holds blockDim.x + 1 doubles (blockDim.x a multiple of
// 32, at most 1024).  All threads must call it.
__device__ __forceinline__ double block_sum(double v, double* red) {
  const int nt = blockDim.x;
  __syncthreads();
  red[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = red[threadIdx.x];
    for (int j = 32 + threadIdx.x; j < nt; j += 32) s += red[j];
    s = warp_sum(s);
    if (threadIdx.x == 0) red[nt] = s;
  }
  __syncthreads();
  return red[nt];
}

// -------------------------------------------- warp-level fixed-point sums

// A partial of an exact fixed-point sum: the integer m at scale 2^(e - 1074),
// e being the largest biased exponent among the values summed; nf: a NaN or
// an infinity was among them.
struct FxPart {
  long long m;
  int32_t e;
  int32_t nf;
};

// Sum over the warp of one integer per lane (modulo 2^64), in limbs of 20, 20 and
// 24 bits: three 32-bit reductions side by side take some 60 cycles, five rounds of
// 64-bit shuffles 175.
__device__ __forceinline__ long long warp_sum_int(long long m) {
  const unsigned int l0 = static_cast<unsigned int>(m) & 0xfffffu;
  const unsigned int l1 = static_cast<unsigned int>(m >> 20) & 0xfffffu;
  const int l2 = static_cast<int>(m >> 40);
  const unsigned int s0 = __reduce_add_sync(0xffffffffu, l0);
  const unsigned int s1 = __reduce_add_sync(0xffffffffu, l1);
  const int s2 = __reduce_add_sync(0xffffffffu, l2);
  return (static_cast<long long>(s2) << 40) + (static_cast<long long>(s1) << 20) + s0;
}

// Sum over the warp of one double per lane, exactly, in fixed point at the
// warp's largest exponent E (spacing 2^(E-1074), about 2^-51 of the largest
// value; 32 values leave ample headroom).  Every lane gets the same result.
__device__ __forceinline__ FxPart fx_warp(double v) {
  const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(v));
  const int e = static_cast<int>((bits >> 52) & 0x7ffull);
  const int E = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned int>(e)));
  const int nf = __any_sync(0xffffffffu, e == 0x7ff);
  long long m = 0;
  if (e != 0 && !nf) {
    const int s = E - e + 1;  // >= 1
    if (s < 64) {
      const unsigned long long M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
      const unsigned long long rnd = (M + (1ull << (s - 1))) >> s;
      m = (bits >> 63) ? -static_cast<long long>(rnd) : static_cast<long long>(rnd);
    }
  }
  return FxPart{warp_sum_int(m), E, nf};
}

// Sum of up to 32 partials, one per lane (`valid` lanes), realigned to the
// largest exponent (each partial rounded once, to nearest, ties away from
// zero).  The result depends only on the partials, not on their order.  Every
// lane gets it.
__device__ __forceinline__ FxPart fx_combine(FxPart p, bool valid) {
  const int E = static_cast<int>(__reduce_max_sync(0xffffffffu, valid ? static_cast<unsigned int>(p.e) : 0u));
  const int nf = __any_sync(0xffffffffu, valid && p.nf);
  long long m = 0;
  if (valid && p.m != 0) {
    const int d = E - p.e;  // >= 0
    if (d == 0) {
      m = p.m;
    } else if (d < 63) {
      const long long a = p.m < 0 ? -p.m : p.m;
      const long long r = (a + (1ll << (d - 1))) >> d;
      m = p.m < 0 ? -r : r;
    }
  }
  return FxPart{warp_sum_int(m), E, nf};
}

// m 2^k for a double m of magnitude below 2^64 (an integer's conversion), by its
// exponent field where the result is a normal number (ldexp takes four FP64
// operations one after another).
__device__ __forceinline__ double fx_scale(double m, int k) {
  const long long bits = __double_as_longlong(m);
  const int e = static_cast<int>((bits >> 52) & 0x7ff);
  if (e != 0 && e + k > 0 && e + k < 2047) return __longlong_as_double(bits + (static_cast<long long>(k) << 52));
  return ldexp(m, k);
}

// The double nearest to a partial.
__device__ __forceinline__ double fx_value(FxPart p) {
  if (p.nf) return __longlong_as_double(0x7ff8000000000000ll);
  if (p.e == 0) return 0.0;
  return fx_scale(static_cast<double>(p.m), p.e - 1074);
}

// Exact fixed-point sum, over the calling warp, of src[0 .. count), read
// through L2 (values written by other CTAs); lane j takes entries j, j + 32,
// ...; count <= 1024 keeps the integer sum within 63 bits.  The loads of a
// batch of 8 entries per lane are all issued before any is used (one L2
// round trip for up to 256 entries); the batch stays in registers for both
// steps (the largest exponent, then the rounded integers).  Every lane gets
// the result.
__device__ __forceinline__ double fx_warp_sum_array(const double* src, int count) {
  constexpr int kB = 8;
  const int lane = threadIdx.x & 31;
  long long m = 0;
  int E = 0, nf = 0;
  // the exponent of the whole array first (so that all batches share one grid)
  {
    unsigned int emax = 0;
    int nfl = 0;
    for (int j0 = 0; j0 < count; j0 += 32 * kB) {
      double v[kB];
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const int j = j0 + lane + 32 * u;
        v[u] = j < count ? __ldcg(src + j) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(v[u]));
        const unsigned int e = static_cast<unsigned int>((bits >> 52) & 0x7ffull);
        emax = e > emax ? e : emax;
        nfl |= (e == 0x7ffu);
      }
      if (j0 + 32 * kB >= count) {
        // last (usually only) batch: sum it from the registers
        E = static_cast<int>(__reduce_max_sync(0xffffffffu, emax));
        nf = __any_sync(0xffffffffu, nfl);
        if (j0 == 0 && !nf) {
#pragma unroll
          for (int u = 0; u < kB; ++u) {
            const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(v[u]));
            const int e = static_cast<int>((bits >> 52) & 0x7ffull);
            const int sh = E - e + 1;
            if (e != 0 && sh < 64) {
              const unsigned long long M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
              const unsigned long long rnd = (M + (1ull << (sh - 1))) >> sh;
              m += (bits >> 63) ? -static_cast<long long>(rnd) : static_cast<long long>(rnd);
            }
          }
        }
      }
    }
  }
  if (count > 32 * kB && !nf) {
    // more than one batch: a second pass over the array at the common grid
    for (int j0 = 0; j0 < count; j0 += 32 * kB) {
      double v[kB];
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const int j = j0 + lane + 32 * u;
        v[u] = j < count ? __ldcg(src + j) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < kB; ++u) {
        const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(v[u]));
        const int e = static_cast<int>((bits >> 52) & 0x7ffull);
        const int sh = E - e + 1;
        if (e != 0 && sh < 64) {
          const unsigned long long M = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
          const unsigned long long rnd = (M + (1ull << (sh - 1))) >> sh;
          m += (bits >> 63) ? -static_cast<long long>(rnd) : static_cast<long long>(rnd);
        }
      }
    }
  }
  return fx_value(FxPart{warp_sum_int(m), E, nf});
}

// ---- sums through accumulators
//
// A group sum costs, beyond its arithmetic, what the CTAs' meeting costs.  The
// general form (publish a value, meet at the barrier, read all values) takes a
// fence before the arrival, a fence behind it and one more trip to the L2, and
// the two sums of a CG step need none of that: the data they order is the sum
// itself.  Here every CTA adds its value, as an integer, into two 64-bit words
// with relaxed atomics, and a count of arrivals travels in the same words: who
// sees all arrivals has the sum.  Integer addition commutes, so every CTA gets
// the same bits.  The words are never cleared: a CTA keeps what it saw last and
// takes the difference; a word is used again only after another such sum, which
// every CTA enters with the last one read.
//
// The integers' unit is set by the last sum of the same kind, of biased exponent
// eb: 2^(eb - 1085), i.e. that sum was about 2^62 units.  A CTA's value is
// rounded to a unit: 152 roundings of half a unit are at most 2^-55.7 of a sum as
// large as the last, and 2^-47.7 of the smallest one accepted, 2^54 units (a sum
// that fell by 2^8).  The general form rounds the CTAs' values to 2^-51 of the
// largest of them: at most 2^-44.7 of a sum that one CTA dominates, and some 2^-52
// of one with even shares, so a sum of even shares that fell by 20 times or more
// from one step to the next is the one case in which this form is the coarser.
// Values of up to 2^73 units go in (growth by 2^11), split in a signed high part
// (53 bits) and 32 low bits; anything else, or a sum below 2^54 units, makes every
// CTA take the general form instead.
// Low word: 42 bits of low parts, 11 of CTAs that could not add theirs, 11 of
// arrivals; high word: 53 bits of high parts, 11 of arrivals.
constexpr int kAccUnit = 1085;
constexpr unsigned int kAccCount = 0x7ff;  // most CTAs of a group: 1024 (cg_create)

// What a CTA adds for the partial p.
__device__ __forceinline__ void acc_words(FxPart p, int eb, unsigned long long* lo, unsigned long long* hi) {
  const unsigned long long a = static_cast<unsigned long long>(p.m < 0 ? -p.m : p.m);
  const int sh = p.e - 1074 - (eb - kAccUnit);  // p is m 2^sh units
  unsigned long long l = 0, h = 0;
  bool fits = p.nf == 0;
  if (a != 0) {
    if (sh >= 0) {
      fits = fits && 64 - __clzll(static_cast<long long>(a)) + sh <= 73;
      if (fits) {  // (then sh < 74)
        l = sh < 64 ? a << sh : 0ull;
        h = sh == 0 ? 0ull : sh < 64 ? a >> (64 - sh) : a << (sh - 64);
      }
    } else if (sh > -64) {
      l = (a + (1ull << (-sh - 1))) >> -sh;
    }
  }
  if (p.m < 0) {  // two's complement
    l = ~l + 1ull;
    h = ~h + (l == 0 ? 1ull : 0ull);
  }
  const unsigned long long high = (h << 32) | (l >> 32);
  *lo = ((l & 0xffffffffull) << 22) + 1ull;
  *hi = (high << 11) + 1ull;
  if (!fits) {
    *lo = (1ull << 11) + 1ull;
    *hi = 1ull;
  }
}

// The sum that the words' differences hold (all arrivals in); false if the
// general form has to give it.
__device__ __forceinline__ bool acc_sum(unsigned long long lo, unsigned long long hi, unsigned int count, int eb,
                                        double* sum) {
  if ((lo >> 11) & kAccCount) return false;
  // both parts are exact doubles, and the FMA rounds once
  const double high = __ll2double_rn(static_cast<long long>(hi - count) >> 11);
  const double low = __ull2double_rn(lo >> 22);
  const double v = fma(high, 4294967296.0, low);
  const long long bits = __double_as_longlong(v);
  const int ev = static_cast<int>((bits >> 52) & 0x7ff), e = ev + eb - kAccUnit;
  if (ev < 1023 + 54 || e <= 0 || e >= 2047) return false;
  *sum = __longlong_as_double(bits + (static_cast<long long>(eb - kAccUnit) << 52));
  return true;
}

// Biased exponent of a sum that the next one of its kind can be measured by (0: none).
__device__ __forceinline__ int acc_exponent(double v) {
  const int e = static_cast<int>((__double_as_longlong(v) >> 52) & 0x7ff);
  return e == 0x7ff ? 0 : e;
}

// Waits until the words at `word` hold `count` arrivals more than lo0, hi0; *lo
// and *hi get their values.  Returns false after a wait longer than limit_ns or
// an abort raised by another CTA.
__device__ __forceinline__ bool acc_wait(SolveCtrl* ctrl, const unsigned long long* word, unsigned long long lo0,
                                         unsigned long long hi0, unsigned int count, unsigned long long limit_ns,
                                         unsigned long long* lo, unsigned long long* hi) {
  unsigned long long t0 = 0;
  uint32_t spins = 0;
  for (;;) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(*lo), "=l"(*hi) : "l"(word) : "memory");
    if (((*lo - lo0) & kAccCount) == count && ((*hi - hi0) & kAccCount) == count) return true;
    if ((++spins & 255u) == 0) {
      if (*reinterpret_cast<const volatile int32_t*>(&ctrl->abort)) return false;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        atomicExch(&ctrl->abort, 1);
        atomicExch(&ctrl->timeout_site, kAccSite);
        return false;
      }
    }
  }
}

// Arrival and bounded wait of thread 0 at the group barrier of a system
// (the caller synchronises its own CTA around it).  `target` is the CTA's
// running target (in shared memory: thread 0 alone keeps it).  The arrival is
// a release pattern (an acq_rel fence, cumulative over what the CTA wrote
// before the CTA barrier that precedes it, then a relaxed add); the wait
// polls with relaxed loads and ends with an acquire pattern (an acq_rel
// fence).  These fences are lighter than the sequentially consistent one of
// __threadfence().  Returns false after a wait longer than limit_ns or an
// abort raised by another CTA.
__device__ __forceinline__ bool group_barrier_t0(SolveCtrl* ctrl, unsigned long long* target, unsigned int count,
                                                 unsigned long long limit_ns, int site) {
  *target += count;
  if (count <= 1) return true;
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(&ctrl->barrier), "l"(1ull) : "memory");
  unsigned long long t0 = 0;
  uint32_t spins = 0;
  const unsigned long long tgt = *target;
  for (;;) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&ctrl->barrier) : "memory");
    if (v >= tgt) break;
    if ((++spins & 255u) == 0) {
      if (*reinterpret_cast<const volatile int32_t*>(&ctrl->abort)) return false;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) {
        atomicExch(&ctrl->abort, 1);
        atomicExch(&ctrl->timeout_site, site);
        return false;
      }
    }
  }
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  return true;
}

// ------------------------------------------------------ streamed CSR product

// What a product reads and writes besides the warp's ring.  In shared memory and
// read where it is used: the product's registers hold what it gathers.
struct PassIo {
  const int4* step;
  const uint8_t* seg_len;
  const double* aux;           // with_dot: the vector whose product with the result is summed
  double* out;
  unsigned long long limit_ns;
  int32_t nsteps;
  int32_t stream_rows;         // tables with the evict-first policy
};
__device__ __forceinline__ PassIo pass_io(const DevCsr& A, int32_t stream_rows, const double* aux, double* out,
                                          unsigned long long limit_ns) {
  return PassIo{A.step, A.seg_len, aux, out, limit_ns, A.nsteps, stream_rows};
}

// Per-CTA state of a solve, in shared memory: written by thread 0 (between
// CTA barriers), read by all.  Keeping it out of registers leaves the
// product in the step loop the registers it needs.
struct CtaState {
  PassIo io;
  double rho;                  // r.z (r.r without a preconditioner)
  double rr;                   // r.r of the current iterate
  double bnorm2;               // b.b
  double thresh2;              // tol^2 b.b
  double alpha, beta;
  long long k;                 // steps done
  long long k_end;             // last step of this launch
  unsigned long long target;   // group-barrier target of this CTA
  int32_t slot;                // partial-sum slot of the next group sum
  int32_t site;                // diagnostics: group waits so far
  int32_t ok;                  // the last group sum or barrier succeeded
  int32_t flags;               // kFlag* below
  int32_t pass;                // what the next product is for (kPass* below)
  unsigned long long acc_seen[3][2];  // accumulators p.q, r.r, r.z: their words when last summed
  int32_t acc_exp[3];                 // and the exponents of those sums (0: none yet)
  int32_t dep_lo, dep_hi;      // CTAs whose rows this CTA's columns reach (columns first, then ranks)
};
enum : int32_t { kFlagDone = 1, kFlagBreakdown = 2, kFlagReplace = 4 };
enum : int32_t { kPassSetup, kPassStep, kPassReplace, kPassEnd };

// Warp partials of a CTA sum (up to three values per thread) and each
// warp's vote.
constexpr int kMaxSumValues = 3;
struct SumScratch {
  FxPart part[kMaxSumValues][kWarps];
  int32_t ok[kWarps];
};

// A warp's stream of the matrix: the chunks of its steps, one after another,
// pass after pass, through the slots of its ring.  The warp's side of it,
// kept here between passes:
struct WarpStream {
  uint32_t consumed;  // chunks of this task the warp is done with (read by the producer)
  uint32_t phases;    // the parity that each slot's barrier completes next (a bit per slot)
  int32_t tail;       // slot of the next chunk
  int32_t failed;     // a wait gave up
  // its first two steps and the lanes' segment lengths: every pass begins with
  // them, and a load from L2 there would be on its critical path
  int4 step[2];
  uint8_t seg_len[2][32];
};

// Dynamic shared memory of a persistent CTA: the full mbarrier of every ring
// slot, the CTA state of a solve, the warp partials of its sums, then the rings
// (values of type T, columns of type C) of every warp, and in the small-share
// solve the r of the CTA's rows.  The parts before the rings sit at the same
// place whatever T and C are.
template <typename T, typename C>
struct RingSmem {
  using Val = T;
  using Col = C;
  static constexpr int kChunk = max_chunk(sizeof(T) == 4, sizeof(C) == 2);
  static constexpr int kSlotBytes = static_cast<int>(kUnit * chunk_units(32 * kChunk, sizeof(C), sizeof(T)));
  static constexpr size_t kStateOff = (8 * kSlots * kWarps + 15) & ~size_t(15);
  static constexpr size_t kSumOff = kStateOff + ((sizeof(CtaState) + 15) & ~size_t(15));
  static constexpr size_t kStreamOff = (kSumOff + sizeof(SumScratch) + 15) & ~size_t(15);
  static constexpr size_t kRingOff = (kStreamOff + sizeof(WarpStream) * kWarps + 16 + 127) & ~size_t(127);
  static constexpr size_t kBytes = kRingOff + static_cast<size_t>(kSlotBytes) * kSlots * kWarps;

  unsigned char* base;
  __device__ unsigned char* slot(int w, int s) const { return base + kRingOff + (w * kSlots + s) * kSlotBytes; }
  __device__ uint64_t* full(int w, int slot) const { return reinterpret_cast<uint64_t*>(base) + w * kSlots + slot; }
  __device__ WarpStream* stream(int w) const { return reinterpret_cast<WarpStream*>(base + kStreamOff) + w; }
  __device__ int32_t* stop() const { return reinterpret_cast<int32_t*>(base + kStreamOff + sizeof(WarpStream) * kWarps); }
  __device__ CtaState* state() const { return reinterpret_cast<CtaState*>(base + kStateOff); }
  __device__ SumScratch* sums() const { return reinterpret_cast<SumScratch*>(base + kSumOff); }
  // r of the CTA's rows in a small-share solve, behind the rings (kLocalRows entries).
  __device__ double* local() const { return reinterpret_cast<double*>(base + kBytes); }
};

// Dynamic shared memory of a kernel whose step-loop product streams values of
// type T and columns of type C; `local`: with the small-share solve's r.
template <typename T, typename C>
constexpr size_t ring_smem_bytes(bool local = false) {
  return RingSmem<T, C>::kBytes + (local ? sizeof(double) * kLocalRows : 0);
}

// Initialises every ring barrier and stream (all threads of the CTA call; ends
// with a CTA barrier).  Once per kernel: the phases are kept count of through
// all tasks.
template <typename Ring>
__device__ __forceinline__ void ring_init(const Ring& sm) {
  if (threadIdx.x < kSlots * kWarps) {
    mbar_init(reinterpret_cast<uint64_t*>(sm.base) + threadIdx.x, 1);
    fence_mbar_init();
  }
  if (threadIdx.x < kWarps) {
    WarpStream* const ws = sm.stream(threadIdx.x);
    ws->consumed = ws->phases = 0;
    ws->tail = ws->failed = 0;
  }
  if (threadIdx.x == 0) *sm.stop() = 0;
  __syncthreads();
}

// Readies the streams for the CTA's next task (the last one's warps are all
// through, the producer included; a CTA barrier follows before the streams are
// used).
template <typename Ring>
__device__ __forceinline__ void ring_reset(const Ring& sm) {
  if (threadIdx.x < kWarps) {
    WarpStream* const ws = sm.stream(threadIdx.x);
    ws->consumed = 0;
    ws->tail = 0;
    ws->failed = 0;
  }
  if (threadIdx.x == 0) *sm.stop() = 0;
}

// Bounded wait on an mbarrier phase; false if it gave up.  If `stop` is
// given, also gives up as soon as *stop becomes non-zero.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, unsigned long long limit_ns,
                                                  const int32_t* stop) {
  uint32_t spins = 0;
  unsigned long long t0 = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++spins & 63u) == 0) {
      if (stop && ld_volatile_i32(stop)) return false;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) return false;
    }
  }
  return true;
}

// The producer warp of CTA `rank`: lane w copies the chunks of warp w's stream,
// pass after pass (`once`: one pass; `keep`: with the L2's default policy, else
// evict-first), into its ring as the warp gives slots back, until the computing warps say stop.  One lane per warp: a copy takes
// some thirty instructions, which are no part of any computing warp's chain,
// and all warps that wait for one are served together.  On stop every lane
// waits for its copies in flight, so that none lands after the CTA is gone or
// in a ring that the next task has taken over, and leaves the phases to that
// task's warps.
//
// Waiting for a slot is no wait of the solve: the ring stays full through a
// step's vector phases, both sums and a whole direct pass, each of which keeps
// its own limit, and computing warps that give up say stop.  So it ends by
// itself; its bound, far beyond theirs, is for a fault in this code only.
// Returns (uniformly) kStreamDone, kStreamIdle if that bound ran out, or
// kStreamLost if a copy did not arrive within limit_ns: then the ring cannot
// be used again.
enum : int { kStreamDone = 0, kStreamIdle = 1, kStreamLost = 2 };
template <typename Ring>
__device__ __forceinline__ int producer(const Ring& sm, const DevCsr& A, int rank, bool once, bool keep,
                                        unsigned long long limit_ns) {
  const int w = threadIdx.x & 31;
  const bool mine = w < kWarps;
  WarpStream* const ws = sm.stream(mine ? w : 0);
  // the bounds of chunk `next`, and the ends of the two after it (the stream
  // goes round: chunk nchunks is chunk 0 again), loaded ahead
  int c0 = 0, nchunks = 0, next = 0;
  uint32_t first = 0, start = 0, end0 = 0, end1 = 0, end2 = 0;
  auto end_of = [&](int j) { return A.chunk_off[c0 + j % nchunks + 1]; };
  if (mine) {
    // (the first copy waits for this load alone)
    const int4 c = A.warp_chunk[rank * kWarps + w];
    c0 = c.x;
    nchunks = c.y;
    first = start = static_cast<uint32_t>(c.z);
    end0 = static_cast<uint32_t>(c.w);
    if (nchunks > 0) {
      end1 = end_of(1);
      end2 = end_of(2);
    }
  }
  const uint64_t pol = l2_evict_first_policy();
  uint32_t phases = ws->phases, issued = 0;
  int head = 0;
  bool stalled = false, arrived = true;
  unsigned long long t0 = 0;
  uint32_t idle = 0;
  for (;;) {
    const bool more = nchunks > 0 && (!once || issued < static_cast<uint32_t>(nchunks));
    if (!__any_sync(0xffffffffu, more) || __any_sync(0xffffffffu, ld_volatile_i32(sm.stop()) != 0)) break;
    const bool free = more && issued - ld_acquire_shared(&ws->consumed) < static_cast<uint32_t>(kSlots);
    if (free) {
      uint64_t* const bar = sm.full(w, head);
      const uint32_t bytes = (end0 - start) * static_cast<uint32_t>(kUnit);
      mbar_arrive_expect_tx(bar, bytes);
      const unsigned char* const from = A.stream + static_cast<size_t>(start) * kUnit;
      if (keep) bulk_g2s(sm.slot(w, head), from, bytes, bar);
      else bulk_g2s_hint(sm.slot(w, head), from, bytes, bar, pol);
      phases ^= 1u << head;
      head = head + 1 == kSlots ? 0 : head + 1;
      ++issued;
      next = next + 1 == nchunks ? 0 : next + 1;
      start = next == 0 ? first : end0;
      end0 = end1;
      end1 = end2;
      end2 = end_of(next + 2);
    }
    if (__any_sync(0xffffffffu, free)) {
      idle = 0;
    } else {
      __nanosleep(32);
      if ((++idle & 255u) == 0) {
        const unsigned long long now = global_timer_ns();
        if (idle == 256u) t0 = now;
        else if (now - t0 > 4 * limit_ns + kProducerIdleNs) {
          stalled = true;
          break;
        }
      }
    }
  }
  if (mine) {
    for (int k = 0; k < kSlots; ++k)  // the latest copy into each slot
      if (issued > static_cast<uint32_t>(k))
        arrived = mbar_wait_bounded(sm.full(w, k), ((phases >> k) & 1u) ^ 1u, limit_ns, nullptr) && arrived;
  }
  arrived = __all_sync(0xffffffffu, arrived);
  // (no computing warp reads its phases any more: in a solve they have said
  // stop, a single pass keeps its own)
  if (!once && mine && nchunks > 0) ws->phases = phases;
  return !arrived ? kStreamLost : __any_sync(0xffffffffu, stalled) ? kStreamIdle : kStreamDone;
}

// The computing warps of a task are through (all of their threads call).
template <typename Ring>
__device__ __forceinline__ void stop_producer(const Ring& sm) {
  cta_sync();
  if (threadIdx.x == 0) *reinterpret_cast<volatile int32_t*>(sm.stop()) = 1;
}

// ---- steps

__device__ __forceinline__ int step_lanes(const int4& d) { return d.y & 0xff; }
__device__ __forceinline__ int step_mode(const int4& d) { return (d.y >> kStepModeShift) & 3; }

__device__ __forceinline__ int step_chunk(const int4& d) { return (d.y >> kStepChunkShift) & kStepChunkMask; }

// Whether step d is stored padded (with columns of type C).
template <typename C>
__device__ __forceinline__ bool step_padded(const int4& d) {
  return sizeof(C) == 2 && (d.y & kStepPadded) != 0;
}

// The tables that are read once per product: step s, and the length of this
// lane's segment in it where the step itself does not tell.  io.stream_rows: with
// the evict-first policy, so that in a solve whose vectors and tables together
// outgrow the L2 the tables give way to the vectors that the step reads again.
__device__ __forceinline__ int4 load_step(const PassIo& io, int s) {
  return io.stream_rows ? __ldcs(io.step + s) : io.step[s];
}
__device__ __forceinline__ int load_seg_len(const PassIo& io, int s, int lane) {
  const uint8_t* p = io.seg_len + static_cast<size_t>(s) * 32 + lane;
  return io.stream_rows ? __ldcs(p) : *p;
}

// Entries of this lane's segment of step d (len: from load_seg_len).
__device__ __forceinline__ int lane_segment(const int4& d, int len, int lane) {
  if (step_mode(d) == kLongRow)
    return d.z - ((d.y & kStepUniform) || lane < ((d.y >> kStepRemShift) & 0x3f) ? 0 : 1);
  return len;
}

// Exclusive sum over the lanes below this one; *total: over the warp.
__device__ __forceinline__ int warp_offset(int v, int lane, int* total) {
  int sum = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int below = __shfl_up_sync(0xffffffffu, sum, o);
    if (lane >= o) sum += below;
  }
  *total = __shfl_sync(0xffffffffu, sum, 31);
  return sum - v;
}

// Where the entries of a chunk lie (entries [u, u + cnt) of every lane's segment
// of step d; seg: this lane's whole segment): this lane's entry k at base + k
// stride, tot stored in all.  Uneven chunks lane after lane: a prefix sum per
// chunk finds a lane's place, where the order by entries took two votes and four
// counts per entry (300,000 rows of 1 to 32 entries: product 31.2 -> 27.1 us,
// mixed step 35.5 -> 26.4; Q1 24^3 and 64^3, whose last steps are short: step
// 12.5 -> 11.0 and 28.1 -> 25.9).
struct ChunkPlace {
  int base, stride, tot;
};
template <typename C>
__device__ __forceinline__ ChunkPlace chunk_place(const int4& d, int u, int cnt, int seg, int lane) {
  if (step_padded<C>(d) || __all_sync(0xffffffffu, u + cnt <= seg)) return ChunkPlace{lane, 32, 32 * cnt};
  if (d.y & kStepUniform) return ChunkPlace{lane, step_lanes(d), step_lanes(d) * cnt};
  ChunkPlace p;
  p.base = warp_offset(max(0, min(seg - u, cnt)), lane, &p.tot);
  p.stride = 1;
  return p;
}

// The row of step d whose result this lane holds once its segment is summed
// (and the lanes of a pair or of a long row are combined); -1 if none.
__device__ __forceinline__ int result_row(const int4& d, int lane) {
  const int mode = step_mode(d);
  if (mode == kLanePerRow) return lane < step_lanes(d) ? d.x + lane : -1;
  if (mode == kPairPerRow) return lane < step_lanes(d) && !(lane & 1) ? d.x + (lane >> 1) : -1;
  return lane == 0 ? d.x : -1;
}

// Sum of a step's row from its lanes' segment sums.
template <typename Acc>
__device__ __forceinline__ Acc combine_lanes(int mode, Acc part) {
  if (mode == kPairPerRow) return part + __shfl_xor_sync(0xffffffffu, part, 1);  // first half + second half
  if (mode == kLongRow) {
    if constexpr (sizeof(Acc) == 8) return warp_sum(part);
    else return warp_sum_f(part);
  }
  return part;
}

// Calls f(std::integral_constant<int, v>) for v in [LO, HI] through a binary
// tree of warp-uniform conditional branches: no indirect jump (a jump table's
// target must be resolved before the warp can go on).
template <int LO, int HI, typename F>
__device__ __forceinline__ void dispatch_tree(int v, F&& f) {
  if constexpr (LO == HI) {
    f(std::integral_constant<int, LO>{});
  } else {
    constexpr int MID = (LO + HI) / 2;
    if (v <= MID) dispatch_tree<LO, MID>(v, f);
    else dispatch_tree<MID + 1, HI>(v, f);
  }
}

// Loads what ring_pass keeps of the warp's first steps (each computing warp of
// the CTA calls, with its steps [s, s1)).
template <typename Ring>
__device__ __forceinline__ void load_first_steps(const Ring& sm, const PassIo& v, int s, int s1) {
  const int lane = threadIdx.x & 31;
  WarpStream* const ws = sm.stream(threadIdx.x >> 5);
  if (s < s1) {
    for (int j = 0; j < 2; ++j) ws->seg_len[j][lane] = v.seg_len[static_cast<size_t>(min(s + j, s1 - 1)) * 32 + lane];
    if (lane < 2) ws->step[lane] = v.step[s + lane < s1 ? s + lane : v.nsteps];
  }
  __syncwarp();
}

// The product over the warp's steps [s, s1) from its ring, gathering x (after
// load_first_steps): out[i] = (A x)_i; with_dot: returns the sum over this
// lane's rows of aux[i] (A x)_i (out and aux from the CTA's PassIo).  Every
// segment is one FMA chain in storage order.
//
// What bounds it in FP64 is the pipe (an FMA occupies a sub-partition for 64
// cycles, whatever its active lanes, and a predicated-off one as well; its
// dependent latency is 115) beside the matrix stream.  So the loop keeps two
// things in flight ahead of the chains: the ring's copies (all slots but the
// two of the chunk being summed and of the next one; the producer warp starts
// them), and the gathers of the warp's next chunk, of the same step or of the
// next one, each issued into the register that the current chunk's FMA has just
// freed.  A warp-uniform branch, not a predicate, ends a chunk's FMAs.  The
// stream's `failed` is raised if a wait gave up.  Against a ring shared by the
// CTA, in CSR order (us, calls back to back): Q1 160^3 240 -> 204, the 110^3 mesh
// 169 -> 81, Q1 64^3 25 -> 19; 109 M FMAs take 176 us at the pipe's peak.
template <typename Ring, typename X>
__device__ __forceinline__ double ring_pass(unsigned char* smem, int s, int s1, const X* x, bool with_dot) {
  using T = typename Ring::Val;
  using C = typename Ring::Col;
  constexpr int kU = Ring::kChunk;
  const Ring sm{smem};
  const PassIo& io = sm.state()->io;
  const int tid = fresh_tid(), w = tid >> 5, lane = tid & 31;
  if (s >= s1) return 0.0;
  double dot = 0.0;
  WarpStream* const ws = sm.stream(w);
  uint32_t consumed = ws->consumed, phases = ws->phases;
  int tail = ws->tail;
  auto leave = [&](bool ok) -> double {
    if (lane == 0) {
      ws->phases = phases;
      ws->tail = tail;
      if (!ok) ws->failed = 1;
    }
    __syncwarp();
    return dot;
  };
  auto wait_next = [&]() -> bool {
    uint64_t* const bar = sm.full(w, tail);
    const uint32_t parity = (phases >> tail) & 1u;
    if (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity)) &&
        !__all_sync(0xffffffffu, mbar_wait_bounded(bar, parity, io.limit_ns, nullptr)))
      return false;
    phases ^= 1u << tail;
    tail = tail + 1 == kSlots ? 0 : tail + 1;
    return true;
  };
  // a chunk: entries [u, u + cnt) of every lane's segment of one step
  struct Chunk {
    int cnt;      // entries per lane (warp-uniform; 0: the step has none; -1: no chunk)
    int len;      // of them, those this lane's segment has
    int place;    // of this lane's entries: base, and the stride in bits 16.. (ChunkPlace); 32 << 16: the full form
    bool ends;    // the last one of its step
    int slot;
    int val_off;  // its values' place in the slot
    int row;      // the step's first row and kind word
    int kind;
    double aux;   // of the row whose sum this lane gets (if it ends the step)
  };
  // steps and their segment lengths are loaded one ahead
  auto step_at = [&](int k) { return k < s1 ? k : io.nsteps; };  // (the sentinel has no entries)
  int4 d = ws->step[0], dn = ws->step[1];
  int seg = ws->seg_len[0][lane], seg_n = ws->seg_len[1][lane];
  seg = lane_segment(d, seg, lane);
  int u = 0;
  // the stream's next chunk
  auto next_chunk = [&]() -> Chunk {
    Chunk c;
    if (s >= s1) {
      c.cnt = -1;
      c.len = 0;
      c.place = 32 << 16;
      c.ends = false;
      c.slot = c.val_off = c.row = c.kind = 0;
      c.aux = 0.0;
      return c;
    }
    c.cnt = min(step_chunk(d), d.z - u);
    c.len = max(0, min(seg - u, c.cnt));
    c.slot = tail;
    if (step_padded<C>(d) || __all_sync(0xffffffffu, u + c.cnt <= seg)) {  // (chunk_place's full form)
      c.place = 32 << 16;
      c.val_off = c.cnt * 32 * static_cast<int>(sizeof(C));
    } else {
      const ChunkPlace at = chunk_place<C>(d, u, c.cnt, seg, lane);
      c.place = at.base | at.stride << 16;
      c.val_off = (at.tot * static_cast<int>(sizeof(C)) + kUnit - 1) & ~(kUnit - 1);
    }
    u += c.cnt;
    c.row = d.x;
    c.kind = d.y;
    c.ends = u >= d.z;
    c.aux = 0.0;
    return c;
  };
  auto next_step = [&] {
    ++s;
    u = 0;
    d = dn;
    seg = lane_segment(d, seg_n, lane);
    dn = load_step(io, step_at(s + 1));
    seg_n = load_seg_len(io, min(s + 1, s1 - 1), lane);
  };
  auto full = [](const Chunk& c) { return c.place == 32 << 16; };
  auto base = [&](const Chunk& c) { return full(c) ? lane : c.place & 0xffff; };
  auto cols = [&](const Chunk& c) { return reinterpret_cast<const C*>(sm.slot(w, c.slot)); };
  auto vals = [&](const Chunk& c) { return reinterpret_cast<const T*>(sm.slot(w, c.slot) + c.val_off); };
  // x of the columns of the step of the chunk being gathered: 16-bit columns are
  // offsets from the step's smallest one
  auto x_of = [&]() -> const X* { return sizeof(C) == 2 ? x + d.w : x; };
  T acc = T(0);
  if constexpr (sizeof(T) == 4) {
    // FP32: an FMA takes no time beside its operands, so nothing hides a chunk's
    // gathers but other gathers: those of two chunks (a 27-entry row) together,
    // and the other warps'.  What bounds it then are the instructions issued: no
    // bookkeeping from chunk to chunk.
    auto gather = [&](const Chunk& c, X* xv) {
      const X* const xb = x_of();
      const C* cp = cols(c);
      if (full(c)) {
        cp += lane;
#pragma unroll
        for (int k = 0; k < kU; ++k) {
          if (k % 3 == 0 && k >= c.cnt) break;
          if (k < c.len) xv[k] = xb[cp[32 * k]];
        }
      } else {
        const int stride = c.place >> 16;
        cp += base(c);
#pragma unroll
        for (int k = 0; k < kU; ++k, cp += stride) {
          if (k % 3 == 0 && k >= c.cnt) break;
          if (k < c.len) xv[k] = xb[*cp];
        }
      }
    };
    auto sum = [&](const Chunk& c, const X* xv) {
      const T* vp = vals(c);
      if (full(c)) {
        vp += lane;
#pragma unroll
        for (int k = 0; k < kU; ++k) {
          if (k % 3 == 0 && k >= c.cnt) break;
          if (k < c.len) acc = fma(vp[32 * k], xv[k], acc);
        }
      } else {
        const int stride = c.place >> 16;
        vp += base(c);
#pragma unroll
        for (int k = 0; k < kU; ++k, vp += stride) {
          if (k % 3 == 0 && k >= c.cnt) break;
          if (k < c.len) acc = fma(*vp, xv[k], acc);
        }
      }
      __syncwarp();  // every lane has read the chunk: its slot is free
      ++consumed;
      if (lane == 0) st_release_shared(&ws->consumed, consumed);
    };
    while (s < s1) {
      const int4 dc = d;
      const int i = result_row(d, lane);
      const double ai = with_dot && i >= 0 ? io.aux[i] : 0.0;
      acc = T(0);
      while (u < d.z) {
        // (zero: a register that is only written under a predicate is live from
        // the kernel's start on, and these would all be spilled)
        X xa[kU], xb[kU];
#pragma unroll
        for (int k = 0; k < kU; ++k) xa[k] = xb[k] = X(0);
        Chunk a = next_chunk(), b;
        if (!wait_next()) return leave(false);
        gather(a, xa);
        const bool two = u < d.z;
        if (two) {
          b = next_chunk();
          if (!wait_next()) return leave(false);
          gather(b, xb);
        }
        sum(a, xa);
        if (two) sum(b, xb);
      }
      next_step();
      const T tot = combine_lanes(step_mode(dc), acc);
      if (i >= 0) {
        const double y = static_cast<double>(tot);
        io.out[i] = y;
        dot = fma(ai, y, dot);
      }
    }
    return leave(true);
  }
  // FP64: behind next_chunk, once its gathers are under way: the next step
  auto after_gather = [&](Chunk& c) {
    if (!c.ends) return;
    const int i = with_dot ? result_row(d, lane) : -1;
    if (i >= 0) c.aux = io.aux[i];
    next_step();
  };
  // the first chunk: gathered, nothing to sum yet
  X xv[kU];
#pragma unroll
  for (int k = 0; k < kU; ++k) xv[k] = X(0);
  Chunk c = next_chunk();
  if (c.cnt > 0) {
    if (!wait_next()) return leave(false);
    const X* const xb = x_of();
    const C* cp = cols(c) + base(c);
    const int stride = c.place >> 16;
#pragma unroll
    for (int k = 0; k < kU; ++k, cp += stride)
      if (k < c.len) xv[k] = xb[*cp];
  }
  after_gather(c);
  // sums chunk c, whose x values are in xv, and gathers those of chunk n
  for (;;) {
    Chunk n = next_chunk();
    if (n.cnt > 0 && !wait_next()) return leave(false);
    const X* const xb = x_of();
    if (full(c) && full(n)) {
      const T* const vp = vals(c) + lane;
      const C* const cp = cols(n) + lane;
      // straight-line code for each size of c
      dispatch_tree<0, kU>(c.cnt, [&](auto N) {
#pragma unroll
        for (int k = 0; k < decltype(N)::value; ++k) {
          if (k < c.len) acc = fma(vp[32 * k], xv[k], acc);
          if (k < n.cnt) xv[k] = xb[cp[32 * k]];
        }
      });
      if (n.cnt > c.cnt) {
#pragma unroll
        for (int k = 0; k < kU; ++k)
          if (k >= c.cnt && k < n.cnt) xv[k] = xb[cp[32 * k]];
      }
    } else {
      // at least one of them in another form
      const T* vp = vals(c) + base(c);
      const C* cp = cols(n) + base(n);
      const int cs = c.place >> 16, ns = n.place >> 16;
#pragma unroll
      for (int k = 0; k < kU; ++k, vp += cs, cp += ns) {
        if (k >= c.cnt) break;
        if (k < c.len) acc = fma(*vp, xv[k], acc);
        if (k < n.len) xv[k] = xb[*cp];
      }
      if (n.cnt > c.cnt) {
        cp = cols(n) + base(n);
#pragma unroll
        for (int k = 0; k < kU; ++k, cp += ns)
          if (k >= c.cnt && k < n.len) xv[k] = xb[*cp];
      }
    }
    after_gather(n);
    if (c.cnt > 0) {
      __syncwarp();  // every lane has read the chunk: its slot is free
      ++consumed;
      if (lane == 0) st_release_shared(&ws->consumed, consumed);
    }
    if (c.ends) {
      const int4 dc = make_int4(c.row, c.kind, 0, 0);
      const T tot = combine_lanes(step_mode(dc), acc);
      const int i = result_row(dc, lane);
      if (i >= 0) {
        const double y = static_cast<double>(tot);
        io.out[i] = y;
        if (with_dot) dot = fma(c.aux, y, dot);
      }
      if (n.cnt < 0) return leave(true);
      acc = T(0);
    }
    c = n;
  }
}

// out = A x in FP64 over the warp's steps [s, s1), read directly from global memory in
// stream order, from chunk `chunk` and (mixed) entry `entry` on: the passes outside a
// mixed solve's step loop (its setup, the final true residual, the residual
// replacements), which leaves the ring's contents alone, and a mixed handle's
// product (kKeep: loads with the L2's default policy).  Latency bounds it: a step's chain would be its chunk's offset, columns,
// x, FMAs, chunk after chunk.  So 32 chunk offsets are loaded at once, and a batch's
// columns while the batch before waits for its x.
template <typename Ring, bool kKeep = false>
__device__ __forceinline__ void direct_pass(const DevCsr& A, uint32_t chunk, int64_t entry, int s, int s1,
                                            const double* x, double* out) {
  using T = typename Ring::Val;
  using C = typename Ring::Col;
  constexpr int kU = 7;  // entries per lane and batch (half an FP32 chunk)
  auto ld = [](const auto* at) { return kKeep ? __ldg(at) : __ldcs(at); };
  const int lane = fresh_tid() & 31;
  for (; s < s1; ++s) {
    const int4 d = A.step[s];
    const int seg = lane_segment(d, A.seg_len[static_cast<size_t>(s) * 32 + lane], lane);
    const double* const xb = sizeof(C) == 2 ? x + d.w : x;
    const int size = step_chunk(d), nchunks = size > 0 ? (d.z + size - 1) / size : 0;
    uint32_t off = lane < nchunks ? A.chunk_off[chunk + lane] : 0;
    // the batch after the one at hand: chunk j of the step, entries [k, ..) of it
    int j = 0, k = 0, cnt = 0;
    ChunkPlace place{0, 0, 0};
    const C* cp = nullptr;
    const double* vp = nullptr;
    int c[kU] = {};
    // columns of the next batch; returns how many of its entries this lane has
    auto load = [&]() -> int {
      const int u = j * size;
      if (k == 0) {
        if (j > 0 && (j & 31) == 0) off = j + lane < nchunks ? A.chunk_off[chunk + j + lane] : 0;
        cnt = min(size, d.z - u);
        place = chunk_place<C>(d, u, cnt, seg, lane);
        const unsigned char* const at = A.stream + static_cast<size_t>(__shfl_sync(0xffffffffu, off, j & 31)) * kUnit;
        cp = reinterpret_cast<const C*>(at) + place.base;
        if constexpr (sizeof(T) == 4) vp = A.val64 + entry + place.base;
        else
          vp = reinterpret_cast<const double*>(at + ((place.tot * static_cast<int>(sizeof(C)) + kUnit - 1) & ~(kUnit - 1))) +
               place.base;
        entry += place.tot;
      }
      const int len = max(0, min(min(seg - u, cnt) - k, kU));
#pragma unroll
      for (int i = 0; i < kU; ++i, cp += place.stride)
        if (i < len) c[i] = static_cast<int>(ld(cp));
      return len;
    };
    double acc = 0.0;
    int len = nchunks > 0 ? load() : 0;
    while (j < nchunks) {
      double a[kU], g[kU];
#pragma unroll
      for (int i = 0; i < kU; ++i) a[i] = g[i] = 0.0;  // (not live before: no spills)
#pragma unroll
      for (int i = 0; i < kU; ++i, vp += place.stride)
        if (i < len) {
          a[i] = ld(vp);
          g[i] = xb[c[i]];
        }
      const int now = len, most = cnt - k;  // (most: warp-uniform)
      k += kU;
      if (k >= cnt) {
        k = 0;
        ++j;
      }
      if (j < nchunks) len = load();
#pragma unroll
      for (int i = 0; i < kU; ++i) {
        if (i >= most) break;  // (a predicated-off FMA would take the pipe's time)
        if (i < now) acc = fma(a[i], g[i], acc);
      }
    }
    chunk += static_cast<uint32_t>(nchunks);
    const double tot = combine_lanes(step_mode(d), acc);
    const int i = result_row(d, lane);
    if (i >= 0) out[i] = tot;
  }
}

}  // namespace cgk
