// Internal structures shared by the host side of the C-ABI and the kernels.
// Not part of the public interface (that is include/cg.h).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace cgk {

// The persistent kernels run one CTA per SM: kWarps warps that compute, each
// its own steps of the CTA's rows from its own ring in shared memory, and one
// producer warp, whose lane w fills warp w's ring with 1-D TMA bulk copies.
// Nineteen computing warps (with the producer five per SM sub-partition), 96
// registers per thread, nothing spilled.  15, 19, 23
// warps, us per step of a Q1 solve: 32^3 14.2, 12.9, 13.1; 64^3 28.9, 27.6, 29.0;
// 160^3 292, 267, 266; 160^3 mixed 230, 214, 207 (before the uneven chunks went
// lane after lane).
constexpr int kWarps = 19;
constexpr int kBlock = kWarps * 32;      // their threads
constexpr int kThreads = kBlock + 32;    // and the producer warp
constexpr int kCtasPerSm = 1;

// A step is what a warp computes at once: 32 lanes, each summing one segment
// of at most kLaneMax entries (up to 32 rows of <= 32 entries, one lane per
// row; up to 16 rows of 33..64 entries, two lanes per row), or one longer row,
// whose entries the lanes stride (a segment per lane of any length).  Step k
// of a CTA goes to computing warp k modulo their number.
//
// The handle stores the matrix as one stream per warp: the entries of the
// warp's steps in the order in which the warp consumes them.  Within a chunk
// (below) that is entry u of every lane's segment, in lane order, then entry
// u + 1, and so on, free of bank conflicts in shared memory; or, where the lanes'
// segments differ in length and are not padded, lane after lane.
// A warp works through a step in chunks of a few entries per lane;
// a chunk is one slot of the warp's ring, so that the ring gives back its
// oldest bytes after every few entries and not only after a whole step.
// FP64 9: a 27-entry row is three full chunks, an 18-entry one two (14, i.e. two
// chunks, was slower: 64^3 33.1 against 29.3 us per step, with 15 warps).  FP32
// 14: a 27-entry row is two chunks, which are gathered together (9, gathered one
// chunk ahead as in FP64: 26.5 against 25.2 us, with 15 warps).
// FP32 with 32-bit columns 11: the rings then leave 92 KB of L1 instead of 28, and
// scattered gathers have one L1 line each (110^3 mesh in random numbering, chunks of
// 9, 10, 11, 12, 14: 145, 144, 144, 155, 250 us per step; in its own numbering 84,
// 84, 84, 87, 115; rows of 1 to 32 entries 31.0, 31.5, 26.1, 27.1, 27.0).
__host__ __device__ constexpr int max_chunk(bool mixed, bool col16) { return !mixed ? 9 : col16 ? 14 : 11; }
// A segment of `len` entries split evenly over as few chunks of at most `most` as
// it takes: the entries of one chunk.
__host__ __device__ constexpr int chunk_of(int len, int most) {
  return len <= 0 ? 0 : (len + (len + most - 1) / most - 1) / ((len + most - 1) / most);
}
// Slots of a warp's ring: the chunk being summed, the next one and a copy in
// flight, 150 to 200 KB in all.  The rest of the SM's 256 KB serves the gathers
// as L1.  (Two slots: 160^3 383 against 292 us per step, with 15 warps.)
constexpr int kSlots = 3;
// The producer warp's wait for a slot, beyond four waits of the computing warps.
constexpr unsigned long long kProducerIdleNs = 60000000000ull;
constexpr int kLaneMax = 32;  // longest row computed by a single lane
// Largest CTA share (rows) of the small-share solve kernels, which keep the
// share's r in shared memory (20 KB behind the ring layout; the FP64 layout
// with 32-bit columns then takes 221 KB of the 227 KB a CTA may have).
constexpr int kLocalRows = 2560;

// A chunk in memory, and in a slot: its columns, then its values, each padded
// to a multiple of kUnit bytes (the granularity of a bulk copy: one copy per
// chunk).  Full chunks (every lane has all of their entries) need no padding.
constexpr int kUnit = 16;
__host__ __device__ constexpr int64_t units(int64_t bytes) { return (bytes + kUnit - 1) / kUnit; }
__host__ __device__ constexpr int64_t chunk_units(int64_t entries, int col_bytes, int val_bytes) {
  return units(entries * col_bytes) + units(entries * val_bytes);
}

enum StepMode : int32_t {
  kLanePerRow = 0,   // lane l computes row r0 + l (rows of <= kLaneMax entries)
  kPairPerRow = 1,   // lanes 2t, 2t+1 split row r0 + t (rows of <= 2 kLaneMax entries)
  kLongRow = 2,      // the whole row r0; lanes stride it
};
// The fields of a step: {first row, kind word, longest segment, smallest column}.
// Kind word: bits 0..7 the lanes that hold a segment (from lane 0), bits 8..9
// the StepMode, bit 10 set if all of them have the longest segment's length,
// bit 11 the padding rule below, bits 16..21 (kLongRow) the lanes of the last,
// partial stride, bits 24..29 the chunk (entries per lane): the segment split
// evenly over as few chunks as it takes.
constexpr int kStepModeShift = 8;
constexpr int kStepUniform = 1 << 10;
constexpr int kStepPadded = 1 << 11;
constexpr int kStepRemShift = 16;
constexpr int kStepChunkShift = 24;
constexpr int kStepChunkMask = 63;
// Columns are stored as 16-bit offsets from their step's smallest column when
// every step of the matrix spans at most this much, and as 32-bit columns
// otherwise.
constexpr int64_t kColSpan16 = 65535;
// With 16-bit columns, a step whose lanes differ in length, or that fills only
// some lanes, is padded to the longest segment in all 32 lanes where that adds
// at most half (`tight`, where memory is short: an eighth): an entry's place is
// then a constant offset.  Other steps hold their entries only (chunk_place).
// Padding is never multiplied.  (At most an eighth, a quarter, a half, all of it,
// when the other steps still cost two votes per entry: product of the 110^3 mesh
// 95, 88, 84, 83 us; step of Q1 64^3 mixed 21.0, 20.9, 19.6, 19.6 us.)
constexpr bool step_pads(int64_t longest, int64_t entries, bool tight) {
  return tight ? 8 * 32 * longest <= 9 * entries : 2 * 32 * longest <= 3 * entries;
}

// Device view of a CSR matrix in stream order.
struct DevCsr {
  const unsigned char* stream;  // the chunks: columns (col16) and FP64 values, or FP32 ones (mixed precision)
  const double* val64;        // mixed precision: FP64 values in stream order (entries, padding included)
  const int4* step;           // [nsteps + 1] see above (one trailing sentinel)
  const int32_t* step_cmax;   // [nsteps] largest column of each step (-1: no entries), or nullptr
  const uint8_t* seg_len;     // [32 * nsteps] entries of each lane's segment (not of kLongRow steps)
  const uint32_t* chunk_off;  // [chunks + 1] first unit of each chunk, stream by stream
  const int4* warp_chunk;     // [nblocks * kWarps] each warp's stream: first chunk, number of chunks,
                              // start and end of the first one (units)
  const uint32_t* warp_entry; // mixed precision: [nblocks * kWarps] its first entry in val64
  const uint32_t* step_chunk; // mixed precision, a handle's: [nsteps] first chunk of each step,
  const uint32_t* step_entry; // [nsteps] and its first entry in val64
  const int32_t* warp_step;   // [nblocks * kWarps + 1] first step of each warp (stream by stream)
  const int32_t* block_row;   // [nblocks + 1] first row of each CTA (vector phases)
  int32_t n;
  int32_t nsteps;
  int32_t nblocks;            // CTAs the partition was balanced for
  int32_t max_rows;           // most rows in one CTA's range (host side; 0 if unknown)
  int64_t nnz;
  int32_t col16;              // 1: 16-bit column offsets
  int32_t keep;               // 1: the streams stay in the L2 (streams_stay)
};

// Whether a solve of A in one launch (chunk_iters <= 0) runs the small-share
// kernel: every CTA's range fits kLocalRows.
inline bool small_share(const DevCsr& A, int64_t chunk_iters) {
  return A.max_rows > 0 && A.max_rows <= kLocalRows && chunk_iters <= 0;
}

// Control block of one solve, in device memory, cleared before its first
// launch.  A solve may run over several launches (batched solves advance
// each system a bounded number of steps per launch): the fields below
// `phase` carry its state from one launch to the next.
enum SolvePhase : int32_t { kPhaseNew = 0, kPhaseRunning = 1, kPhaseDone = 2 };
struct SolveCtrl {
  unsigned long long barrier;   // monotonic arrival counter of the group barrier
  int32_t abort;                // set by any CTA that gives up (timeout)
  int32_t status;               // CG_* code
  int64_t iters;                // steps done
  double rho;                   // r.z of the current iterate (r.r without preconditioner)
  double bnorm2;                // b.b
  double relres_rec;            // ||r||/||b|| of the recursive residual
  double relres_true;           // ||b - A x|| / ||b||
  int32_t timeout_site;         // which wait gave up (diagnostics)
  int32_t phase;                // SolvePhase
  unsigned long long rounds;    // group-barrier rounds completed so far
  int32_t slot;                 // partial-sum slot the next group sum uses
  int32_t pad;
  // The step sums' accumulators (acc_words): two words for each of p.q, r.r
  // and r.z, never cleared during a solve; their values and the exponents of the
  // last sums at the end of a launch.
  alignas(16) unsigned long long acc[3][2];
  unsigned long long acc_seen[3][2];
  int32_t acc_exp[3];
  int32_t pad2;
};
static_assert(sizeof(SolveCtrl) % 16 == 0, "accumulators on 16 bytes in a table");

struct SolveParams {
  DevCsr A;
  const double* b;
  double* x;
  double* r;
  double* p;
  double* q;
  float* p32;                   // FP32 shadow of p (mixed precision) or nullptr
  double* partials;             // [2][nblocks][2] per-CTA partial sums, two slots
  SolveCtrl* ctrl;
  double tol;
  int64_t maxit;
  int64_t replace_every;        // mixed precision: true-residual period
  unsigned long long wait_limit_ns;  // bound on every device-side wait
  int32_t group;                // CTAs that solve this system together (its partition's CTA count)
  int32_t stream_rows;          // single-system kernels: row tables evict-first (stream_row_tables)
  int64_t chunk_iters;          // steps per launch (<= 0: until the solve ends)
  const double* dinv;           // Jacobi preconditioner 1/diag(A), or nullptr (plain CG)
  // Single-system solves: one epoch flag per CTA (zeroed before the launch).
  // In the large-share kernel a CTA publishes the step number in its flag
  // after its p update and waits only for the CTAs whose rows its own rows'
  // columns reach, instead of a barrier of the whole group.  nullptr (and
  // the other kernels): the group barrier.
  unsigned long long* flags;
};

// Batched solves: one persistent launch over many systems.  Every CTA takes
// tasks from a queue; a task is one CTA's share (rank) of one system.
struct BatchTask {
  int32_t sys;                  // index into the system table
  int32_t rank;                 // 0 .. group-1
};
struct BatchQueue {
  int32_t ntasks;
  int32_t stream_rows;          // row tables evict-first in this launch (stream_row_tables)
  int32_t keep;                 // the streams stay in the L2 (streams_stay)
  int32_t pad;
  BatchTask task[1];            // ntasks entries (allocated to capacity)
};
struct BatchParams {
  const SolveParams* sys;       // system table (one entry per slot)
  const BatchQueue* queue;      // tasks of this launch, longest time per CTA first
  int32_t* next;                // next task to take (zeroed before each launch)
};

// Bytes that a step of the CG iteration on n rows reads again in the next
// step: p, q and r, up to 4 bytes per row of row and step tables, the FP32
// copy of p (mixed precision) and 1/diag(A) (Jacobi).  x and the matrix stream
// through with the evict-first policy.
inline int64_t step_reused_bytes(int64_t n, bool mixed, bool jacobi) {
  return n * (28 + (mixed ? 4 : 0) + (jacobi ? 8 : 0));
}

// Whether the product loads the row and step tables (read once per product)
// with the evict-first policy: when the bytes that the running steps read
// again take more than 4/7 of the L2.  Below that, tables and vectors both
// stay in the L2 from step to step; above it the tables are the better ones
// to give up.
inline bool stream_row_tables(int64_t reused_bytes, int64_t l2_bytes) {
  return l2_bytes > 0 && 7 * reused_bytes > 4 * l2_bytes;
}

// Whether the matrix streams are read with the L2's default policy instead of
// evict-first: when they and the bytes that the running steps read again take at
// most 3/4 of the L2, and so stay there.  Evict-first then only costs energy (Q1
// 64^3, FP64 step 14.1 -> 10.6 mJ at the same 25 us, mixed 9.4 -> 7.8); where they do
// not fit, it keeps the vectors in (72^3 35.5 us with it, 35.8 without; 90^3 53.9,
// 58.8; 160^3 274, 283).
inline bool streams_stay(int64_t stream_bytes, int64_t reused_bytes, int64_t l2_bytes) {
  return 4 * (stream_bytes + reused_bytes) <= 3 * l2_bytes;
}

// Status codes (same values as include/cg.h).
enum : int32_t {
  kOK = 0, kEINVAL = 1, kENOMEM = 2, kECUDA = 3, kENOTCONV = 4,
  kEBREAKDOWN = 5, kETIMEOUT = 6, kEBUSY = 7,
};

// Launchers (defined in the .cu files; return the CUDA error of the launch).
// ---- stream order (layout.cu)
// Source of a matrix in CSR form on the device: row_ptr 0-based; col_idx and
// val hold the entries from e_first on, columns based at `base`.
struct CsrSource {
  const int32_t* row_ptr;
  const int32_t* col_idx;
  const double* val;
  int64_t e_first;
  int32_t base;
};
// What layout_scan found, cleared before it: the widest step (largest minus
// smallest column), and (if asked to check) the first entry whose column lies
// outside [base, n + base).
struct LayoutScan {
  int32_t span;
  int32_t pad;
  unsigned long long bad_entry;  // ~entry (so that a maximum finds the first), 0: none
};
// For the steps among [s0, s1) that begin in rows [row0, row1): the lanes' segment lengths into seg_len[], the smallest
// column into step[].w (0 for a step without entries), the largest into cmax[]
// (if not nullptr; -1 without entries), span and bad entries into *out.
cudaError_t launch_layout_scan(const CsrSource& src, int4* step, uint8_t* seg_len, int32_t* cmax, int32_t s0, int32_t s1,
                               int32_t row0, int32_t row1, int64_t n, bool check, LayoutScan* out, cudaStream_t s);
// Writes the entries of the same steps in stream order: into `stream` the
// chunks step_chunk[k].. of step k, at the units that chunk_off gives (16-bit
// column offsets if col16, else 32-bit columns; FP32 values, rounded to nearest,
// if mixed), and if mixed the FP64 values from val64[step_entry[k]] on.
// Padding of entries: zeros.  Sets the steps' chunk sizes to those of the column
// width (max_chunk).
struct StreamPlace {
  const uint32_t* chunk_off;
  const uint32_t* step_chunk;
  const uint32_t* step_entry;  // mixed
  unsigned char* stream;
  double* val64;               // mixed
};
cudaError_t launch_layout_fill(const CsrSource& src, int4* step, const StreamPlace& to, int32_t s0, int32_t s1,
                               int32_t row0, int32_t row1, bool col16, bool mixed, cudaStream_t s);
// dinv[i] = 1 / (sum of row i's stored entries in column i) for rows [row0, row1);
// err set to the first row (+1) found whose diagonal is not positive.
cudaError_t launch_jacobi_dinv(const CsrSource& src, int64_t row0, int64_t row1, double* dinv, int32_t* err,
                               cudaStream_t s);

cudaError_t launch_spmv(const DevCsr& A, const double* x, double* y, int32_t* err, cudaStream_t s);
cudaError_t launch_dot(int64_t n, const double* x, const double* y, double* out,
                       double* partials, unsigned int* counter, int grid, cudaStream_t s);
cudaError_t launch_axpy(int64_t n, double a, const double* x, double* y, cudaStream_t s);
cudaError_t launch_ewmul(int64_t n, const double* x, const double* y, double* z, cudaStream_t s);
cudaError_t launch_solve(const SolveParams& P, bool mixed, cudaStream_t s);
int solve_blocks_per_sm(bool mixed, bool jacobi);   // occupancy of the persistent kernel
// The batched solve (cooperative launch of `nblocks` CTAs, one per SM).
cudaError_t launch_batch(const BatchParams& B, bool mixed, bool jacobi, int nblocks, cudaStream_t s);
int batch_blocks_per_sm(bool mixed, bool jacobi);
int dot_grid(int64_t n, int num_sms);
// Streamed dot product (x and y 16-byte aligned, n >= dot_stream_min_n()):
// `grid` = dot_stream_grid(n, SMs) CTAs; err[0] is raised by a wait that gave
// up, and the last CTA moves it to err[1] (the result is then NaN) and clears
// it.
cudaError_t launch_dot_stream(int64_t n, const double* x, const double* y, double* out, double* partials,
                              unsigned int* counter, int32_t* err, int grid, unsigned long long limit_ns,
                              cudaStream_t s);
int dot_stream_grid(int64_t n, int num_sms);
int64_t dot_stream_min_n();
// FP64 FMA throughput probe: `grid` CTAs of 256 threads, each thread 8
// independent chains of 4 x iters FMAs.
constexpr int kFp64ProbeThreads = 256;
constexpr int kFp64ProbeFmasPerIter = 32;
cudaError_t launch_fp64_probe(int64_t iters, int grid, double* sink, cudaStream_t s);
cudaError_t launch_wait_timeout_selftest(SolveCtrl* ctrl, unsigned long long limit_ns, cudaStream_t s);

// Small systems on one thread-block cluster (cluster_solve.cu): kClusterCtas
// CTAs of kClusterThreads threads, each holding R consecutive rows (R a power
// of two, at most kClusterMaxRows) and up to E entries in shared memory.
constexpr int kClusterCtas = 16;  // a non-portable cluster size (opted in)
constexpr int kClusterThreads = 512;
constexpr int kClusterMaxRows = 1024;
size_t cluster_smem_bytes(int R, int E);
// Clusters of this layout that can be resident at once (0: none, or an error).
int cluster_max_active(int R, int E);
cudaError_t launch_cluster_solve(const int32_t* row_ptr, const int32_t* col_idx, const double* val,
                                 const double* b, double* x, SolveCtrl* ctrl, double tol, int64_t maxit, int32_t n,
                                 int32_t R, int32_t E, cudaStream_t s);
// timeout_site the self-test's wait records
constexpr int32_t kSelftestSite = 99;
// timeout_site of a single-system solve's wait for its neighbours' p
constexpr int32_t kNeighborSite = 98;
// timeout_site of a wait for a sum through the accumulators
constexpr int32_t kAccSite = 96;
// timeout_site of the matrix stream: a copy that did not arrive, or a ring that
// stayed full
constexpr int32_t kStreamSite = 95;
// timeout_site of the synchronisation probe's barrier
constexpr int32_t kProbeSite = 97;
// The solves' group-wide synchronisations timed alone (cg_probe_group_sync):
// a cooperative launch of `nblocks` CTAs (one per SM) running `iters` group
// barriers (mode 0) or group sums (mode 1); ctrl zeroed before the launch,
// partials 2 * nblocks doubles, out nblocks doubles.
cudaError_t launch_sync_probe(SolveCtrl* ctrl, double* partials, int iters, int mode, int nblocks,
                              unsigned long long limit_ns, double* out, cudaStream_t s);
// Shared-memory bytes of a persistent solve CTA (FP32 ring values if mixed,
// 16- or 32-bit columns;
// `local`: the small-share kernels, with r of the share).
size_t solve_smem_bytes(bool mixed, bool col16, bool local = false);
// Opt a kernel in to `bytes` of dynamic shared memory with the smallest
// carveout that holds them (once per kernel and device).
cudaError_t ensure_smem_attr(const void* kernel, size_t bytes);

}  // namespace cgk
