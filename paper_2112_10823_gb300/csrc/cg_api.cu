// Host side of the C ABI declared in include/cg.h: argument checks, CSR
// validation and upload, the row partition of the persistent kernels, device
// memory ownership, and the launch + read-back of each call.
#include <cmath>
#include <cstdio>
#include <algorithm>
#include <cstring>
#include <initializer_list>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <tuple>
#include <utility>
#include <vector>

#include "../../include/cg.h"
#include "cg_internal.h"
#include "host_util.h"

using cgh::Partition;
using cgh::build_partition;

namespace cgk {
cudaError_t launch_dot_noalloc(int64_t n, const double* x, const double* y, double* out, cudaStream_t s);
int64_t dot_noalloc_max_n();
}

namespace cgh {

// Row partition of the persistent kernels.  Rows are split into `nblocks`
// contiguous CTA ranges of about equal cost (stored entries + kRowCost per
// row, the per-row vector work), and each CTA range into steps (see
// cg_internal.h): up to 32 rows of <= 32 entries (one lane per row), up to 16
// rows of <= 64 entries (two lanes per row), or one longer row.  kRowCost is
// flat between 10 and 18 (160^3 within 0.3 %, 100^3 2 %).
constexpr int64_t kRowCost = 14;

int64_t cost_split(const std::vector<int32_t>& rp, int64_t lo_row, int64_t hi_row, int64_t part, int64_t parts) {
  // first row i in [lo_row, hi_row] with cost(lo_row, i) >= cost(lo_row, hi_row) * part / parts
  const int64_t c0 = static_cast<int64_t>(rp[lo_row]) + kRowCost * lo_row;
  const int64_t c1 = static_cast<int64_t>(rp[hi_row]) + kRowCost * hi_row;
  const int64_t goal = c0 + ((c1 - c0) * part) / parts;
  int64_t lo = lo_row, hi = hi_row;
  while (lo < hi) {
    const int64_t mid = (lo + hi) / 2;
    if (static_cast<int64_t>(rp[mid]) + kRowCost * mid >= goal) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

StepShape::StepShape() {
  for (int L = 0; L <= kShapeMaxLen; ++L)
    mode[L] = static_cast<int8_t>(L <= cgk::kLaneMax ? cgk::kLanePerRow : cgk::kPairPerRow);
}

bool StepShape::valid() const {
  for (int L = 0; L <= kShapeMaxLen; ++L) {
    const int m = mode[L];
    if (m != cgk::kLanePerRow && m != cgk::kPairPerRow && m != cgk::kLongRow) return false;
    if (m == cgk::kLanePerRow && L > cgk::kLaneMax) return false;
  }
  return true;
}

// (the chunk size is left to place_steps)
static int4 make_step(int64_t row, int lanes, int mode, bool uniform, int rem, int64_t seg, int64_t entries,
                      bool tight) {
  const bool pads = (lanes < 32 || !uniform) && cgk::step_pads(seg, entries, tight);
  unsigned int y = static_cast<unsigned int>(lanes) | static_cast<unsigned int>(mode) << cgk::kStepModeShift |
                   (uniform ? static_cast<unsigned int>(cgk::kStepUniform) : 0u) |
                   (pads ? static_cast<unsigned int>(cgk::kStepPadded) : 0u) |
                   static_cast<unsigned int>(rem) << cgk::kStepRemShift;
  return make_int4(static_cast<int>(row), static_cast<int>(y), static_cast<int>(seg), 0);
}

// The steps of rows [row, end) in row order into out[] (room for a step per row);
// returns their number and adds up P.chunks and P.padded.
static size_t warp_steps(const std::vector<int32_t>& rp, int64_t row, int64_t end, const StepShape& shape, bool mixed,
                         int4* out, Partition& P) {
  // (the column width is not known yet: 32-bit columns have the smaller chunks)
  constexpr int kChunk64 = cgk::max_chunk(false, false), kChunk32 = cgk::max_chunk(true, false);
  static_assert(kChunk32 <= cgk::max_chunk(true, true), "an upper bound of the chunks");
  size_t count = 0;
  int64_t chunks = 0, padded = 0;
  auto step = [&](int64_t first, int lanes, int mode, bool uniform, int rem, int64_t seg, int64_t entries) {
    const int4 d = make_step(first, lanes, mode, uniform, rem, seg, entries, shape.tight);
    out[count++] = d;
    chunks += mixed ? (seg + kChunk32 - 1) / kChunk32 : (seg + kChunk64 - 1) / kChunk64;
    padded += (d.y & cgk::kStepPadded) ? 32 * seg : entries;
  };
  auto kind = [&](int64_t len) -> int { return len > kShapeMaxLen ? cgk::kLongRow : shape.mode[len]; };
  int short_rows = -1;  // rows of up to this many entries are all of one lane
  while (short_rows < kShapeMaxLen && shape.mode[short_rows + 1] == cgk::kLanePerRow) ++short_rows;
  while (row < end) {
    // 32 such rows are a step (the usual case, in loops that the compiler vectorises:
    // 4.1 M rows 10.1 ms row by row, 1.9 so)
    if (row + 32 <= end && rp[row + 1] - rp[row] <= short_rows) {
      const int32_t* const at = rp.data() + row;
      int32_t longest = 0, shortest = INT32_MAX;
      for (int k = 0; k < 32; ++k) {
        const int32_t len = at[k + 1] - at[k];
        longest = longest > len ? longest : len;
        shortest = shortest < len ? shortest : len;
      }
      if (longest <= short_rows) {
        step(row, 32, cgk::kLanePerRow, shortest == longest, 0, longest, at[32] - at[0]);
        row += 32;
        continue;
      }
    }
    const int64_t len0 = rp[row + 1] - rp[row];
    if (kind(len0) == cgk::kLongRow) {  // a warp per row
      const int rem = static_cast<int>(len0 % 32);
      step(row, 32, cgk::kLongRow, rem == 0, rem, (len0 + 31) / 32, len0);
      ++row;
      continue;
    }
    const int64_t start = row;
    int64_t maxlen = 0, minlen = 0;
    int m = cgk::kLanePerRow;  // the widest kind so far (one lane < two lanes)
    while (row < end) {
      const int64_t len = rp[row + 1] - rp[row];
      const int k = kind(len);
      if (k == cgk::kLongRow) break;
      const int nm = std::max(m, k);
      const int64_t cap = nm == cgk::kLanePerRow ? 32 : 16;
      if (row - start + 1 > cap) break;
      maxlen = std::max(maxlen, len);
      minlen = row == start ? len : std::min(minlen, len);
      m = nm;
      ++row;
    }
    const int rows = static_cast<int>(row - start);
    const int64_t cnt = rp[row] - rp[start];
    if (m == cgk::kLanePerRow)
      step(start, rows, m, minlen == maxlen, 0, maxlen, cnt);
    else  // two segments per row, the first one longer by an odd entry
      step(start, 2 * rows, m, minlen == maxlen && maxlen % 2 == 0, 0, (maxlen + 1) / 2, cnt);
  }
  P.chunks += chunks;
  P.padded += padded;
  return count;
}

// Rows of step k of P.
static int64_t rows_of(const int4& d) {
  const int lanes = d.y & 0xff, mode = (d.y >> cgk::kStepModeShift) & 3;
  return mode == cgk::kLanePerRow ? lanes : mode == cgk::kPairPerRow ? lanes / 2 : 1;
}

void build_partition(const std::vector<int32_t>& rp, int64_t n, int nblocks, bool mixed, Partition& P,
                     const StepShape& shape) {
  P.step.clear();
  P.block_row.assign(static_cast<size_t>(nblocks) + 1, 0);
  for (int b = 0; b <= nblocks; ++b) P.block_row[b] = static_cast<int32_t>(cost_split(rp, 0, n, b, nblocks));
  P.block_row[nblocks] = static_cast<int32_t>(n);
  P.warp_step.clear();
  P.chunks = P.padded = 0;
  int32_t most_rows = 1;
  for (int b = 0; b < nblocks; ++b) most_rows = std::max(most_rows, P.block_row[b + 1] - P.block_row[b]);
  std::unique_ptr<int4[]> rows(new int4[static_cast<size_t>(most_rows)]);  // a CTA's steps in row order (not cleared)
  for (int b = 0; b < nblocks; ++b) {
    const size_t count = warp_steps(rp, P.block_row[b], P.block_row[b + 1], shape, mixed, rows.get(), P);
    if (b == 0) P.step.reserve((count + count / 8 + 1) * static_cast<size_t>(nblocks));  // (CTAs are alike)
    for (int w = 0; w < cgk::kWarps; ++w) {
      P.warp_step.push_back(static_cast<int32_t>(P.step.size()));
      for (size_t k = static_cast<size_t>(w); k < count; k += cgk::kWarps) P.step.push_back(rows[k]);
    }
  }
  P.warp_step.push_back(static_cast<int32_t>(P.step.size()));
  P.step.push_back(make_step(n, 32, cgk::kLanePerRow, true, 0, 0, 0, false));  // the sentinel: no entries
}

// Calls f(entries) for each chunk of step d, in order.
template <bool kCol16, bool kMixed, typename F>
static void for_chunks(const std::vector<int32_t>& rp, const int4& d, F&& f) {
  const int size = cgk::chunk_of(d.z, cgk::max_chunk(kMixed, kCol16)), lanes = d.y & 0xff, seg = d.z;
  const int mode = (d.y >> cgk::kStepModeShift) & 3;
  const bool padded = kCol16 && (d.y & cgk::kStepPadded);
  if (padded || (d.y & cgk::kStepUniform)) {
    const int64_t each = padded ? 32 : lanes;
    for (int u = 0; u < seg; u += size) f(each * std::min(size, seg - u));  // (size > 0 when seg is)
  } else if (mode == cgk::kLongRow) {  // all lanes but in the last, partial stride
    const int rem = (d.y >> cgk::kStepRemShift) & 0x3f;
    for (int u = 0; u < seg; u += size) {
      const int64_t cnt = std::min(size, seg - u);
      f(u + cnt == seg ? 32 * (cnt - 1) + rem : 32 * cnt);
    }
  } else {
    int32_t len[32] = {};
    const int rows = static_cast<int>(rows_of(d));
    const int32_t* const at = rp.data() + d.x;
    if (mode == cgk::kLanePerRow) {
      for (int i = 0; i < rows; ++i) len[i] = at[i + 1] - at[i];
    } else {
      for (int i = 0; i < rows; ++i) {
        len[i] = (at[i + 1] - at[i] + 1) / 2;
        len[16 + i] = (at[i + 1] - at[i]) / 2;
      }
    }
    for (int u = 0; u < seg; u += size) {
      const int cnt = std::min(size, seg - u);
      int tot = 0;
      for (int i = 0; i < 32; ++i) {
        const int left = len[i] - u < cnt ? len[i] - u : cnt;
        tot += left > 0 ? left : 0;
      }
      f(tot);
    }
  }
}

template <bool kCol16, bool kMixed>
static void place(const std::vector<int32_t>& rp, int nblocks, Partition& P) {
  const size_t warps = static_cast<size_t>(nblocks) * cgk::kWarps;
  P.step_chunk.assign(P.step.size(), 0);
  P.step_entry.assign(kMixed ? P.step.size() : 0, 0);
  P.warp_chunk.assign(warps, int4{0, 0, 0, 0});
  P.warp_entry.assign(kMixed ? warps : 0, 0);
  P.chunk_off.resize(static_cast<size_t>(P.chunks) + 1);
  int64_t at = 0, entry = 0;
  size_t chunk = 0;
  for (size_t bw = 0; bw < warps; ++bw) {
    const size_t c0 = chunk;
    if (kMixed) P.warp_entry[bw] = static_cast<uint32_t>(entry);
    for (int k = P.warp_step[bw]; k < P.warp_step[bw + 1]; ++k) {
      P.step_chunk[k] = static_cast<uint32_t>(chunk);
      if (kMixed) P.step_entry[k] = static_cast<uint32_t>(entry);
      for_chunks<kCol16, kMixed>(rp, P.step[k], [&](int64_t cnt) {
        P.chunk_off[chunk++] = static_cast<uint32_t>(at);
        at += cgk::chunk_units(cnt, kCol16 ? 2 : 4, kMixed ? 4 : 8);
        entry += cnt;
      });
    }
    P.warp_chunk[bw].x = static_cast<int32_t>(c0);
    P.warp_chunk[bw].y = static_cast<int32_t>(chunk - c0);
  }
  P.chunk_off[chunk] = static_cast<uint32_t>(at);
  P.chunk_off.resize(chunk + 1);
  for (int4& c : P.warp_chunk) {
    c.z = static_cast<int32_t>(P.chunk_off[static_cast<size_t>(c.x)]);
    c.w = static_cast<int32_t>(P.chunk_off[static_cast<size_t>(c.x) + (c.y > 0)]);
  }
  P.stream_units = at;
  P.entries = entry;
}

void place_steps(const std::vector<int32_t>& rp, int nblocks, bool col16, bool mixed, Partition& P) {
  if (mixed) col16 ? place<true, true>(rp, nblocks, P) : place<false, true>(rp, nblocks, P);
  else col16 ? place<true, false>(rp, nblocks, P) : place<false, false>(rp, nblocks, P);
}

void stream_bound(int64_t nnz, bool mixed, const Partition& P, int64_t* stream_units, int64_t* entries) {
  // 32-bit columns without padding or 16-bit ones with it; at most a unit lost
  // behind the columns and behind the values of a chunk
  const int64_t value = mixed ? 4 : 8;
  *stream_units = cgk::units(std::max((4 + value) * nnz, (2 + value) * P.padded)) + 2 * P.chunks;
  *entries = P.padded;
}

}  // namespace cgh

struct cg_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  int precision = CG_PREC_FP64;
  int preconditioner = CG_PRECOND_NONE;
  int replace_every = 50;
  unsigned long long wait_limit_ns = 2000000000ull;
  int64_t n = 0, nnz = 0;
  int num_sms = 0;
  int nblocks = 0;
  int nsteps = 0;
  int max_rows = 0;  // most rows in one CTA's range
  int cluster_R = 0;  // > 0: cg_solve runs the cluster kernel, R rows and E entries per CTA
  int cluster_E = 0;
  bool col16 = false;  // columns stored as 16-bit offsets
  int64_t stream_bytes = 0;
  // device memory owned by the handle: the matrix in stream order
  unsigned char* d_stream = nullptr;
  double* d_val64 = nullptr;
  int4* d_step = nullptr;
  int32_t* d_step_cmax = nullptr;
  uint8_t* d_seg_len = nullptr;
  uint32_t* d_chunk_off = nullptr;
  int4* d_warp_chunk = nullptr;
  uint32_t* d_warp_entry = nullptr;
  uint32_t* d_step_chunk = nullptr;  // mixed precision
  uint32_t* d_step_entry = nullptr;
  int32_t* d_warp_step = nullptr;
  int32_t* d_block_row = nullptr;
  // the CSR arrays (0-based), kept for the cluster kernel only
  int32_t* d_csr_row_ptr = nullptr;
  int32_t* d_csr_col = nullptr;
  double* d_csr_val = nullptr;
  double* d_r = nullptr;
  double* d_p = nullptr;
  double* d_q = nullptr;
  float* d_p32 = nullptr;
  double* d_dinv = nullptr;   // Jacobi: 1 / diag(A)
  double* d_xbuf = nullptr;   // staging of host x
  double* d_bbuf = nullptr;   // staging of host b
  double* d_partials = nullptr;
  cgk::SolveCtrl* d_ctrl = nullptr;  // followed by the CTAs' epoch flags (one allocation, one memset per solve)
  unsigned long long* d_flags = nullptr;
  int32_t* d_err = nullptr;
  cgk::SolveCtrl* h_ctrl = nullptr;  // pinned
  std::vector<void*> allocs;
  std::string err;
};

namespace {

thread_local std::string g_create_err;

int fail(cg_ctx* h, int code, const std::string& msg) {
  if (h) h->err = msg;
  else g_create_err = msg;
  return code;
}

int cuda_fail(cg_ctx* h, cudaError_t e, const char* what) {
  std::string m = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
  return fail(h, e == cudaErrorMemoryAllocation ? CG_ENOMEM : CG_ECUDA, m);
}

// The control block of a solve followed by one epoch flag per CTA.
constexpr size_t ctrl_flags_offset() { return (sizeof(cgk::SolveCtrl) + 15) & ~size_t(15); }
size_t ctrl_block_bytes(int nblocks) {
  return ctrl_flags_offset() + sizeof(unsigned long long) * static_cast<size_t>(nblocks > 0 ? nblocks : 1);
}

// Arrays of one device allocation, each on a 256-byte boundary: a handle has some
// twenty of them, and an allocation of its own for each took a third of the time
// that a small system's handle needs.
struct Block {
  size_t bytes = 0;
  std::vector<std::pair<void**, size_t>> parts;
  template <typename T>
  size_t add(T** p, size_t count) {
    const size_t at = bytes;
    parts.push_back({reinterpret_cast<void**>(p), at});
    bytes += (std::max<size_t>(count * sizeof(T), 16) + 255) & ~size_t(255);
    return at;
  }
  cudaError_t alloc(std::vector<void*>& owner) {
    void* q = nullptr;
    const cudaError_t e = cudaMalloc(&q, std::max<size_t>(bytes, 16));
    if (e != cudaSuccess) return e;
    owner.push_back(q);
    for (auto& a : parts) *a.first = static_cast<char*>(q) + a.second;
    return cudaSuccess;
  }
};

// Uploads host arrays into consecutive parts of a Block, `at` bytes behind base:
// small ones in one copy, large ones as they are (assembling them would cost more
// than the copies).
struct Table {
  size_t at;
  const void* src;
  size_t bytes;
};
cudaError_t upload(void* base, std::initializer_list<Table> parts) {
  size_t total = 0;
  for (const Table& t : parts) total = std::max(total, t.at + t.bytes);
  cudaError_t e = cudaSuccess;
  if (total <= (size_t(256) << 10)) {
    std::vector<char> all(total);
    for (const Table& t : parts)
      if (t.bytes) std::memcpy(all.data() + t.at, t.src, t.bytes);
    return total ? cudaMemcpy(base, all.data(), total, cudaMemcpyHostToDevice) : e;
  }
  for (const Table& t : parts)
    if (e == cudaSuccess && t.bytes)
      e = cudaMemcpy(static_cast<char*>(base) + t.at, t.src, t.bytes, cudaMemcpyHostToDevice);
  return e;
}
template <typename T>
Table table(size_t at, const std::vector<T>& v) {
  return Table{at, v.data(), sizeof(T) * v.size()};
}

void release(cg_ctx* h) {
  if (!h) return;
  int cur = -1;
  cudaGetDevice(&cur);
  cudaSetDevice(h->device);
  for (void* p : h->allocs) cudaFree(p);
  h->allocs.clear();
  if (h->h_ctrl) cudaFreeHost(h->h_ctrl);
  h->h_ctrl = nullptr;
  if (cur >= 0) cudaSetDevice(cur);
}

bool is_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();  // clear the sticky-free error of an unknown pointer
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

cgk::DevCsr dev_view(const cg_ctx* h) {
  cgk::DevCsr A;
  A.stream = h->d_stream;
  A.val64 = h->d_val64;
  A.step = h->d_step;
  A.step_cmax = h->d_step_cmax;
  A.seg_len = h->d_seg_len;
  A.chunk_off = h->d_chunk_off;
  A.warp_chunk = h->d_warp_chunk;
  A.warp_entry = h->d_warp_entry;
  A.step_chunk = h->d_step_chunk;
  A.step_entry = h->d_step_entry;
  A.warp_step = h->d_warp_step;
  A.block_row = h->d_block_row;
  A.n = static_cast<int32_t>(h->n);
  A.nsteps = h->nsteps;
  A.nblocks = h->nblocks;
  A.max_rows = h->max_rows;
  A.nnz = h->nnz;
  A.col16 = h->col16 ? 1 : 0;
  A.keep = 0;
  return A;
}

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

}  // namespace

// ---- BLAS-1 without a handle (Sec. 5.2): scratch per (device, stream)

namespace {

// Scratch of the dot product for one (device, stream) pair, allocated by the
// first call on that pair: kBlasPartials CTA sums, then the arrival counter
// and the two error words, then the device scalar of cg_dot_host.  Calls on
// one stream run one after another, so they can share it; calls on
// different streams use different scratch.
constexpr int kBlasPartials = 1024;
constexpr size_t kBlasScratchBytes = sizeof(double) * (kBlasPartials + 4);
struct BlasScratch {
  double* partials;
  unsigned int* counter;
  int32_t* err;  // [0] raised by the kernel, [1] outcome of the last call
  double* result;
};
// Key: (device, stream, host thread).  The thread is part of the key only for
// cudaStreamPerThread, whose one handle value names a different stream in
// every host thread.
std::mutex g_blas_mu;
std::map<std::tuple<int, uintptr_t, size_t>, double*> g_blas;

int sm_count(int dev) {
  static std::mutex mu;
  static int cache[64] = {0};
  if (dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (!cache[dev] && cudaDeviceGetAttribute(&cache[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    cache[dev] = 0;
  }
  return cache[dev];
}

int64_t l2_bytes(int dev) {
  static std::mutex mu;
  static int cache[64] = {0};
  if (dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (!cache[dev] && cudaDeviceGetAttribute(&cache[dev], cudaDevAttrL2CacheSize, dev) != cudaSuccess) {
    cudaGetLastError();
    cache[dev] = 0;
  }
  return cache[dev];
}

cudaError_t blas_scratch(cudaStream_t s, int* dev_out, BlasScratch* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(g_blas_mu);
  const size_t thread_part = s == cudaStreamPerThread ? std::hash<std::thread::id>{}(std::this_thread::get_id()) : 0;
  auto key = std::make_tuple(dev, reinterpret_cast<uintptr_t>(s), thread_part);
  auto it = g_blas.find(key);
  double* base = nullptr;
  if (it == g_blas.end()) {
    e = cudaMalloc(&base, kBlasScratchBytes);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(base, 0, kBlasScratchBytes, s);
    if (e != cudaSuccess) {
      cudaFree(base);
      return e;
    }
    g_blas.emplace(key, base);
  } else {
    base = it->second;
  }
  out->partials = base;
  out->counter = reinterpret_cast<unsigned int*>(base + kBlasPartials);
  out->err = reinterpret_cast<int32_t*>(base + kBlasPartials + 1);
  out->result = base + kBlasPartials + 2;
  *dev_out = dev;
  return cudaSuccess;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The dot product into `result` (device; NULL: the scratch's scalar);
// *streamed tells which kernel ran.
int dot_launch(const char* who, int64_t n, const double* x, const double* y, double* result, cudaStream_t s,
               BlasScratch* sc, bool* streamed) {
  int dev = 0;
  cudaError_t e = blas_scratch(s, &dev, sc);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, (std::string(who) + ": scratch").c_str());
  const int sms = sm_count(dev);
  if (sms <= 0 || 4 * sms > kBlasPartials)
    return fail(nullptr, CG_ECUDA, std::string(who) + ": unsupported SM count");
  if (!result) result = sc->result;
  *streamed = n >= cgk::dot_stream_min_n() && aligned16(x) && aligned16(y);
  if (*streamed)
    e = cgk::launch_dot_stream(n, x, y, result, sc->partials, sc->counter, sc->err, cgk::dot_stream_grid(n, sms),
                               2000000000ull, s);
  else
    e = cgk::launch_dot(n, x, y, result, sc->partials, sc->counter, cgk::dot_grid(n, sms), s);
  return e == cudaSuccess ? CG_OK : cuda_fail(nullptr, e, (std::string(who) + ": launch").c_str());
}

}  // namespace

extern "C" {

void cg_opts_default(cg_opts* o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->stream = nullptr;
  o->device = -1;
  o->precision = CG_PREC_FP64;
  o->replace_every = 50;
  o->validate = 1;
  o->wait_limit_ms = 2000;
  o->preconditioner = CG_PRECOND_NONE;
  o->ctas = 0;
}

const char* cg_last_error(cg_handle h) { return h ? h->err.c_str() : g_create_err.c_str(); }

int cg_create(cg_handle* out, const cg_csr* csr, int64_t n, int64_t nnz, const cg_opts* opts) {
  if (!out) return fail(nullptr, CG_EINVAL, "cg_create: out is NULL");
  *out = nullptr;
  if (!csr) return fail(nullptr, CG_EINVAL, "cg_create: csr is NULL");
  cg_opts o;
  cg_opts_default(&o);
  if (opts) o = *opts;
  const int base = csr->index_base;
  if (base != 0 && base != 1) return fail(nullptr, CG_EINVAL, "cg_create: index_base must be 0 or 1");
  const int64_t kMaxIdx = 2147483647LL - 16;
  if (n < 0 || nnz < 0 || n > kMaxIdx || nnz > kMaxIdx)
    return fail(nullptr, CG_EINVAL, "cg_create: n and nnz must be in [0, 2^31 - 16)");
  if (o.precision != CG_PREC_FP64 && o.precision != CG_PREC_MIXED)
    return fail(nullptr, CG_EINVAL, "cg_create: unknown precision");
  if (o.replace_every < 0) return fail(nullptr, CG_EINVAL, "cg_create: replace_every must be >= 0");
  if (o.preconditioner != CG_PRECOND_NONE && o.preconditioner != CG_PRECOND_JACOBI)
    return fail(nullptr, CG_EINVAL, "cg_create: unknown preconditioner");
  if (o.ctas < 0) return fail(nullptr, CG_EINVAL, "cg_create: ctas must be >= 0");
  if (!csr->row_ptr || (nnz > 0 && (!csr->col_idx || !csr->val)))
    return fail(nullptr, CG_EINVAL, "cg_create: NULL CSR array");

  // Host copies of row_ptr and col_idx (needed for validation and partitioning).
  std::vector<int32_t> rp(static_cast<size_t>(n) + 1), ci;
  const bool need_cols_on_host = o.validate || base != 0 || !csr->on_device;
  if (!csr->on_device) {
    std::memcpy(rp.data(), csr->row_ptr, sizeof(int32_t) * (n + 1));
    ci.assign(csr->col_idx, csr->col_idx + nnz);
  }

  // Host inputs are validated before any CUDA call (see the block below).
  auto validate_csr = [&](std::string& bad) {
    bad.clear();
    if (rp[0] != base) bad = "row_ptr[0] != index_base";
    for (int64_t i = 0; bad.empty() && i < n; ++i)
      if (rp[i + 1] < rp[i]) bad = "row_ptr decreases at row " + std::to_string(i);
    if (bad.empty() && static_cast<int64_t>(rp[n]) - base != nnz) bad = "row_ptr[n] != nnz + index_base";
    for (int64_t k = 0; bad.empty() && k < nnz; ++k)
      if (ci[k] < base || static_cast<int64_t>(ci[k]) - base >= n)
        bad = "column index out of range at entry " + std::to_string(k);
    return bad.empty();
  };
  if (!csr->on_device && o.validate) {
    std::string bad;
    if (!validate_csr(bad)) return fail(nullptr, CG_EINVAL, "cg_create: invalid CSR: " + bad);
  }

  cg_ctx* h = new (std::nothrow) cg_ctx();
  if (!h) return fail(nullptr, CG_ENOMEM, "cg_create: host allocation failed");
  if (o.device >= 0) h->device = o.device;
  else if (cudaGetDevice(&h->device) != cudaSuccess) h->device = 0;
  DeviceGuard guard(h->device);
  h->stream = static_cast<cudaStream_t>(o.stream);
  h->precision = o.precision;
  h->preconditioner = o.preconditioner;
  h->replace_every = o.replace_every;
  h->wait_limit_ns = static_cast<unsigned long long>(o.wait_limit_ms > 0 ? o.wait_limit_ms : 2000) * 1000000ull;
  h->n = n;
  h->nnz = nnz;
  cudaError_t e;
#define CG_TRY(call, what)                       \
  do {                                           \
    e = (call);                                  \
    if (e != cudaSuccess) {                      \
      int rc__ = cuda_fail(nullptr, e, what);    \
      release(h);                                \
      delete h;                                  \
      return rc__;                               \
    }                                            \
  } while (0)

  if (csr->on_device) {
    CG_TRY(cudaMemcpy(rp.data(), csr->row_ptr, sizeof(int32_t) * (n + 1), cudaMemcpyDefault),
           "cg_create: copy of row_ptr");
    if (need_cols_on_host && nnz > 0) {
      ci.resize(static_cast<size_t>(nnz));
      CG_TRY(cudaMemcpy(ci.data(), csr->col_idx, sizeof(int32_t) * nnz, cudaMemcpyDefault),
             "cg_create: copy of col_idx");
    }
  }
  // Validation of the CSR structure (Sec. 2.3 definition) for device inputs.
  if (csr->on_device && o.validate) {
    std::string bad;
    if (!validate_csr(bad)) {
      delete h;
      return fail(nullptr, CG_EINVAL, "cg_create: invalid CSR: " + bad);
    }
  }
  if (base) {
    for (auto& v : rp) v -= 1;
    for (auto& v : ci) v -= 1;
  }

  int sms = 0;
  CG_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device), "cg_create: SM count");
  h->num_sms = sms;
  const int per_sm = cgk::solve_blocks_per_sm(o.precision == CG_PREC_MIXED, o.preconditioner == CG_PRECOND_JACOBI);
  if (per_sm <= 0) {
    int rc = fail(nullptr, CG_ECUDA, "cg_create: the solve kernel cannot be resident (occupancy 0)");
    release(h);
    delete h;
    return rc;
  }
  h->nblocks = sms * per_sm;
  // every SM unless the caller asks for fewer: measured on GB300, fewer CTAs
  // do not shorten the solve of small systems (a 16^3 7-point system takes
  // 0.90 ms on 152 CTAs, 0.93 ms on 16 and 1.85 ms on one)
  if (o.ctas > 0) h->nblocks = std::min(h->nblocks, o.ctas);
  if (h->nblocks > 1024) {  // the group-wide fixed-point sum takes at most 1024 CTA values
    int rc = fail(nullptr, CG_ECUDA, "cg_create: more persistent CTAs than the grid-wide sum supports");
    release(h);
    delete h;
    return rc;
  }

  Partition part;
  const bool mixed = o.precision == CG_PREC_MIXED;
  // A system of at most 12 rows per warp of the whole GPU with rows long enough:
  // two lanes per row, so that more warps work and each row's FMA chain, which
  // bounds so small a product, is half as long (whole-grid step with one lane, with
  // two, us: Q1 16^3 11.9, 10.7; 24^3 11.9, 11.0; 32^3 12.5, 12.2; beyond the line
  // 35^3 12.9, 13.6, its mesh 13.5, 15.1; rows of 7 entries 32^3 10.1, 10.4).  By the
  // matrix alone, so that a product's bits do not depend on the CTA count.
  cgh::StepShape shape;
  if (n <= static_cast<int64_t>(sms) * 12 * cgk::kWarps && nnz >= 12 * n)
    for (int L = 0; L <= cgk::kLaneMax; ++L) shape.mode[L] = static_cast<int8_t>(cgk::kPairPerRow);
  build_partition(rp, n, h->nblocks, mixed, part, shape);
  h->nsteps = static_cast<int>(part.step.size()) - 1;
  for (int b = 0; b < h->nblocks; ++b)
    h->max_rows = std::max(h->max_rows, part.block_row[b + 1] - part.block_row[b]);
  // Small plain FP64 systems (the CTA count left automatic): one cluster of
  // CTAs holding the system in shared memory, if its layout fits and such a
  // cluster can be resident.
  if (h->precision == CG_PREC_FP64 && h->preconditioner == CG_PRECOND_NONE && o.ctas <= 0 && n > 0 &&
      n <= static_cast<int64_t>(cgk::kClusterCtas) * cgk::kClusterMaxRows) {
    int R = 1;  // rows per CTA: a power of two, so the owner of a column is a shift
    while (static_cast<int64_t>(R) * cgk::kClusterCtas < n) R <<= 1;
    int E = 0;
    for (int c = 0; c < cgk::kClusterCtas; ++c) {
      const int64_t r0 = std::min<int64_t>(static_cast<int64_t>(c) * R, n);
      const int64_t r1 = std::min<int64_t>(r0 + R, n);
      E = std::max(E, rp[r1] - rp[r0]);
    }
    E = std::max(E, 1);
    if (cgk::cluster_max_active(R, E) > 0) {  // 0 if the layout is too large or no cluster fits
      h->cluster_R = R;
      h->cluster_E = E;
    }
  }

  // the cluster kernel reads CSR: its handles keep 0-based copies
  const bool keep_csr = h->cluster_R > 0;
  const size_t nn = static_cast<size_t>(n), nz = static_cast<size_t>(nnz);
  Block blk;
  const size_t at_step = blk.add(&h->d_step, part.step.size());  // (the tables of one upload first)
  const size_t at_wstep = blk.add(&h->d_warp_step, part.warp_step.size());
  const size_t at_brow = blk.add(&h->d_block_row, part.block_row.size());
  blk.add(&h->d_step_cmax, part.step.size());
  blk.add(&h->d_seg_len, 32 * static_cast<size_t>(h->nsteps) + 64);
  blk.add(&h->d_r, nn);
  blk.add(&h->d_p, nn);
  blk.add(&h->d_q, nn);
  blk.add(&h->d_xbuf, nn);
  blk.add(&h->d_bbuf, nn);
  blk.add(&h->d_partials, static_cast<size_t>(6) * h->nblocks);
  unsigned char* ctrl = nullptr;
  blk.add(&ctrl, ctrl_block_bytes(h->nblocks));
  blk.add(&h->d_err, 16);
  if (mixed) blk.add(&h->d_p32, nn);
  if (o.preconditioner == CG_PRECOND_JACOBI) blk.add(&h->d_dinv, nn);
  if (keep_csr) {
    blk.add(&h->d_csr_row_ptr, nn + 1);
    blk.add(&h->d_csr_col, nz);
    blk.add(&h->d_csr_val, nz);
  }
  // The streams, whose size the scan tells: with the rest where their bound is
  // small (an allocation of more than a megabyte takes 100 us, and 50 to free)
  int64_t most_units = 0, most_entries = 0;
  cgh::stream_bound(nnz, mixed, part, &most_units, &most_entries);
  const size_t most = static_cast<size_t>(most_units) * cgk::kUnit + sizeof(double) * static_cast<size_t>(mixed ? most_entries : 0);
  const bool one_block = most <= (size_t(16) << 20);
  Block str;
  Block& sb = one_block ? blk : str;
  const size_t warps = static_cast<size_t>(h->nblocks) * cgk::kWarps, steps = mixed ? static_cast<size_t>(h->nsteps) : 0;
  size_t at_wchunk = 0, at_wentry = 0, at_coff = 0, at_schunk = 0, at_sentry = 0;
  auto add_streams = [&](size_t chunks, int64_t units, int64_t entries) {
    at_wchunk = sb.add(&h->d_warp_chunk, warps);
    at_wentry = sb.add(&h->d_warp_entry, mixed ? warps : 0) - at_wchunk;
    at_schunk = sb.add(&h->d_step_chunk, steps) - at_wchunk;
    at_sentry = sb.add(&h->d_step_entry, steps) - at_wchunk;
    at_coff = sb.add(&h->d_chunk_off, chunks + 1) - at_wchunk;
    sb.add(&h->d_stream, static_cast<size_t>(units) * cgk::kUnit);
    if (mixed) sb.add(&h->d_val64, static_cast<size_t>(entries));
    at_wchunk = 0;
  };
  if (one_block) add_streams(static_cast<size_t>(part.chunks), most_units, most_entries);
  CG_TRY(blk.alloc(h->allocs), "cg_create: cudaMalloc");
  h->d_ctrl = reinterpret_cast<cgk::SolveCtrl*>(ctrl);
  h->d_flags = reinterpret_cast<unsigned long long*>(ctrl + ctrl_flags_offset());
  CG_TRY(cudaMallocHost(&h->h_ctrl, sizeof(cgk::SolveCtrl)), "cg_create: cudaMallocHost");
  CG_TRY(upload(h->d_step, {table(at_step, part.step), table(at_wstep, part.warp_step), table(at_brow, part.block_row)}),
         "cg_create: upload");
  CG_TRY(cudaMemset(h->d_err, 0, 64), "cg_create: memset");

  // The CSR arrays on the device for the time of the conversion: the caller's
  // own where they are there already, the kept copies, or copies that go when
  // this returns.
  std::vector<void*> temps;
  struct TempGuard {
    std::vector<void*>& v;
    ~TempGuard() {
      for (void* q : v) cudaFree(q);
    }
  } temp_guard{temps};
  int32_t* d_rp = h->d_csr_row_ptr;
  int32_t* d_ci = h->d_csr_col;
  double* d_va = h->d_csr_val;
  const bool in_place = csr->on_device && cgh::readable_in_place(csr->row_ptr, h->device) &&
                        (nnz == 0 || (cgh::readable_in_place(csr->col_idx, h->device) &&
                                      cgh::readable_in_place(csr->val, h->device)));
  const bool callers_rp = !keep_csr && in_place && base == 0;  // (the caller's row pointers serve as they are)
  if (!keep_csr && !callers_rp) {
    Block tmp;
    tmp.add(&d_rp, nn + 1);
    if (!in_place) {
      tmp.add(&d_ci, nz);
      tmp.add(&d_va, nz);
    }
    CG_TRY(tmp.alloc(temps), "cg_create: cudaMalloc");
  }
  if (!callers_rp)
    CG_TRY(cudaMemcpy(d_rp, rp.data(), sizeof(int32_t) * (nn + 1), cudaMemcpyHostToDevice), "cg_create: upload");
  cgk::CsrSource src{};
  src.row_ptr = callers_rp ? csr->row_ptr : d_rp;
  src.col_idx = csr->col_idx;
  src.val = csr->val;
  src.base = base;
  if (d_ci != nullptr && nnz > 0) {
    if (csr->on_device && base == 0)
      CG_TRY(cudaMemcpy(d_ci, csr->col_idx, sizeof(int32_t) * nz, cudaMemcpyDefault), "cg_create: copy");
    else
      CG_TRY(cudaMemcpy(d_ci, ci.data(), sizeof(int32_t) * nz, cudaMemcpyHostToDevice), "cg_create: upload");
    CG_TRY(cudaMemcpy(d_va, csr->val, sizeof(double) * nz, csr->on_device ? cudaMemcpyDefault : cudaMemcpyHostToDevice),
           "cg_create: upload");
    src.col_idx = d_ci;
    src.val = d_va;
    src.base = 0;  // ci is rebased
  }
  cgk::LayoutScan* const d_scan = reinterpret_cast<cgk::LayoutScan*>(h->d_err + 4);
  CG_TRY(cgk::launch_layout_scan(src, h->d_step, h->d_seg_len, h->d_step_cmax, 0, h->nsteps, 0, static_cast<int32_t>(n), n,
                                 false, d_scan, nullptr),
         "cg_create: column scan");
  if (o.preconditioner == CG_PRECOND_JACOBI)
    CG_TRY(cgk::launch_jacobi_dinv(src, 0, n, h->d_dinv, h->d_err, nullptr),
           "cg_create: Jacobi diagonal");
  struct {
    int32_t err[4];
    cgk::LayoutScan scan;
  } found{};
  CG_TRY(cudaMemcpy(&found, h->d_err, sizeof(found), cudaMemcpyDeviceToHost), "cg_create: read-back");
  if (found.err[0] != 0) {
    release(h);
    delete h;
    return fail(nullptr, CG_EINVAL, "cg_create: Jacobi preconditioner: diagonal of row " +
                                        std::to_string(found.err[0] - 1) + " is not positive (A is not SPD)");
  }
  h->col16 = found.scan.span <= cgk::kColSpan16;
  cgh::place_steps(rp, h->nblocks, h->col16, mixed, part);
  h->stream_bytes = part.stream_units * cgk::kUnit;
  if (!one_block) {
    add_streams(part.chunk_off.size() - 1, part.stream_units, part.entries);
    CG_TRY(str.alloc(h->allocs), "cg_create: cudaMalloc");
  }
  // in FP64 the steps' places in the streams serve the conversion only: q holds
  // them until the handle's first solve (a step has at least one row)
  static_assert(sizeof(double) >= sizeof(uint32_t), "step_chunk fits q");
  uint32_t* const d_step_chunk = mixed ? h->d_step_chunk : reinterpret_cast<uint32_t*>(h->d_q);
  part.step_chunk.resize(static_cast<size_t>(h->nsteps));  // (no sentinel)
  part.step_entry.resize(steps);
  if (!mixed) CG_TRY(upload(d_step_chunk, {table(0, part.step_chunk)}), "cg_create: upload");
  part.step_chunk.resize(steps);
  CG_TRY(upload(h->d_warp_chunk, {table(at_wchunk, part.warp_chunk), table(at_wentry, part.warp_entry),
                                  table(at_schunk, part.step_chunk), table(at_sentry, part.step_entry),
                                  table(at_coff, part.chunk_off)}),
         "cg_create: upload");
  const cgk::StreamPlace to{h->d_chunk_off, d_step_chunk, h->d_step_entry, h->d_stream, h->d_val64};
  CG_TRY(cgk::launch_layout_fill(src, h->d_step, to, 0, h->nsteps, 0, static_cast<int32_t>(n), h->col16, mixed, nullptr),
         "cg_create: stream order");
  CG_TRY(cudaDeviceSynchronize(), "cg_create: synchronize");
#undef CG_TRY
  *out = h;
  return CG_OK;
}

int cg_destroy(cg_handle h) {
  if (!h) return CG_OK;
  release(h);
  delete h;
  return CG_OK;
}

int cg_info(cg_handle h, int64_t* n, int64_t* nnz, int32_t* nblocks) {
  if (!h) return fail(nullptr, CG_EINVAL, "cg_info: NULL handle");
  if (n) *n = h->n;
  if (nnz) *nnz = h->nnz;
  if (nblocks) *nblocks = h->nblocks;
  return CG_OK;
}

int cg_partition_info(cg_handle h, int32_t* max_rows, int32_t* kernel) {
  if (!h) return fail(nullptr, CG_EINVAL, "cg_partition_info: NULL handle");
  if (max_rows) *max_rows = h->cluster_R > 0 ? h->cluster_R : h->max_rows;
  if (kernel)
    *kernel = h->cluster_R > 0                      ? CG_SOLVE_KERNEL_CLUSTER
              : cgk::small_share(dev_view(h), 0) ? CG_SOLVE_KERNEL_SMALL_SHARE
                                                  : CG_SOLVE_KERNEL_LARGE_SHARE;
  return CG_OK;
}

int cg_spmv(cg_handle h, const double* x, double* y) {
  if (!h) return fail(nullptr, CG_EINVAL, "cg_spmv: NULL handle");
  if (h->n == 0) return CG_OK;
  if (!x || !y) return fail(h, CG_EINVAL, "cg_spmv: NULL vector");
  DeviceGuard g(h->device);
  cgk::DevCsr A = dev_view(h);
  // (a mixed handle's product reads the columns and FP64 values)
  const int64_t matrix = h->precision == CG_PREC_MIXED ? 12 * h->nnz : h->stream_bytes;
  A.keep = cgk::streams_stay(matrix, 16 * h->n, l2_bytes(h->device)) ? 1 : 0;
  cudaError_t e = cgk::launch_spmv(A, x, y, h->d_err, h->stream);
  return e == cudaSuccess ? CG_OK : cuda_fail(h, e, "cg_spmv: launch");
}

int cg_dot(int64_t n, const double* x, const double* y, double* result, void* stream) {
  if (n < 0 || !result || (n > 0 && (!x || !y))) return fail(nullptr, CG_EINVAL, "cg_dot: bad arguments");
  BlasScratch sc;
  bool streamed = false;
  return dot_launch("cg_dot", n, x, y, result, static_cast<cudaStream_t>(stream), &sc, &streamed);
}

int cg_dot_host(int64_t n, const double* x, const double* y, double* result, void* stream) {
  if (n < 0 || !result || (n > 0 && (!x || !y))) return fail(nullptr, CG_EINVAL, "cg_dot_host: bad arguments");
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  BlasScratch sc;
  bool streamed = false;
  const int rc = dot_launch("cg_dot_host", n, x, y, nullptr, s, &sc, &streamed);
  if (rc != CG_OK) return rc;
  double v = 0.0;
  int32_t bad = 0;
  cudaError_t e = cudaMemcpyAsync(&v, sc.result, sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && streamed) e = cudaMemcpyAsync(&bad, sc.err + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cg_dot_host");
  if (bad) return fail(nullptr, CG_ETIMEOUT, "cg_dot_host: a device-side wait of the dot kernel gave up");
  *result = v;
  return CG_OK;
}

int cg_axpy(int64_t n, double a, const double* x, double* y, void* stream) {
  if (n < 0 || (n > 0 && (!x || !y))) return fail(nullptr, CG_EINVAL, "cg_axpy: bad arguments");
  if (n == 0) return CG_OK;
  cudaError_t e = cgk::launch_axpy(n, a, x, y, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? CG_OK : cuda_fail(nullptr, e, "cg_axpy: launch");
}

int cg_ewmul(int64_t n, const double* x, const double* y, double* z, void* stream) {
  if (n < 0 || (n > 0 && (!x || !y || !z))) return fail(nullptr, CG_EINVAL, "cg_ewmul: bad arguments");
  if (n == 0) return CG_OK;
  cudaError_t e = cgk::launch_ewmul(n, x, y, z, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? CG_OK : cuda_fail(nullptr, e, "cg_ewmul: launch");
}

int cg_probe_fp64_peak(int32_t device, double* gflops) {
  if (!gflops) return fail(nullptr, CG_EINVAL, "cg_probe_fp64_peak: NULL output");
  *gflops = 0.0;
  int dev = device;
  if (dev < 0 && cudaGetDevice(&dev) != cudaSuccess) return fail(nullptr, CG_ECUDA, "cg_probe_fp64_peak: no device");
  DeviceGuard g(dev);
  const int sms = sm_count(dev);
  if (sms <= 0) return fail(nullptr, CG_ECUDA, "cg_probe_fp64_peak: SM count");
  double* sink = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaMalloc(&sink, sizeof(double) * static_cast<size_t>(sms) * 8);
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  double best = 0.0;
  // two, four and eight CTAs of 256 threads per SM; for each, two launches
  // warm up and size the next three to about 40 ms, the best of which counts
  for (int per_sm = 2; e == cudaSuccess && per_sm <= 8; per_sm *= 2) {
    const int grid = sms * per_sm;
    const double per_iter = static_cast<double>(grid) * cgk::kFp64ProbeThreads * cgk::kFp64ProbeFmasPerIter;
    int64_t iters = 500;
    for (int rep = 0; e == cudaSuccess && rep < 5; ++rep) {
      e = cudaEventRecord(e0, nullptr);
      if (e == cudaSuccess) e = cgk::launch_fp64_probe(iters, grid, sink, nullptr);
      if (e == cudaSuccess) e = cudaEventRecord(e1, nullptr);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e != cudaSuccess || ms <= 0.f) break;
      if (rep >= 2) best = std::max(best, 2.0 * per_iter * static_cast<double>(iters) / (ms * 1e-3) / 1e9);
      if (rep == 1) iters = std::max<int64_t>(iters, static_cast<int64_t>(iters * (40.0 / ms)));
    }
  }
  if (e1) cudaEventDestroy(e1);
  if (e0) cudaEventDestroy(e0);
  if (sink) cudaFree(sink);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cg_probe_fp64_peak");
  *gflops = best;
  return CG_OK;
}

int cg_probe_group_sync(int32_t device, int32_t iters, double* barrier_us, double* sum_us) {
  if (!barrier_us || !sum_us || iters < 1 || iters > 1000000)
    return fail(nullptr, CG_EINVAL, "cg_probe_group_sync: iters in [1, 10^6] and two outputs");
  *barrier_us = 0.0;
  *sum_us = 0.0;
  int dev = device;
  if (dev < 0 && cudaGetDevice(&dev) != cudaSuccess) return fail(nullptr, CG_ECUDA, "cg_probe_group_sync: no device");
  DeviceGuard g(dev);
  const int sms = sm_count(dev);
  if (sms <= 0) return fail(nullptr, CG_ECUDA, "cg_probe_group_sync: SM count");
  const int nb = sms * cgk::kCtasPerSm;
  char* buf = nullptr;
  cgk::SolveCtrl* ctrl = nullptr;
  double* partials = nullptr;
  double* out = nullptr;
  const size_t ctrl_bytes = (sizeof(cgk::SolveCtrl) + 255) & ~size_t(255);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaMalloc(&buf, ctrl_bytes + sizeof(double) * 3 * static_cast<size_t>(nb));
  if (e == cudaSuccess) {
    ctrl = reinterpret_cast<cgk::SolveCtrl*>(buf);
    partials = reinterpret_cast<double*>(buf + ctrl_bytes);
    out = partials + 2 * static_cast<size_t>(nb);
    e = cudaEventCreate(&e0);
  }
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  bool timed_out = false;
  double per_iter[2] = {0.0, 0.0};
  for (int mode = 0; e == cudaSuccess && mode < 2 && !timed_out; ++mode) {
    // a short launch first (clocks, first-touch), then the timed one
    for (int rep = 0; e == cudaSuccess && rep < 2; ++rep) {
      const int n_it = rep == 0 ? std::max(1, iters / 10) : iters;
      e = cudaMemset(ctrl, 0, sizeof(cgk::SolveCtrl));
      if (e == cudaSuccess) e = cudaEventRecord(e0, nullptr);
      if (e == cudaSuccess) e = cgk::launch_sync_probe(ctrl, partials, n_it, mode, nb, 2000000000ull, out, nullptr);
      if (e == cudaSuccess) e = cudaEventRecord(e1, nullptr);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      float ms = 0.f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      int32_t abort_flag = 0;
      if (e == cudaSuccess)
        e = cudaMemcpy(&abort_flag, &ctrl->abort, sizeof(int32_t), cudaMemcpyDeviceToHost);
      if (e == cudaSuccess && abort_flag) timed_out = true;
      if (e == cudaSuccess && rep == 1) per_iter[mode] = 1000.0 * static_cast<double>(ms) / n_it;
      if (timed_out) break;
    }
  }
  if (e1) cudaEventDestroy(e1);
  if (e0) cudaEventDestroy(e0);
  if (buf) cudaFree(buf);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cg_probe_group_sync");
  if (timed_out) return fail(nullptr, CG_ETIMEOUT, "cg_probe_group_sync: a group barrier wait gave up");
  *barrier_us = per_iter[0];
  *sum_us = per_iter[1];
  return CG_OK;
}

int cg_blas_release(void) {
  std::lock_guard<std::mutex> lock(g_blas_mu);
  int cur = -1;
  cudaGetDevice(&cur);
  for (auto& kv : g_blas) {
    cudaSetDevice(std::get<0>(kv.first));
    cudaFree(kv.second);
  }
  g_blas.clear();
  if (cur >= 0) cudaSetDevice(cur);
  return CG_OK;
}

int cg_solve(cg_handle h, const double* b, double* x, double tol, int64_t maxit, int64_t* iters, double* relres) {
  if (!h) return fail(nullptr, CG_EINVAL, "cg_solve: NULL handle");
  if (!iters || !relres) return fail(h, CG_EINVAL, "cg_solve: NULL output");
  if (!(tol >= 0.0)) return fail(h, CG_EINVAL, "cg_solve: tol must be >= 0");
  if (maxit < 0) return fail(h, CG_EINVAL, "cg_solve: maxit must be >= 0");
  *iters = 0;
  *relres = 0.0;
  if (h->n == 0) return CG_OK;
  if (!b || !x) return fail(h, CG_EINVAL, "cg_solve: NULL vector");
  DeviceGuard g(h->device);
  const size_t bytes = sizeof(double) * static_cast<size_t>(h->n);
  const bool b_dev = is_device_ptr(b), x_dev = is_device_ptr(x);
  const double* db = b;
  double* dx = x;
  cudaError_t e;
  if (!b_dev) {
    e = cudaMemcpyAsync(h->d_bbuf, b, bytes, cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: copy of b");
    db = h->d_bbuf;
  }
  if (!x_dev) {
    e = cudaMemcpyAsync(h->d_xbuf, x, bytes, cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: copy of x");
    dx = h->d_xbuf;
  }
  e = cudaMemsetAsync(h->d_ctrl, 0, ctrl_block_bytes(h->nblocks), h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: memset");
  cgk::SolveParams P;
  P.A = dev_view(h);
  P.b = db;
  P.x = dx;
  P.r = h->d_r;
  P.p = h->d_p;
  P.q = h->d_q;
  P.p32 = h->d_p32;
  P.partials = h->d_partials;
  P.ctrl = h->d_ctrl;
  P.tol = tol;
  P.maxit = maxit;
  P.replace_every = h->replace_every;
  P.wait_limit_ns = h->wait_limit_ns;
  P.group = h->nblocks;
  const int64_t reused = cgk::step_reused_bytes(h->n, h->precision == CG_PREC_MIXED, h->d_dinv != nullptr);
  P.stream_rows = cgk::stream_row_tables(reused, l2_bytes(h->device));
  P.A.keep = cgk::streams_stay(h->stream_bytes, reused, l2_bytes(h->device)) ? 1 : 0;
  P.chunk_iters = 0;
  P.dinv = h->d_dinv;
  P.flags = h->nblocks > 1 ? h->d_flags : nullptr;
  if (h->cluster_R > 0)
    e = cgk::launch_cluster_solve(h->d_csr_row_ptr, h->d_csr_col, h->d_csr_val, db, dx, h->d_ctrl, tol, maxit,
                                  static_cast<int32_t>(h->n), h->cluster_R, h->cluster_E, h->stream);
  else
    e = cgk::launch_solve(P, h->precision == CG_PREC_MIXED, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: launch");
  e = cudaMemcpyAsync(h->h_ctrl, h->d_ctrl, sizeof(cgk::SolveCtrl), cudaMemcpyDeviceToHost, h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: read-back");
  if (!x_dev) {
    e = cudaMemcpyAsync(x, h->d_xbuf, bytes, cudaMemcpyDeviceToHost, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: copy of x");
  }
  e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "cg_solve: synchronize");
  *iters = h->h_ctrl->iters;
  *relres = h->h_ctrl->relres_true;
  const int st = h->h_ctrl->status;
  if (st == CG_ETIMEOUT)
    return fail(h, CG_ETIMEOUT, "cg_solve: a device-side wait gave up (site " +
                                    std::to_string(h->h_ctrl->timeout_site) + ")");
  if (st == CG_EBREAKDOWN) return fail(h, CG_EBREAKDOWN, "cg_solve: breakdown (p.Ap <= 0 or not finite)");
  if (st == CG_ENOTCONV) return fail(h, CG_ENOTCONV, "cg_solve: maxit reached before the tolerance");
  return st;
}

int cg_dot_noalloc(int64_t n, const double* x, const double* y, double* result, void* stream) {
  const int64_t max_n = cgk::dot_noalloc_max_n();
  if (n < 0 || !result || (n > 0 && (!x || !y))) return fail(nullptr, CG_EINVAL, "cg_dot_noalloc: bad arguments");
  if (n > max_n)
    return fail(nullptr, CG_EINVAL,
                "cg_dot_noalloc: n = " + std::to_string(n) + " exceeds the fixed scratch capacity of " +
                    std::to_string(max_n) + " elements; use cg_dot");
  cudaError_t e = cgk::launch_dot_noalloc(n, x, y, result, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? CG_OK : cuda_fail(nullptr, e, "cg_dot_noalloc");
}

int cg_selftest_wait_timeout(int32_t limit_ms, int32_t* kernel_status) {
  if (!kernel_status || limit_ms <= 0 || limit_ms > 10000)
    return fail(nullptr, CG_EINVAL, "cg_selftest_wait_timeout: limit_ms in (0, 10000] and a status pointer");
  cgk::SolveCtrl* d = nullptr;
  cudaError_t e = cudaMalloc(&d, sizeof(cgk::SolveCtrl));
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cg_selftest_wait_timeout: cudaMalloc");
  cgk::SolveCtrl hc;
  e = cudaMemset(d, 0, sizeof(cgk::SolveCtrl));
  if (e == cudaSuccess)
    e = cgk::launch_wait_timeout_selftest(d, static_cast<unsigned long long>(limit_ms) * 1000000ull, nullptr);
  if (e == cudaSuccess) e = cudaMemcpy(&hc, d, sizeof(hc), cudaMemcpyDeviceToHost);
  cudaFree(d);
  if (e != cudaSuccess) return cuda_fail(nullptr, e, "cg_selftest_wait_timeout");
  *kernel_status = hc.status;
  if (hc.status == CG_ETIMEOUT && (hc.abort != 1 || hc.timeout_site != cgk::kSelftestSite))
    return fail(nullptr, CG_ECUDA, "cg_selftest_wait_timeout: the wait gave up without raising the abort flag");
  return CG_OK;
}

}  // extern "C"
