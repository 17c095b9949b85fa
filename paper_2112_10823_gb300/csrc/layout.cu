// Stream order of a matrix (cg_internal.h): what a handle or an admitted
// system keeps of its CSR arrays, built on the device, one warp per step.
// Both kernels are bound by the CSR arrays' bytes and, with few or long steps, by
// latency: the scan reads the columns once, eight loads of a lane under way; the fill
// reads every entry once (lanes at the stride of a row, so that a warp's reads of
// consecutive entries of 32 rows meet again in L1; a batch of loads before its
// stores) and writes it once.  Q1 160^3: 108 and 711 us.
#include <algorithm>
#include "cg_device.cuh"

namespace cgk {

namespace {
constexpr int kLayoutBlock = 256;
constexpr int kFillWarps = 152 * 48;  // what the fill of long rows is spread over
constexpr int kBatch = 5;  // entries per lane whose loads are under way together

unsigned layout_grid(int32_t s0, int32_t s1) {
  return static_cast<unsigned>((static_cast<int64_t>(s1 - s0) * 32 + kLayoutBlock - 1) / kLayoutBlock);
}

__device__ __forceinline__ int step_rows(const int4& d) {
  const int mode = step_mode(d);
  return mode == kLanePerRow ? step_lanes(d) : mode == kPairPerRow ? step_lanes(d) >> 1 : 1;
}
}  // namespace

__global__ void __launch_bounds__(kLayoutBlock)
    layout_scan_kernel(const CsrSource src, int4* step, uint8_t* seg_len, int32_t* cmax, int32_t s0, int32_t s1,
                       int32_t row0, int32_t row1, int64_t n, int check, LayoutScan* out) {
  const int s = s0 + static_cast<int>((static_cast<int64_t>(blockIdx.x) * kLayoutBlock + threadIdx.x) >> 5);
  if (s >= s1) return;
  const int lane = threadIdx.x & 31;
  const int4 d = step[s];
  if (d.x < row0 || d.x >= row1) return;
  const int64_t e0 = src.row_ptr[d.x], e1 = src.row_ptr[d.x + step_rows(d)];
  int lo = 0x7fffffff, hi = -1;
  unsigned long long bad = 0;
#pragma unroll 8
  for (int64_t k = e0 + lane; k < e1; k += 32) {
    // (unsigned: a column below the base wraps to a large value)
    const unsigned int c =
        static_cast<unsigned int>(__ldg(src.col_idx + (k - src.e_first))) - static_cast<unsigned int>(src.base);
    if (check && static_cast<int64_t>(c) >= n) {
      const unsigned long long at = ~static_cast<unsigned long long>(k);
      bad = at > bad ? at : bad;
    } else {
      lo = min(lo, static_cast<int>(c));
      hi = max(hi, static_cast<int>(c));
    }
  }
  if (step_mode(d) != kLongRow) {
    int len = 0;
    if (lane < step_lanes(d)) {
      const int row = d.x + (step_mode(d) == kLanePerRow ? lane : lane >> 1);
      len = src.row_ptr[row + 1] - src.row_ptr[row];
      if (step_mode(d) == kPairPerRow) len = (lane & 1) ? len >> 1 : (len + 1) >> 1;
    }
    seg_len[static_cast<size_t>(s) * 32 + lane] = static_cast<uint8_t>(len);
  }
  if (bad) atomicMax(&out->bad_entry, bad);
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    step[s].w = hi < 0 ? 0 : lo;
    if (cmax != nullptr) cmax[s] = hi;
    // (one address for all: mostly a read that an older value cannot mislead)
    if (hi > lo && hi - lo > *static_cast<const volatile int32_t*>(&out->span)) atomicMax(&out->span, hi - lo);
  }
}

template <typename T, typename C>
__global__ void __launch_bounds__(kLayoutBlock)
    layout_fill_kernel(const CsrSource src, int4* __restrict__ step, const StreamPlace to, int32_t s0,
                       int32_t s1, int32_t row0, int32_t row1) {
  const int s = s0 + static_cast<int>((static_cast<int64_t>(blockIdx.x) * kLayoutBlock + threadIdx.x) >> 5);
  if (s >= s1) return;
  const int lane = threadIdx.x & 31;
  int4 d = step[s];
  if (d.x < row0 || d.x >= row1) return;
  const int size = chunk_of(d.z, max_chunk(sizeof(T) == 4, sizeof(C) == 2));
  d.y = (d.y & ~(kStepChunkMask << kStepChunkShift)) | size << kStepChunkShift;
  const int mode = step_mode(d);
  // a long row's chunks are shared by the blocks (x, 0..): chunks [j0, j1)
  const int nchunks = d.z > 0 ? (d.z + size - 1) / size : 0, part = static_cast<int>(blockIdx.y);
  if (part > 0 && mode != kLongRow) return;
  const int per = mode == kLongRow ? (nchunks + static_cast<int>(gridDim.y) - 1) / static_cast<int>(gridDim.y) : nchunks;
  const int j0 = part * per, u1 = min(d.z, (j0 + per) * size);
  if (lane == 0 && part == 0) step[s].y = d.y;
  // this lane's segment in CSR order: entries a, a + stride, ...
  int64_t a = 0;
  int len = 0;
  const int stride = mode == kLongRow ? 32 : 1;
  if (mode == kLongRow) {
    a = src.row_ptr[d.x] + static_cast<int64_t>(lane);
    const int64_t left = src.row_ptr[d.x + 1] - a;
    len = left > 0 ? static_cast<int>((left + 31) >> 5) : 0;
  } else if (lane < step_lanes(d)) {
    const int row = d.x + (mode == kLanePerRow ? lane : lane >> 1);
    a = src.row_ptr[row];
    len = static_cast<int>(src.row_ptr[row + 1] - a);
    if (mode == kPairPerRow) {
      const int half = (len + 1) >> 1;
      if (lane & 1) {
        a += half;
        len -= half;
      } else {
        len = half;
      }
    }
  }
  a -= src.e_first;
  const int base = src.base + (sizeof(C) == 2 ? d.w : 0);
  const bool padded = step_padded<C>(d);
  uint32_t chunk = to.step_chunk[s] + static_cast<uint32_t>(j0);
  // (a long row's chunks are full but the last)
  int64_t entry = sizeof(T) == 4 ? to.step_entry[s] + static_cast<int64_t>(32) * j0 * size : 0;
  a += static_cast<int64_t>(j0) * size * stride;
  for (int u0 = j0 * size; u0 < u1; u0 += size, ++chunk) {
    const int cnt = min(size, d.z - u0);
    const int mine = padded ? cnt : max(0, min(len - u0, cnt));
    const ChunkPlace place = chunk_place<C>(d, u0, cnt, len, lane);
    unsigned char* const at = to.stream + static_cast<size_t>(to.chunk_off[chunk]) * kUnit;
    C* const col = reinterpret_cast<C*>(at);
    T* const val = reinterpret_cast<T*>(at + units(static_cast<int64_t>(place.tot) * sizeof(C)) * kUnit);
    // a batch's loads before its stores
    int dst = place.base;
    for (int k0 = 0; k0 < mine; k0 += kBatch) {
      int c[kBatch] = {};
      double v[kBatch] = {};
#pragma unroll
      for (int k = 0; k < kBatch; ++k)
        if (k0 + k < mine && u0 + k0 + k < len) {
          c[k] = __ldg(src.col_idx + (a + k * stride)) - base;
          v[k] = __ldg(src.val + (a + k * stride));
        }
#pragma unroll
      for (int k = 0; k < kBatch; ++k, dst += place.stride)
        if (k0 + k < mine) {
          col[dst] = static_cast<C>(c[k]);
          val[dst] = static_cast<T>(v[k]);  // (round to nearest)
          if (sizeof(T) == 4) to.val64[entry + dst] = v[k];
        }
      a += kBatch * stride;
    }
    a += (mine - (mine + kBatch - 1) / kBatch * kBatch) * stride;
    entry += place.tot;
  }
}

cudaError_t launch_layout_scan(const CsrSource& src, int4* step, uint8_t* seg_len, int32_t* cmax, int32_t s0, int32_t s1,
                               int32_t row0, int32_t row1, int64_t n, bool check, LayoutScan* out, cudaStream_t s) {
  if (s1 <= s0) return cudaSuccess;
  layout_scan_kernel<<<layout_grid(s0, s1), kLayoutBlock, 0, s>>>(src, step, seg_len, cmax, s0, s1, row0, row1, n,
                                                                 check ? 1 : 0, out);
  return cudaGetLastError();
}

cudaError_t launch_layout_fill(const CsrSource& src, int4* step, const StreamPlace& to, int32_t s0, int32_t s1,
                               int32_t row0, int32_t row1, bool col16, bool mixed, cudaStream_t s) {
  if (s1 <= s0) return cudaSuccess;
  // where steps are few, up to eight warps for each long row (1000 rows of 20,000
  // entries: 399 -> 72 us)
  const unsigned parts = static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(8, kFillWarps / (s1 - s0))));
  const dim3 grid(layout_grid(s0, s1), parts);
  auto fill = [&](auto kernel) { kernel<<<grid, kLayoutBlock, 0, s>>>(src, step, to, s0, s1, row0, row1); };
  if (mixed) col16 ? fill(layout_fill_kernel<float, uint16_t>) : fill(layout_fill_kernel<float, int32_t>);
  else col16 ? fill(layout_fill_kernel<double, uint16_t>) : fill(layout_fill_kernel<double, int32_t>);
  return cudaGetLastError();
}

}  // namespace cgk
