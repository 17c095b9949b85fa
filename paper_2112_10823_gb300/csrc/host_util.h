// Host-side helpers shared by the single-system and batched entry points:
// the step partition of a CSR matrix for the persistent kernels.
#pragma once
#include <cstdint>
#include <vector>
#include <vector_types.h>
#include "cg_internal.h"

namespace cgh {

// Row partition of the persistent kernels for `nblocks` CTAs: CTA ranges of
// about equal cost (block_row), each split into steps (see cg_internal.h),
// which are listed warp by warp (warp_step).  One sentinel step follows the
// last one.  The steps' smallest columns are left 0.
// place_steps adds the streams: the chunks of every warp (warp_chunk,
// chunk_off), each step's place in them and the stream's size.
struct Partition {
  std::vector<int4> step;
  std::vector<int32_t> warp_step;
  std::vector<int32_t> block_row;
  int64_t chunks = 0;        // of all streams (at most)
  int64_t padded = 0;        // entries with the padding of 16-bit columns
  // by place_steps
  std::vector<int4> warp_chunk;
  std::vector<uint32_t> chunk_off;
  std::vector<uint32_t> step_chunk;
  std::vector<uint32_t> warp_entry;  // mixed precision
  std::vector<uint32_t> step_entry;
  int64_t stream_units = 0;
  int64_t entries = 0;       // stored, padding included
};

// Which kind of step (cgk::StepMode: one lane per row, two lanes per row, or
// a warp per row) rows of each length 0..64 go to; longer rows always take a
// warp each.  A step's kind is the widest kind among its rows; a one-lane
// step holds up to 32 rows, a two-lane step up to 16.  The built-in table is
// one lane for rows of up to 32 entries and two lanes for 33..64.  A lane
// computes at most 32 entries, so mode[L] may be "one lane" only for L <= 32.
constexpr int kShapeMaxLen = 64;
struct StepShape {
  int8_t mode[kShapeMaxLen + 1];
  bool tight = false;  // little padding (cgk::step_pads)
  StepShape();
  bool valid() const;
};

void build_partition(const std::vector<int32_t>& rp, int64_t n, int nblocks, bool mixed, Partition& P,
                     const StepShape& shape = StepShape());
void place_steps(const std::vector<int32_t>& rp, int nblocks, bool col16, bool mixed, Partition& P);
// Upper bounds of stream_units and entries for either column width.
void stream_bound(int64_t nnz, bool mixed, const Partition& P, int64_t* stream_units, int64_t* entries);

// Whether kernels on `device` may read p in place: its own or managed memory.
// Another GPU's memory can be copied, but not always read by a kernel.
inline bool readable_in_place(const void* p, int device) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeManaged || (a.type == cudaMemoryTypeDevice && a.device == device);
}
}  // namespace cgh
