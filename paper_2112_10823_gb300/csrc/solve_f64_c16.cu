// Single-system solve kernels: FP64 values, 16-bit column offsets.
#include "solve_kernel.cuh"

namespace cgk {
template const void* solve_kernel_of<false, uint16_t>(bool jacobi, bool small);
}
